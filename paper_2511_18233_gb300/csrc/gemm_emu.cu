// FP64-accurate GEMM on the FP16 tensor cores (tcgen05) of sm_103a by exact
// splitting of both operands into small-integer slices: the error-free
// transformation of matrix products of Ozaki, Ogita, Oishi and Rump
// (Numer. Algorithms 59, 2012), with digit slices in one fixed-point frame
// per row.
//
// With x_rk = 2^(E_r - F) sum_{p=0..S-1} dA_p(r,k) 2^(b(S-1-p)) (b bits per
// slice, F fraction bits of the frame) and y_ck likewise,
//   (X Y^T)_rc = 2^(E_r + E_c - 2F + b(S-1)) sum_{g=0..S-1} 2^(b(S-1-g)) V_g(r,c),
//   V_g = sum_{p+q=g} sum_k dA_p(r,k) dB_q(c,k),
// products with p + q >= S being dropped (below the frames' resolution).
// Digits are FP16 integers, their products are exact, and over a chunk of
// at most Form::kChunk values of k every V_g that matters stays within 2^24
// and is summed exactly in its FP32 tensor-memory accumulator:
//   10 x 6 bits  512 * 63^2 * 8 < 2^24 (the two lowest accumulators, nine and
//                ten terms, may lose their last bit, 2^-60 below the frame)
//   9 x 7 bits   balanced digits: 448 * 64^2 * 9 < 2^24, all nine exact
// The epilogue combines the accumulators of a chunk in 64-bit integers.  The
// 10 x 6 form converts each chunk to FP64 and adds chunks in FP64; the 9 x 7
// form keeps adding integers over all chunks (also over the CTAs of a split
// contraction) and rounds once at the end.
//
// Kernel (one 128 x BN output tile per CTA, 320 threads, one CTA per SM):
//   warp 0 / lane 0 : TMA producer, 4-stage ring; a stage is K = 16 of all
//                     slices of A (128 rows) and of B (BN rows), two 3-D
//                     loads with 32-byte swizzle
//   warp 1          : allocates 512 TMEM columns (S accumulators of BN
//                     columns); lane 0 issues the slice products.  The B
//                     slices of a stage lie one after the other, and so do
//                     the accumulators g = p, p + 1, ..., so one
//                     tcgen05.mma of N = (up to 256 / BN) BN multiplies A
//                     slice p with several B slices at once: the 128-row A
//                     slice is read from shared memory once per such group
//                     instead of once per product (15 instructions a stage
//                     instead of 55 at 10 x 6, BN = 48)
//   warps 2-9       : epilogue, one output row and every other block of 8
//                     columns per thread
// FP64 arithmetic is kept out of the epilogue (GB300 issues about 1.7 FP64
// operations per clock per SM, so five per output would cost a 128 x 48 tile
// 18k cycles, the time of 500 values of k): the result is rounded to FP64
// with integer operations, bit for bit what the FP64 combination gives.
// Every mbarrier wait is bounded; a timeout sets the error flag, drains what
// the CTA has in flight and frees its tensor memory.
#include <cuda.h>

#include <algorithm>

#include "gemm_emu.cuh"
#include "tc_ptx.cuh"

namespace ris {

namespace {
using namespace tcx;

constexpr int EBM = 128, EBK = 16, ESTAGES = 4;
constexpr int A_SLICE = EBM * EBK * 2;  // 4 KB
constexpr int TMEM_COLS = 512;
constexpr int EPI_WARPS = 8, ETHREADS = 64 + 32 * EPI_WARPS;

struct Form10x6 {
  static constexpr int S = 10, kFrac = 60, kChunk = 512, kMaxBN = 48;
  static constexpr bool kBalanced = false;
};
struct Form9x7 {
  static constexpr int S = 9, kFrac = 62, kChunk = 448, kMaxBN = 48;
  static constexpr bool kBalanced = true;
};

template <class F>
struct Tile {
  static constexpr int kABytes = F::S * A_SLICE;
  static constexpr int kStage = ((kABytes + F::S * F::kMaxBN * EBK * 2) + 1023) & ~1023;
  static constexpr int kSmem = ESTAGES * kStage + 1024 + 256;
  static_assert(F::S * F::kMaxBN <= TMEM_COLS, "accumulators exceed tensor memory");
  static_assert(kSmem <= 232448, "pipeline exceeds shared memory");
};

// 3-D map {K, rows, slice} of FP16 digits, box {16, box_rows, S}, 32-byte swizzle.
CUtensorMap make_map(const EmuOperand& op, int slices, int box_rows) {
  RIS_REQUIRE(((uintptr_t)op.s & 15) == 0, RIS_ERR_ARG, "emu_gemm: slices not 16-byte aligned");
  RIS_REQUIRE(op.ldk % 8 == 0 && op.ldk >= op.K, RIS_ERR_ARG, "emu_gemm: ldk must be a multiple of 8");
  CUtensorMap m;
  cuuint64_t dims[3] = {(cuuint64_t)op.K, (cuuint64_t)op.rows, (cuuint64_t)slices};
  cuuint64_t strides[2] = {(cuuint64_t)op.ldk * 2, (cuuint64_t)op.plane * 2};
  cuuint32_t box[3] = {EBK, (cuuint32_t)box_rows, (cuuint32_t)slices};
  cuuint32_t es[3] = {1, 1, 1};
  CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, (void*)op.s, dims, strides, box, es,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  RIS_REQUIRE(r == CUDA_SUCCESS, RIS_ERR_CUDA, "cuTensorMapEncodeTiled failed (" + std::to_string((int)r) + ")");
  return m;
}

// K-major operand tile, rows of 32 bytes with 32-byte swizzle: start
// address, leading offset unused (1), 256 B between 8-row groups,
// descriptor version 1, layout type 6 (SWIZZLE_32B).
__device__ __forceinline__ uint64_t desc_sw32(const void* p) {
  const uint64_t a = sa(p);
  return ((a & 0x3FFFFull) >> 4) | (1ull << 16) | ((uint64_t)(256 >> 4) << 32) | (1ull << 46) |
         (6ull << 61);
}

// kind::f16 instruction descriptor: D FP32 (bit 4), A and B FP16 (0 at bits
// 7 and 10), both K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t idesc_f16(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(EBM >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

// four consecutive accumulator columns of this warp's 32 lanes (not waited on)
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float (&v)[4]) {
  uint32_t r[4];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr)
               : "memory");
#pragma unroll
  for (int i = 0; i < 4; i++) v[i] = __uint_as_float(r[i]);
}

struct EmuArgs {
  int M, N, K, bn;
  int ntn;         // column tiles (fastest on grid.x)
  int nchunk, cps; // chunks of the contraction, chunks per slice of it (blockIdx.y)
  const int* ea;
  const int* eb;
  longlong2* ws;   // split contraction: [blockIdx.y][M][N] integer partial sums
  EmuEpilogue ep;
  int* err;
};

__device__ __forceinline__ long long emu_off(int i, int in, long long ld, long long s) {
  return in > 0 ? (long long)(i / in) * ld + (long long)(i % in) * s : (long long)i * s;
}

// (hi 2^sh + lo) 2^e rounded to the nearest FP64 (ties to even), 0 < sh < 64,
// |hi| 2^sh + |lo| < 2^126.  Integer operations; results outside the normal
// range go through ldexp.
__device__ __forceinline__ double emu_round(long long hi, long long lo, int sh, int e) {
  unsigned long long L = (unsigned long long)hi << sh;
  long long H = hi >> (64 - sh);
  const unsigned long long L0 = L;
  L += (unsigned long long)lo;
  H += (lo >> 63) + (L < L0 ? 1 : 0);
  const bool neg = H < 0;
  if (neg) {
    L = ~L + 1ull;
    H = ~H + (L == 0 ? 1 : 0);
  }
  if ((H | (long long)L) == 0) return 0.0;
  const int lz = H ? __clzll(H) : 64 + __clzll((long long)L);
  unsigned long long top, rest;
  if (lz >= 64) {
    top = L << (lz - 64);
    rest = 0;
  } else {
    top = lz ? ((unsigned long long)H << lz) | (L >> (64 - lz)) : (unsigned long long)H;
    rest = L << lz;
  }
  unsigned long long m = top >> 11;
  const unsigned rb = (unsigned)(top & 0x7FFu);
  if (rb > 0x400u || (rb == 0x400u && (rest != 0 || (m & 1)))) m++;
  const int ex = 127 - lz + e;  // exponent of the leading bit
  if (ex < -1021 || ex > 1022) {
    const double x = ldexp((double)(long long)m, ex - 52);
    return neg ? -x : x;
  }
  // m in [2^52, 2^53]: adding it onto the exponent field carries by itself
  const unsigned long long b = ((unsigned long long)(ex + 1022) << 52) + m;
  return __longlong_as_double((long long)(neg ? b | 0x8000000000000000ull : b));
}

// lo rounded to a 53-bit significand (what a conversion to FP64 keeps)
__device__ __forceinline__ long long emu_round53(long long lo) {
  unsigned long long a = lo < 0 ? 0ull - (unsigned long long)lo : (unsigned long long)lo;
  const int drop = 11 - __clzll((long long)a);  // bits beyond 53
  if (drop > 0) {
    const unsigned long long half = 1ull << (drop - 1), mask = (half << 1) - 1;
    const unsigned long long r = a & mask;
    a -= r;
    if (r > half || (r == half && (a & (mask + 1)))) a += mask + 1;
  }
  return lo < 0 ? -(long long)a : (long long)a;
}

// Sum of one output over the chunks.
template <class F>
struct EmuAcc;
// 9 x 7: hi = sum_{g<4} V_g 2^(7(3-g)), lo = sum_{g>=4} V_g 2^(7(8-g)),
// integers over all chunks (below 2^46 and 2^53 per chunk)
template <>
struct EmuAcc<Form9x7> {
  static constexpr int kShift = 35;
  long long hi, lo;
  __device__ __forceinline__ void zero() { hi = lo = 0; }
  __device__ __forceinline__ void add(const float (&v)[9], int, bool) {
#pragma unroll
    for (int g = 0; g < 4; g++) hi += (long long)__float2int_rn(v[g]) * (1 << (7 * (3 - g)));
#pragma unroll
    for (int g = 4; g < 9; g++) lo += (long long)__float2int_rn(v[g]) * (1 << (7 * (8 - g)));
  }
  static __device__ __forceinline__ double value(long long hi, long long lo, int e) {
    return emu_round(hi, lo, kShift, e - 2 * Form9x7::kFrac + 56);
  }
  __device__ __forceinline__ double result(int e) const { return value(hi, lo, e); }
};
// 10 x 6: hi = V_0 2^12 + V_1 2^6 + V_2, lo = sum_{g>=3} V_g 2^(6(9-g)) < 2^61;
// each chunk is fl(hi 2^42 + fl(lo)) (one conversion and one FMA in FP64),
// chunks added in FP64
template <>
struct EmuAcc<Form10x6> {
  double s;
  __device__ __forceinline__ void zero() { s = 0.0; }
  __device__ __forceinline__ void add(const float (&v)[10], int e, bool first) {
    const long long hi = (long long)__float2int_rn(v[0]) * 4096 +
                         (long long)__float2int_rn(v[1]) * 64 + __float2int_rn(v[2]);
    long long lo = 0;
#pragma unroll
    for (int g = 3; g < 6; g++) lo += (long long)__float2int_rn(v[g]) * (1ll << (6 * (9 - g)));
    long long l2 = 0;
#pragma unroll
    for (int g = 6; g < 10; g++) l2 += (long long)__float2int_rn(v[g]) * (1 << (6 * (9 - g)));
    const double x = emu_round(hi, emu_round53(lo + l2), 42, e - 2 * 6 - 54);
    s = first ? x : s + x;
  }
  __device__ __forceinline__ double result(int) const { return s; }
};

template <class F>
__global__ void __launch_bounds__(ETHREADS, 1) k_emu_gemm(const __grid_constant__ CUtensorMap mA,
                                                           const __grid_constant__ CUtensorMap mB,
                                                           EmuArgs args) {
  constexpr int S = F::S;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + ESTAGES * Tile<F>::kStage);
  uint64_t* empty = full + ESTAGES;
  uint64_t* acc_full = empty + ESTAGES;   // a chunk's accumulators are complete
  uint64_t* acc_empty = acc_full + 1;     // the epilogue has read them
  uint64_t* done = acc_empty + 1;         // every product issued has completed
  uint32_t* tmem_slot = (uint32_t*)(done + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int bn = args.bn;
  const int n0 = (int)(blockIdx.x % args.ntn) * bn, m0 = (int)(blockIdx.x / args.ntn) * EBM;
  const int c0 = blockIdx.y * args.cps, c1 = min(args.nchunk, c0 + args.cps);
  const int kbeg = c0 * F::kChunk, kend = min(args.K, c1 * F::kChunk);
  const int nk = (kend - kbeg + EBK - 1) / EBK;  // stages (kChunk is a multiple of EBK)
  const uint32_t stage_tx = (uint32_t)(Tile<F>::kABytes + S * bn * EBK * 2);

  if (threadIdx.x == 0) {
    for (int s = 0; s < ESTAGES; s++) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, EPI_WARPS);
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(sa(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      // producer
      int issued = 0;
      for (int i = 0; i < nk; i++) {
        const int s = i % ESTAGES;
        if (i >= ESTAGES && !mbar_wait(&empty[s], ((i / ESTAGES) - 1) & 1)) {
          *abort_flag = 1;
          break;
        }
        if (*abort_flag) break;
        uint8_t* st = smem + s * Tile<F>::kStage;
        mbar_expect_tx(&full[s], stage_tx);
        tma_load(st, &mA, &full[s], kbeg + i * EBK, m0, 0);
        tma_load(st + Tile<F>::kABytes, &mB, &full[s], kbeg + i * EBK, n0, 0);
        issued = i + 1;
      }
      for (int i = (issued > ESTAGES ? issued - ESTAGES : 0); i < issued; i++)
        mbar_wait(&full[i % ESTAGES], (i / ESTAGES) & 1);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // MMA issuer: slice products p + q < S into accumulator p + q
      const int per = 256 / bn;  // B slices per instruction
      constexpr int kSteps = F::kChunk / EBK;
      for (int i = 0; i < nk; i++) {
        const int s = i % ESTAGES, in = i % kSteps, ch = i / kSteps;
        // a new chunk: the epilogue must have read the previous one
        if (in == 0 && ch > 0 && !mbar_wait(acc_empty, (ch - 1) & 1)) {
          *abort_flag = 1;
          break;
        }
        if (!mbar_wait(&full[s], (i / ESTAGES) & 1)) {
          *abort_flag = 1;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint8_t* st = smem + s * Tile<F>::kStage;
#pragma unroll 1
        for (int p = 0; p < S; p++) {
          const uint64_t da = desc_sw32(st + p * A_SLICE);
          for (int q = 0; q < S - p; q += per) {
            const int nq = min(per, S - p - q);
            const uint64_t db = desc_sw32(st + Tile<F>::kABytes + q * bn * EBK * 2);
            mma_f16(tmem + (uint32_t)((p + q) * bn), da, db, idesc_f16(nq * bn),
                    (in > 0 || p > 0) ? 1u : 0u);
          }
        }
        mma_commit(&empty[s]);
        if (in == kSteps - 1 || i == nk - 1) mma_commit(acc_full);
      }
      // nothing is left in flight when the tensor memory is freed, whatever happened
      mma_commit(done);
      if (!mbar_wait(done, 0)) *abort_flag = 1;
    }
  } else {
    // epilogue: row = TMEM lane of this warp's quadrant, column blocks of 8
    // shared between the two warps of a quadrant
    constexpr int NB = F::kMaxBN / 16;
    EmuAcc<F> acc[NB][8];
#pragma unroll
    for (int b = 0; b < NB; b++)
#pragma unroll
      for (int j = 0; j < 8; j++) acc[b][j].zero();
    const int quad = warp & 3, half = (warp - 2) >> 2;
    const int row = m0 + quad * 32 + lane;
    const bool live = row < args.M;
    const int er = live ? args.ea[row] : 0;
    const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16);
    bool good = true;
    for (int ch = 0; ch < c1 - c0; ch++) {
      if (!mbar_wait(acc_full, ch & 1) || *abort_flag) {
        good = false;
        break;
      }
      __syncwarp();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int b = 0; b < NB; b++) {
        const int cb = b * 16 + half * 8;
        if (cb < bn) {
#pragma unroll
          for (int h = 0; h < 2; h++) {
            float v[S][4];
#pragma unroll
            for (int g = 0; g < S; g++) tmem_ld4(lane_base + (uint32_t)(g * bn + cb + 4 * h), v[g]);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int j = 0; j < 4; j++) {
              float u[S];
#pragma unroll
              for (int g = 0; g < S; g++) u[g] = v[g][j];
              int e = 0;
              if (!F::kBalanced) e = er + args.eb[min(n0 + cb + 4 * h + j, args.N - 1)];
              acc[b][4 * h + j].add(u, e, ch == 0);
            }
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty);
    }
    if (!good) *abort_flag = 1;
    const EmuEpilogue& ep = args.ep;
    if (good && live) {
      const long long roff = emu_off(row, ep.rin, ep.rld, ep.rs);
#pragma unroll
      for (int b = 0; b < NB; b++) {
        const int cb = b * 16 + half * 8;
#pragma unroll
        for (int j = 0; j < 8; j++) {
          const int col = n0 + cb + j;
          if (cb >= bn || col >= args.N) continue;
          if constexpr (F::kBalanced) {
            if (args.ws) {  // one slice of the contraction: integer partial sums
              longlong2 t;
              t.x = acc[b][j].hi;
              t.y = acc[b][j].lo;
              args.ws[((size_t)blockIdx.y * args.M + row) * args.N + col] = t;
              continue;
            }
          }
          const int ec = args.eb[col];
          double x = acc[b][j].result(er + ec);
          if (er >= kEmuNonFinite / 2 || ec >= kEmuNonFinite / 2) x = __longlong_as_double(0x7ff8000000000000ll);
          double* p = ep.c64 + roff + emu_off(col, ep.cin, ep.cld, ep.cs);
          if (ep.beta != 0.0)
            *p = fma(ep.alpha, x, ep.beta * *p);
          else
            *p = ep.alpha == 1.0 ? x : ep.alpha * x;
        }
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) atomicExch(args.err, 1);
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS)
                 : "memory");
  }
}

// Adds the integer partial sums of a split contraction (exact in any order)
// and rounds once.
__global__ void __launch_bounds__(256) k_emu_finish(EmuArgs args, int nsplit) {
  const long long t = (long long)blockIdx.x * 256 + threadIdx.x;
  const long long mn = (long long)args.M * args.N;
  if (t >= mn) return;
  long long hi = 0, lo = 0;
  for (int z = 0; z < nsplit; z++) {
    const longlong2 w = args.ws[(size_t)z * mn + t];
    hi += w.x;
    lo += w.y;
  }
  const int row = (int)(t / args.N), col = (int)(t % args.N);
  const int er = args.ea[row], ec = args.eb[col];
  double x = EmuAcc<Form9x7>::value(hi, lo, er + ec);
  if (er >= kEmuNonFinite / 2 || ec >= kEmuNonFinite / 2) x = __longlong_as_double(0x7ff8000000000000ll);
  const EmuEpilogue& ep = args.ep;
  double* p = ep.c64 + emu_off(row, ep.rin, ep.rld, ep.rs) + emu_off(col, ep.cin, ep.cld, ep.cs);
  if (ep.beta != 0.0)
    *p = fma(ep.alpha, x, ep.beta * *p);
  else
    *p = ep.alpha == 1.0 ? x : ep.alpha * x;
}

// ------------------------------------------------------------------ slicing
// Row exponents: E_r = 1 + max_k floor(log2 |x_rk|) (subnormals included;
// 0 for a row of zeros), so that every |x_rk| < 2^(E_r).
constexpr int kNoLead = -4096;
constexpr int kLeadBad = 1024;  // lead_exp of an infinity or a NaN
__device__ __forceinline__ int lead_exp(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ef = (int)((b >> 52) & 0x7FF);
  if (ef) return ef - 1023;
  const unsigned long long m = b & 0xFFFFFFFFFFFFFull;
  return m ? -1011 - __clzll(m) : kNoLead;  // -1074 + (63 - clz)
}
__device__ __forceinline__ int row_frame(int lead) {
  return lead == kNoLead ? 0 : lead >= kLeadBad ? kEmuNonFinite : lead + 1;
}

// Digits of two elements in their row frame as FP16 pairs d[p] = (digit p of
// x0, digit p of x1), on the integer pipe.  A digit u + bias is turned into
// FP16 by or-ing it into the significand of 1024 and subtracting 1024 + bias.
template <class F>
struct Digits;
template <>
struct Digits<Form10x6> {
  // X = floor(|x| 2^(60 - E)), d_p = its bits [60 - 6(p+1), 60 - 6p), signed like x
  static __device__ __forceinline__ unsigned long long fixed(double x, int E, unsigned& neg) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ef = (int)((b >> 52) & 0x7FF);
    unsigned long long m = b & 0xFFFFFFFFFFFFFull;
    int q = -1074;  // |x| = m 2^q
    if (ef) {
      m |= 1ull << 52;
      q = ef - 1075;
    }
    neg = (unsigned)(b >> 63);
    const int sh = q + Form10x6::kFrac - E;
    return sh >= 0 ? (m << sh) : (sh <= -64 ? 0ull : (m >> -sh));
  }
  static __device__ __forceinline__ void cut(double x0, double x1, int E, unsigned (&d)[10]) {
    unsigned n0, n1;
    const unsigned long long X0 = fixed(x0, E, n0), X1 = fixed(x1, E, n1);
    const unsigned sign = (n0 << 15) | (n1 << 31);
    const __half2 bias = __halves2half2(__ushort_as_half(0x6400), __ushort_as_half(0x6400));
#pragma unroll
    for (int p = 0; p < 10; p++) {
      const int sh = 60 - 6 * (p + 1);
      const unsigned w = ((unsigned)(X0 >> sh) & 63u) | (((unsigned)(X1 >> sh) & 63u) << 16) | 0x64006400u;
      const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), bias);
      d[p] = *reinterpret_cast<const unsigned*>(&h) ^ sign;
    }
  }
};
template <>
struct Digits<Form9x7> {
  // X = round(x 2^(62 - E)), |X| <= 2^62; with 64 added to each of the eight
  // lower digits, digit p is a 7-bit field less 64 and the top digit, in
  // [-64, 64], what is left above
  static __device__ __forceinline__ long long fixed(double x, int E) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ef = (int)((b >> 52) & 0x7FF);
    unsigned long long m = b & 0xFFFFFFFFFFFFFull;
    int q = -1074;
    if (ef) {
      m |= 1ull << 52;
      q = ef - 1075;
    }
    const int sh = q + Form9x7::kFrac - E;
    const unsigned long long X =
        sh >= 0 ? (m << sh) : (sh <= -60 ? 0ull : ((m >> (-sh - 1)) + 1) >> 1);
    return (b >> 63) ? -(long long)X : (long long)X;
  }
  static __device__ __forceinline__ void cut(double x0, double x1, int E, unsigned (&d)[9]) {
    constexpr long long kBias = 64ll * ((1ll << 56) - 1) / 127;  // 64 in each of eight 7-bit fields
    const long long X0 = fixed(x0, E) + kBias, X1 = fixed(x1, E) + kBias;
    const __half2 bias = __halves2half2(__ushort_as_half(0x6440), __ushort_as_half(0x6440));  // 1088
    const unsigned t0 = (unsigned)((int)(X0 >> 56) + 64), t1 = (unsigned)((int)(X1 >> 56) + 64);
    unsigned w = t0 | (t1 << 16) | 0x64006400u;
    __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), bias);
    d[0] = *reinterpret_cast<const unsigned*>(&h);
#pragma unroll
    for (int p = 1; p < 9; p++) {
      const int sh = 7 * (8 - p);
      w = ((unsigned)(X0 >> sh) & 127u) | (((unsigned)(X1 >> sh) & 127u) << 16) | 0x64006400u;
      h = __hsub2(*reinterpret_cast<const __half2*>(&w), bias);
      d[p] = *reinterpret_cast<const unsigned*>(&h);
    }
  }
};

// four consecutive digits per slice of one row, 8-byte stores
template <class F>
__device__ __forceinline__ void put4(const double (&x)[4], int E, __half* o, size_t plane) {
  unsigned a[F::S], b[F::S];
  if (E == kEmuNonFinite) E = 0;  // digits are not used
  Digits<F>::cut(x[0], x[1], E, a);
  Digits<F>::cut(x[2], x[3], E, b);
#pragma unroll
  for (int p = 0; p < F::S; p++) *reinterpret_cast<uint2*>(o + (size_t)p * plane) = make_uint2(a[p], b[p]);
}

// Rows contiguous in k: TPR threads per row find the row's exponent, then cut
// it (the second read comes from L2: one pass over DRAM instead of two).
template <class F, int TPR>
__global__ void __launch_bounds__(256) k_emu_slice_rows(EmuSource src, int rows, int K,
                                                        int* __restrict__ E, __half* __restrict__ out,
                                                        int ldk) {
  __shared__ int red[8];
  const int r = blockIdx.x * (256 / TPR) + threadIdx.x / TPR;
  const int t = threadIdx.x % TPR;
  const bool on = r < rows;
  const double* x = on ? src.p + emu_off(r, src.rin, src.rld, src.rs) : src.p;
  int m = kNoLead;
  if (on)
    for (int k = t; k < K; k += TPR) m = max(m, lead_exp(x[k]));
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (TPR > 32) {
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    for (int w = 0; w < 8; w++) m = max(m, red[w]);
  }
  if (!on) return;
  const int e = row_frame(m);
  if (t == 0) E[r] = e;
  const size_t plane = (size_t)rows * ldk;
  for (int k = 4 * t; k < ldk; k += 4 * TPR) {
    double v[4];
#pragma unroll
    for (int i = 0; i < 4; i++) v[i] = k + i < K ? x[k + i] : 0.0;
    put4<F>(v, e, out + (size_t)r * ldk + k, plane);
  }
}

// Rows strided in k (consecutive rows adjacent in memory): 32 rows per CTA,
// lanes along the rows for the reads, transposed through shared memory.
template <class F>
__global__ void __launch_bounds__(256) k_emu_slice_cols(EmuSource src, int rows, int K,
                                                        int* __restrict__ E, __half* __restrict__ out,
                                                        int ldk) {
  __shared__ double tile[64][33];  // [k][r]
  __shared__ int red[8][32];
  const int r0 = blockIdx.x * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const bool on = r0 + tx < rows;
  const double* x = src.p + (on ? emu_off(r0 + tx, src.rin, src.rld, src.rs) : 0);
  int m = kNoLead;
  if (on)
#pragma unroll 4
    for (int k = ty; k < K; k += 8) m = max(m, lead_exp(x[(size_t)k * src.ks]));
  red[ty][tx] = m;
  __syncthreads();
  if (ty == 0) {
    for (int y = 1; y < 8; y++) m = max(m, red[y][tx]);
    m = row_frame(m);
    red[0][tx] = m;
    if (on) E[r0 + tx] = m;
  }
  const size_t plane = (size_t)rows * ldk;
  const int q = threadIdx.x & 15, rr0 = threadIdx.x >> 4;  // 16 threads x 4 digits per row
  for (int k0 = 0; k0 < ldk; k0 += 64) {
    __syncthreads();
#pragma unroll
    for (int kk = ty; kk < 64; kk += 8)
      tile[kk][tx] = (on && k0 + kk < K) ? x[(size_t)(k0 + kk) * src.ks] : 0.0;
    __syncthreads();
#pragma unroll
    for (int rr = rr0; rr < 32; rr += 16) {
      const int k = k0 + 4 * q;
      if (r0 + rr >= rows || k >= ldk) continue;
      double v[4];
#pragma unroll
      for (int i = 0; i < 4; i++) v[i] = tile[4 * q + i][rr];
      put4<F>(v, red[0][rr], out + (size_t)(r0 + rr) * ldk + k, plane);
    }
  }
}

template <class F>
void slice_form(const EmuSource& src, int rows, int K, EmuOperand& op, cudaStream_t st) {
  if (src.ks == 1) {
    // long rows take a CTA each so that a few hundred rows fill the device
    if (K >= 2048)
      k_emu_slice_rows<F, 256><<<rows, 256, 0, st>>>(src, rows, K, op.e, op.s, op.ldk);
    else
      k_emu_slice_rows<F, 32><<<cdiv(rows, 8), 256, 0, st>>>(src, rows, K, op.e, op.s, op.ldk);
  } else {
    k_emu_slice_cols<F><<<cdiv(rows, 32), 256, 0, st>>>(src, rows, K, op.e, op.s, op.ldk);
  }
  RIS_CHECK_LAUNCH();
}

// Tile width: a stage brings (128 + BN) rows of digits through shared memory
// whatever the products, so the total over the column tiles is taken least;
// ties go to the wider tile.
int pick_bn(int N, int max_bn) {
  int bn = max_bn;
  for (int c = max_bn; c >= 16; c -= 16)
    if ((long long)cdiv(N, c) * (EBM + c) < (long long)cdiv(N, bn) * (EBM + bn)) bn = c;
  return bn;
}

template <class F>
void gemm_pass(int M, int N, const EmuOperand& A, const EmuOperand& B, const EmuEpilogue& ep,
               int* d_err, cudaStream_t st) {
  ensure_smem_attr((const void*)k_emu_gemm<F>, Tile<F>::kSmem);
  EmuArgs a;
  a.M = M;
  a.N = N;
  a.K = A.K;
  a.bn = pick_bn(N, F::kMaxBN);
  a.ntn = cdiv(N, a.bn);
  a.nchunk = cdiv(A.K, F::kChunk);
  a.ea = A.e;
  a.eb = B.e;
  a.ws = nullptr;
  a.ep = ep;
  a.err = d_err;
  const long long tiles = (long long)a.ntn * cdiv(M, EBM);
  RIS_REQUIRE(tiles < (1LL << 31), RIS_ERR_ARG, "emu_gemm: too many tiles");
  // slices of a long contraction: the number of chunk rounds of the busiest
  // SM, plus about a chunk's time for each CTA's start and end
  int ns = 1;
  if (F::kBalanced && a.nchunk > 1) {
    long long best = -1;
    for (int s = 1; s <= std::min(a.nchunk, 64); s++) {
      const int cps = cdiv(a.nchunk, s);
      if (cdiv(a.nchunk, cps) != s) continue;
      if (s > 1 && (double)s * M * N * sizeof(longlong2) > 1e9) break;
      const long long cost = (long long)cdiv(tiles * s, 152) * (2 * cps + 1);
      if (best < 0 || cost < best) {
        best = cost;
        ns = s;
      }
    }
  }
  a.cps = cdiv(a.nchunk, ns);
  MemTrack* tr = nullptr;
  const size_t wsb = (size_t)ns * M * N * sizeof(longlong2);
  if (ns > 1) a.ws = (longlong2*)dev_alloc(wsb, st, &tr);
  const CUtensorMap mA = make_map(A, F::S, EBM);
  const CUtensorMap mB = make_map(B, F::S, a.bn);
  k_emu_gemm<F><<<dim3((unsigned)tiles, ns), ETHREADS, Tile<F>::kSmem, st>>>(mA, mB, a);
  RIS_CHECK_LAUNCH();
  if (ns > 1) {
    k_emu_finish<<<cdiv((long long)M * N, 256), 256, 0, st>>>(a, ns);
    RIS_CHECK_LAUNCH();
    dev_free(a.ws, wsb, st, tr);
  }
}

// Contractions beyond kPassChunks chunks (the 64-bit sums hold 2^10 of them)
// run as passes added in FP64 through the output.
constexpr int kPassChunks = 512;
template <class F>
void gemm_form(int M, int N, const EmuOperand& A, const EmuOperand& B, const EmuEpilogue& ep,
               int* d_err, cudaStream_t st) {
  prof_begin(kProfEmuGemm, st);
  constexpr int kPass = kPassChunks * F::kChunk;
  for (int k0 = 0; k0 < A.K; k0 += kPass) {
    EmuOperand a = A, b = B;
    EmuEpilogue e = ep;
    a.s = A.s + k0;
    b.s = B.s + k0;
    a.K = b.K = std::min(kPass, A.K - k0);
    if (k0 > 0) e.beta = 1.0;
    gemm_pass<F>(M, N, a, b, e, d_err, st);
  }
  prof_end(kProfEmuGemm, st, 2.0 * M * N * (double)A.K);
}

}  // namespace

void emu_slice(EmuForm f, const EmuSource& src, int rows, int K, EmuOperand& op, cudaStream_t st) {
  RIS_REQUIRE(rows > 0 && K > 0 && op.s && op.e, RIS_ERR_ARG, "emu_slice: bad operand");
  op.rows = rows;
  op.K = K;
  op.ldk = ld8(K);
  op.plane = (long long)rows * op.ldk;
  if (f == kEmu10x6)
    slice_form<Form10x6>(src, rows, K, op, st);
  else
    slice_form<Form9x7>(src, rows, K, op, st);
}

void emu_gemm(EmuForm f, int M, int N, const EmuOperand& A, const EmuOperand& B,
              const EmuEpilogue& ep, int* d_err, cudaStream_t st) {
  if (M <= 0 || N <= 0) return;
  RIS_REQUIRE(A.K == B.K && A.K > 0, RIS_ERR_ARG, "emu_gemm: contraction lengths differ");
  RIS_REQUIRE(A.rows >= M && B.rows >= N, RIS_ERR_ARG, "emu_gemm: operand rows");
  if (f == kEmu10x6)
    gemm_form<Form10x6>(M, N, A, B, ep, d_err, st);
  else
    gemm_form<Form9x7>(M, N, A, B, ep, d_err, st);
}

}  // namespace ris

// Test hooks (declared in include/ris.h): C = A B^T through the emulating
// GEMM for FP64 device operands on the current device.
namespace {
int debug_emu(ris::EmuForm f, int M, int N, int K, const double* A, const double* B, double* C) {
  using namespace ris;
  try {
    if (M <= 0 || N <= 0 || K <= 0 || !A || !B || !C) return (int)RIS_ERR_ARG;
    cudaStream_t st = 0;
    EmuOperand a, b;
    int* err;
    RIS_ALLOC(cudaMalloc(&a.s, sizeof(__half) * emu_size(f, M, K)));
    RIS_ALLOC(cudaMalloc(&b.s, sizeof(__half) * emu_size(f, N, K)));
    RIS_ALLOC(cudaMalloc(&a.e, sizeof(int) * (size_t)M));
    RIS_ALLOC(cudaMalloc(&b.e, sizeof(int) * (size_t)N));
    RIS_ALLOC(cudaMalloc(&err, sizeof(int)));
    RIS_CUDA(cudaMemset(err, 0, sizeof(int)));
    EmuSource sa_, sb_;
    sa_.p = A;
    sb_.p = B;
    sa_.rs = sb_.rs = K;
    emu_slice(f, sa_, M, K, a, st);
    emu_slice(f, sb_, N, K, b, st);
    EmuEpilogue ep;
    ep.c64 = C;
    ep.rs = N;
    ep.cs = 1;
    emu_gemm(f, M, N, a, b, ep, err, st);
    int h_err = 0;
    RIS_CUDA(cudaMemcpy(&h_err, err, sizeof(int), cudaMemcpyDeviceToHost));
    cudaFree(a.s); cudaFree(b.s); cudaFree(a.e); cudaFree(b.e); cudaFree(err);
    return h_err ? (int)RIS_ERR_TIMEOUT : 0;
  } catch (const Error& e) {
    fprintf(stderr, "ris_debug_gemm_f64emu: %s\n", e.msg.c_str());
    return (int)e.code;
  }
}
}  // namespace

extern "C" int ris_debug_gemm_f64emu(int M, int N, int K, const double* A, const double* B, double* C) {
  return debug_emu(ris::kEmu10x6, M, N, K, A, B, C);
}
extern "C" int ris_debug_gemm_f64emu97(int M, int N, int K, const double* A, const double* B, double* C) {
  return debug_emu(ris::kEmu9x7, M, N, K, A, B, C);
}
