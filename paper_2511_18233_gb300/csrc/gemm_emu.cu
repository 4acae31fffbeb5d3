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
// Kernel (persistent, one CTA of 576 threads per SM looping over 128 x BN
// output tiles):
//   warp 0          : producer, 4-stage ring; a stage is K = 16 of all slices
//                     of A (128 rows) and of B (BN rows), one contiguous bulk
//                     copy each (the slicing writes the operands in the layout
//                     of the stages)
//   warp 1          : allocates 512 TMEM columns (S accumulators of BN
//                     columns) and issues the slice products.  The B
//                     slices of a stage lie one after the other, and so do
//                     the accumulators g = p, p + 1, ..., so one
//                     tcgen05.mma of N = (up to 256 / BN) BN multiplies A
//                     slice p with several B slices at once: the 128-row A
//                     slice is read from shared memory once per such group
//                     instead of once per product (14 instructions a stage
//                     instead of 45 at 9 x 7, BN = 48)
//   warps 2-17      : epilogue, one output row and a quarter of the columns
//                     per thread.  A chunk's accumulators are read into
//                     integers first and handed back, so that the next chunk
//                     or tile runs on the tensor cores while the results are
//                     rounded and stored
// FP64 arithmetic is scarce in the epilogue (GB300 issues about 1.7 FP64
// operations per clock per SM, so each per output costs a 128 x 48 tile 3.6k
// cycles, the time of 55 values of k): a single conversion and FMA round the
// result of up to eight chunks, longer sums are rounded with integer
// operations, bit for bit the same.
// Every mbarrier wait is bounded; a timeout sets the error flag, drains what
// the CTA has in flight and frees its tensor memory.
#include <algorithm>
#include <cmath>

#include "gemm_emu.cuh"
#include "tc_ptx.cuh"

namespace ris {

namespace {
using namespace tcx;

constexpr int EBM = 128, EBK = 16, ESTAGES = 4;
constexpr int A_SLICE = EBM * EBK * 2;  // 4 KB
constexpr int TMEM_COLS = 512;
constexpr int EPI_WARPS = 16, ETHREADS = 64 + 32 * EPI_WARPS;

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
  int M, N, K;
  int ntn, tiles1, tiles;  // column tiles (fastest), tiles of a product, all tiles
  int nchunk, cps, ns;  // chunks of the contraction, chunks per slice of it, slices
  const __half* sa;     // digits; elements between K steps
  const __half* sb;
  long long pa, pb;
  const int* ea;
  const int* eb;
  longlong2* ws;   // split contraction: [slice][product][M][N] integer partial sums
  EmuEpilogue ep;
  EmuBatch bt;
  int mode;        // 0: C = x, 1: C = alpha x, 2: C = alpha x + beta C
  int ashift;      // x is taken times 2^ashift, negated if aneg (a power of two
  int aneg;        // as alpha costs no FP64 operation)
  int* err;
};

// bulk copy of contiguous bytes into shared memory (16-byte aligned, a
// multiple of 16 bytes), completing on bar
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(sa(dst)),
      "l"(src), "r"(bytes), "r"(sa(bar))
      : "memory");
}

// Row exponent -> row frame: E_r = 1 + exponent of the largest magnitude, so
// that every |x_rk| < 2^(E_r) (0 for a row of zeros).
__device__ __forceinline__ int row_frame(int lead) { return lead == kEmuNoLead ? 0 : lead + 1; }
__device__ __forceinline__ bool row_bad(int lead) { return lead >= kEmuLeadBad; }
__device__ __forceinline__ int lead_exp(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ef = (int)((b >> 52) & 0x7FF);
  if (ef) return ef - 1023;
  const unsigned long long m = b & 0xFFFFFFFFFFFFFull;
  return m ? -1011 - __clzll(m) : kEmuNoLead;  // -1074 + (63 - clz)
}

__device__ __forceinline__ long long emu_off(int i, int in, long long ld, long long s) {
  return in > 0 ? (long long)(i / in) * ld + (long long)(i % in) * s : (long long)i * s;
}

// C = x, or out of line C = alpha x (+ beta C), so that no FP64 operation is
// predicated into the plain store
__device__ __noinline__ void store_scaled(double* p, double x, int mode, double alpha, double beta) {
  *p = mode == 2 ? fma(alpha, x, beta * *p) : alpha * x;
}
__device__ __forceinline__ void store_out(double* p, double x, int mode, double alpha, double beta) {
  if (mode == 0)
    *p = x;
  else
    store_scaled(p, x, mode, alpha, beta);
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

constexpr int kQuickK = 112;  // EmuAcc::quick from this contraction length on
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
  // The same from at most kQuickChunks chunks (|hi + lo 2^-35| < 2^50) with two
  // FP64 operations: lo's upper bits are carried into hi, which is turned into
  // FP64 by its bit pattern and one subtraction, and one FMA adds the lower 35
  // bits and rounds.  They enter as the bit pattern of 2^52 + bits, the 2^52
  // having been taken from hi.  emu_round's hundred integer instructions in a
  // row take longer (21504 x 512 over 142, an exchange density of C20H22: 165
  // -> 148 us), but below kQuickK the products of a tile are done before its
  // FP64 operations (2982 x 512 over 71: 27 -> 30 us), so it stays there.
  static constexpr int kQuickChunks = 8;
  __device__ __forceinline__ double quick(int e) const {
    const long long h = hi + (lo >> kShift) - (1ll << 17);
    const double lm = __longlong_as_double(0x4330000000000000ll | (lo & ((1ll << kShift) - 1)));
    const double hd = __longlong_as_double(0x4338000000000000ll + h) - 6755399441055744.0;  // 1.5 2^52
    const double x = fma(hd, 34359738368.0, lm);
    const int sh = e - 2 * Form9x7::kFrac + 56;
    const long long b = __double_as_longlong(x);
    const int ex = (int)((b >> 52) & 0x7FF) + sh;
    if ((b << 1) == 0) return x;
    if (ex < 1 || ex > 2046) return ldexp(x, sh);
    return __longlong_as_double(b + ((long long)sh << 52));
  }
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
  static constexpr int kQuickChunks = 0;
  __device__ __forceinline__ double quick(int) const { return s; }
};

template <class F, int bn>
__global__ void __launch_bounds__(ETHREADS, 1) k_emu_gemm(EmuArgs args) {
  constexpr int S = F::S;
  constexpr int kSteps = F::kChunk / EBK;
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
  const int items = args.tiles * args.ns;

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

  // work item w: tile w % tiles, contraction slice w / tiles
  // (the two feeding warps run their loops with all lanes and elect one for
  // the copies and products: counters and descriptors then live in uniform
  // registers, where those instructions take them from)
  if (warp == 0) {
    // producer
    int it = 0;  // stages issued
    bool stop = false;  // warp-uniform
    for (int w = blockIdx.x; w < items && !stop; w += gridDim.x) {
      const int t = w % args.tiles, c0 = (w / args.tiles) * args.cps;
      const int pr = t / args.tiles1, t1 = t - pr * args.tiles1;
      const int n0 = (t1 % args.ntn) * bn + args.bt.b[pr], m0 = (t1 / args.ntn) * EBM + args.bt.a[pr];
      const int s0 = c0 * kSteps;
      const int s1 = min((args.K + EBK - 1) / EBK, (c0 + args.cps) * kSteps);
      const __half* ga = args.sa + (size_t)s0 * args.pa + (size_t)m0 * (16 * S);
      const __half* gb = args.sb + (size_t)s0 * args.pb + (size_t)n0 * (16 * S);
      for (int i = s0; i < s1; i++, it++) {
        const int s = it % ESTAGES;
        if (it >= ESTAGES && !mbar_wait(&empty[s], ((it / ESTAGES) - 1) & 1)) *abort_flag = 1;
        stop = __any_sync(0xffffffffu, *abort_flag);
        if (stop) break;
        if (elect_one()) {
          uint8_t* st = smem + s * Tile<F>::kStage;
          mbar_expect_tx(&full[s], Tile<F>::kABytes + S * bn * EBK * 2);
          bulk_load(st, ga, Tile<F>::kABytes, &full[s]);
          bulk_load(st + Tile<F>::kABytes, gb, S * bn * EBK * 2, &full[s]);
        }
        __syncwarp();
        ga += args.pa;
        gb += args.pb;
      }
    }
    // no copy is left in flight
    for (int i = (it > ESTAGES ? it - ESTAGES : 0); i < it; i++)
      mbar_wait(&full[i % ESTAGES], (i / ESTAGES) & 1);
  } else if (warp == 1) {
    // MMA issuer: slice products p + q < S into accumulator p + q
    constexpr int per = 256 / bn;  // B slices per instruction
    int it = 0, nch = 0;           // stages, chunks issued
    bool stop = false;             // warp-uniform
    for (int w = blockIdx.x; w < items && !stop; w += gridDim.x) {
      const int c0 = (w / args.tiles) * args.cps;
      const int s0 = c0 * kSteps;
      const int s1 = min((args.K + EBK - 1) / EBK, (c0 + args.cps) * kSteps);
      for (int i = s0; i < s1; i++, it++) {
        const int s = it % ESTAGES, in = i % kSteps;
        // a new chunk: the epilogue must have read the previous one
        if (in == 0) {
          if (nch > 0 && !mbar_wait(acc_empty, (nch - 1) & 1)) *abort_flag = 1;
          nch++;
        }
        stop = __any_sync(0xffffffffu, *abort_flag);
        if (!stop && !mbar_wait(&full[s], (it / ESTAGES) & 1)) *abort_flag = 1;
        stop = __any_sync(0xffffffffu, *abort_flag);
        if (stop) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        // (fully unrolled: descriptors, columns and shapes are the stage's
        // base plus constants.  One thread feeds the tensor core, and an
        // instruction of N = 240 lasts about 120 cycles)
        const uint64_t d0 = desc_sw32(smem + s * Tile<F>::kStage);
        const uint32_t acc = in > 0 ? 1u : 0u;
        if (elect_one()) {
          auto mma = [&](int p, int g0, int g1, uint32_t on) {  // accumulators g0 .. g1 - 1
            mma_f16(tmem + (uint32_t)(g0 * bn), d0 + (p * A_SLICE >> 4),
                    d0 + ((Tile<F>::kABytes + (g0 - p) * bn * EBK * 2) >> 4), idesc_f16((g1 - g0) * bn), on);
          };
          if (per < S && acc) {
            // accumulators below and above `per` in turn, so that an
            // instruction does not start on columns that the one before it is
            // still writing (3% of the loop)
#pragma unroll
            for (int x = 0; x < S; x++) {
              const int p = S - 1 - x;
              mma(p, p > per ? p : per, S, 1u);
              if (x < per) mma(x, x, per, 1u);
            }
          } else {  // the first step clears the accumulators
#pragma unroll
            for (int p = 0; p < S; p++) {
#pragma unroll
              for (int g = p; g < S; g += per) mma(p, g, g + per < S ? g + per : S, p > 0 ? 1u : acc);
            }
          }
          mma_commit(&empty[s]);
          if (in == kSteps - 1 || i == s1 - 1) mma_commit(acc_full);
        }
        __syncwarp();
      }
    }
    // nothing is left in flight when the tensor memory is freed, whatever happened
    if (elect_one()) mma_commit(done);
    __syncwarp();
    if (!mbar_wait(done, 0)) *abort_flag = 1;
  } else {
    // epilogue: row = TMEM lane of this warp's quadrant; the four warps of a
    // quadrant take bn / 4 columns each, read four at a time
    constexpr int ncol = bn / 4, NB = ncol / 4;  // blocks of four columns
    const int quad = warp & 3, cg = (warp - 2) >> 2;
    const uint32_t lane_base = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(cg * ncol);
    const EmuEpilogue& ep = args.ep;
    int nch = 0;
    bool good = true;
    for (int w = blockIdx.x; w < items && good; w += gridDim.x) {
      const int t = w % args.tiles, z = w / args.tiles, c0 = z * args.cps;
      const int nc = min(args.nchunk, c0 + args.cps) - c0;
      const int pr = t / args.tiles1, t1 = t - pr * args.tiles1;
      const int n0 = (t1 % args.ntn) * bn + cg * ncol;
      const int row = (t1 / args.ntn) * EBM + quad * 32 + lane;
      const bool live = row < args.M;
      const int lr = live ? args.ea[row + args.bt.a[pr]] : kEmuNoLead;
      const int er = row_frame(lr);
      // lane j < ncol holds column j's exponent and output offset
      const int mc = n0 + lane;
      const int lc = (lane < ncol && mc < args.N) ? args.eb[mc + args.bt.b[pr]] : kEmuNoLead;
      long long coff = 0;
      int lidx = 0;
      if (lane < ncol && mc < args.N) {
        coff = emu_off(mc, ep.cin, ep.cld, ep.cs);
        if (ep.lead) lidx = ((mc / ep.lcd) % ep.lcm) * ep.lcs;
      }
      EmuAcc<F> acc[NB][4];
#pragma unroll
      for (int b = 0; b < NB; b++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[b][j].zero();
      for (int ch = 0; ch < nc; ch++, nch++) {
        if (!mbar_wait(acc_full, nch & 1)) *abort_flag = 1;
        good = !__any_sync(0xffffffffu, *abort_flag);
        if (!good) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int b = 0; b < NB; b++) {
          float v[S][4];
#pragma unroll
          for (int g = 0; g < S; g++) tmem_ld4(lane_base + (uint32_t)(g * bn + 4 * b), v[g]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int j = 0; j < 4; j++) {
            float u[S];
#pragma unroll
            for (int g = 0; g < S; g++) u[g] = v[g][j];
            int e = 0;
            if (!F::kBalanced) e = er + row_frame(__shfl_sync(0xffffffffu, lc, 4 * b + j));
            acc[b][j].add(u, e, ch == 0);
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty);
      }
      if (!good) break;
      double* prow = ep.c64 + args.bt.c[pr] + emu_off(row, ep.rin, ep.rld, ep.rs);
      const int lrow = ep.lead ? ((row / ep.lrd) % ep.lrm) * ep.lrs : 0;
      const bool quick = args.cps <= EmuAcc<F>::kQuickChunks && args.K >= kQuickK;
      const bool bad = __any_sync(0xffffffffu, row_bad(lr) || row_bad(lc));
      const bool one_row = __all_sync(0xffffffffu, lrow == __shfl_sync(0xffffffffu, lrow, 0) && live);
      int lcur = -1, lmax = kEmuNoLead;
      auto flush = [&] {  // the running exponent of lead column lcur
        if (lcur < 0) return;
        if (one_row) {
          const int m = __reduce_max_sync(0xffffffffu, lmax);
          if (lane == 0) atomicMax(ep.lead + lrow + lcur, m);
        } else if (live) {
          atomicMax(ep.lead + lrow + lcur, lmax);
        }
        lmax = kEmuNoLead;
      };
#pragma unroll
      for (int b = 0; b < NB; b++) {
#pragma unroll
        for (int j = 0; j < 4; j++) {
          const int jc = 4 * b + j;
          if (n0 + jc >= args.N) continue;  // warp-uniform
          const int lcj = __shfl_sync(0xffffffffu, lc, jc);
          const long long cj = ep.cin > 0 ? __shfl_sync(0xffffffffu, coff, jc) : (long long)(n0 + jc) * ep.cs;
          if constexpr (F::kBalanced) {
            if (args.ws) {  // one slice of the contraction: integer partial sums
              longlong2 s;
              s.x = acc[b][j].hi;
              s.y = acc[b][j].lo;
              if (live) args.ws[((size_t)(z * args.bt.n + pr) * args.M + row) * args.N + n0 + jc] = s;
              continue;
            }
          }
          const int e = er + row_frame(lcj) + args.ashift;
          double x = quick ? acc[b][j].quick(e) : acc[b][j].result(e);
          if (args.aneg) x = __longlong_as_double(__double_as_longlong(x) ^ (1ll << 63));
          if (bad && (row_bad(lr) || row_bad(lcj))) x = __longlong_as_double(0x7ff8000000000000ll);
          if (ep.lead) {
            const int li = __shfl_sync(0xffffffffu, lidx, jc);
            if (li != lcur) {
              flush();
              lcur = li;
            }
            lmax = max(lmax, lead_exp(x));
          }
          if (!live) continue;
          double* p = prow + cj;
          store_out(p, x, args.mode, ep.alpha, ep.beta);
        }
      }
      if (ep.lead) flush();
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
  const long long mn = (long long)args.M * args.N * args.bt.n;
  if (t >= mn) return;
  long long hi = 0, lo = 0;
  for (int z = 0; z < nsplit; z++) {
    const longlong2 w = args.ws[(size_t)z * mn + t];
    hi += w.x;
    lo += w.y;
  }
  const int pr = (int)(t / ((long long)args.M * args.N));
  const long long q = t - (long long)pr * args.M * args.N;
  const int row = (int)(q / args.N), col = (int)(q % args.N);
  const int lr = args.ea[row + args.bt.a[pr]], lc = args.eb[col + args.bt.b[pr]];
  double x = EmuAcc<Form9x7>::value(hi, lo, row_frame(lr) + row_frame(lc) + args.ashift);
  if (args.aneg) x = __longlong_as_double(__double_as_longlong(x) ^ (1ll << 63));
  if (row_bad(lr) || row_bad(lc)) x = __longlong_as_double(0x7ff8000000000000ll);
  const EmuEpilogue& ep = args.ep;
  if (ep.lead)
    atomicMax(ep.lead + ((row / ep.lrd) % ep.lrm) * ep.lrs + ((col / ep.lcd) % ep.lcm) * ep.lcs,
              lead_exp(x));
  double* p = ep.c64 + args.bt.c[pr] + emu_off(row, ep.rin, ep.rld, ep.rs) + emu_off(col, ep.cin, ep.cld, ep.cs);
  store_out(p, x, args.mode, ep.alpha, ep.beta);
}

// ------------------------------------------------------------------ slicing
// Digits of elements in their row frame, on the integer pipe: a fixed-point
// number per element, then word(p) = digits p of two of them as an FP16 pair.
// A digit u + bias is turned into FP16 by or-ing it into the significand of
// 1024 and subtracting 1024 + bias.
__device__ __forceinline__ unsigned sub_half2(unsigned w, unsigned short bias) {
  const __half2 b = __halves2half2(__ushort_as_half(bias), __ushort_as_half(bias));
  const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&w), b);
  return *reinterpret_cast<const unsigned*>(&h);
}
// |x| = m 2^q
__device__ __forceinline__ unsigned long long split_double(double x, int& q) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ef = (int)((b >> 52) & 0x7FF);
  const unsigned long long m = b & 0xFFFFFFFFFFFFFull;
  q = ef ? ef - 1075 : -1074;
  return ef ? m | (1ull << 52) : m;
}
template <class F>
struct Fixed;
template <>
struct Fixed<Form10x6> {
  // X = floor(|x| 2^(60 - E)), d_p = its bits [60 - 6(p+1), 60 - 6p), signed like x
  unsigned long long X;
  unsigned sign;
  __device__ __forceinline__ void set(double x, int E) {
    int q;
    const unsigned long long m = split_double(x, q);
    sign = (unsigned)((unsigned long long)__double_as_longlong(x) >> 63) << 15;
    const int sh = q + Form10x6::kFrac - E;
    X = sh >= 0 ? (m << sh) : (sh <= -64 ? 0ull : (m >> -sh));
  }
  static __device__ __forceinline__ unsigned word(const Fixed& a, const Fixed& b, int p) {
    const int sh = 60 - 6 * (p + 1);
    const unsigned w = ((unsigned)(a.X >> sh) & 63u) | (((unsigned)(b.X >> sh) & 63u) << 16) | 0x64006400u;
    return sub_half2(w, 0x6400) ^ (a.sign | (b.sign << 16));
  }
};
template <>
struct Fixed<Form9x7> {
  // X = round(x 2^(62 - E)), |X| <= 2^62, plus 64 in each of the eight lower
  // digits: digit p is then a 7-bit field less 64 and the top digit, in
  // [-64, 64], what is left above
  long long X;
  __device__ __forceinline__ void set(double x, int E) {
    constexpr long long kBias = 64ll * (((1ll << 56) - 1) / 127);
    int q;
    const unsigned long long m = split_double(x, q);
    const int sh = q + Form9x7::kFrac - E;
    const unsigned long long a =
        sh >= 0 ? (m << sh) : (sh <= -60 ? 0ull : ((m >> (-sh - 1)) + 1) >> 1);
    X = (__double_as_longlong(x) < 0 ? -(long long)a : (long long)a) + kBias;
  }
  static __device__ __forceinline__ unsigned word(const Fixed& a, const Fixed& b, int p) {
    unsigned w;
    if (p == 0) {
      w = (unsigned)((int)(a.X >> 56) + 64) | ((unsigned)((int)(b.X >> 56) + 64) << 16);
    } else {
      const int sh = 7 * (8 - p);
      w = ((unsigned)(a.X >> sh) & 127u) | (((unsigned)(b.X >> sh) & 127u) << 16);
    }
    return sub_half2(w | 0x64006400u, 0x6440);  // 1024 + 64
  }
};

// eight consecutive digits per slice of one row (half of a K step): 16-byte
// stores, o = the K step's digits
template <class F>
__device__ __forceinline__ void put8(const double (&x)[8], int lead, __half* o, int rb, int r,
                                     int half) {
  Fixed<F> f[8];
  const int E = row_bad(lead) ? 0 : row_frame(lead);  // digits of a bad row are not used
#pragma unroll
  for (int i = 0; i < 8; i++) f[i].set(row_bad(lead) ? 0.0 : x[i], E);
  const int b = r / rb, i = r - b * rb;
  o += (size_t)b * (F::S * 16 * rb) + (i >> 3) * 128 + (i & 7) * 16 + ((half ^ ((i >> 2) & 1)) << 3);
#pragma unroll
  for (int p = 0; p < F::S; p++)
    *reinterpret_cast<uint4*>(o + p * (16 * rb)) =
        make_uint4(Fixed<F>::word(f[0], f[1], p), Fixed<F>::word(f[2], f[3], p),
                   Fixed<F>::word(f[4], f[5], p), Fixed<F>::word(f[6], f[7], p));
}

__device__ __forceinline__ bool src_row(const EmuSource& src, int r, int rows, long long& off) {
  if (r >= rows) return false;
  long long base = 0;
  if (src.bin > 0) {
    const int blk = r / src.bin;
    r -= blk * src.bin;
    base = (long long)blk * src.bld;
    if (r >= src.bvalid) {
      off = base;
      return false;
    }
  }
  off = base + emu_off(r, src.rin, src.rld, src.rs);
  return src.rvalid == 0 || r % src.rin < src.rvalid;
}

// Row exponents of rows contiguous in k, one CTA per row.
__global__ void __launch_bounds__(256) k_emu_lead(EmuSource src, int rows, int K, int* __restrict__ E) {
  __shared__ int red[8];
  long long off = 0;
  const int r = blockIdx.x;
  int m = kEmuNoLead;
  if (src_row(src, r, rows, off))
    for (int k = threadIdx.x; k < K; k += 256) m = max(m, lead_exp(src.p[off + k]));
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; w++) m = max(m, red[w]);
    E[r] = m;
  }
}

// Rows contiguous in k: 16 rows per CTA; lane = (row, half of a K step), one K
// step per warp, so that a warp's stores fill two row groups of a slice.  With
// LEAD the CTA first finds its rows' exponents (two rows per warp; the second
// read comes from L2: one pass over DRAM) and takes every K step; otherwise E
// holds them and the K steps are spread over blockIdx.y.
template <class F, bool LEAD>
__global__ void __launch_bounds__(256) k_emu_slice_rows(EmuSource src, int rows, int K,
                                                        int* __restrict__ E, __half* __restrict__ out,
                                                        int rb, int prows) {
  __shared__ int ex[16];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, r0 = blockIdx.x * 16;
  if (LEAD) {
#pragma unroll
    for (int h = 0; h < 2; h++) {
      const int r = r0 + 2 * warp + h;
      long long off = 0;
      int m = kEmuNoLead;
      if (src_row(src, r, rows, off))
        for (int k = lane; k < K; k += 32) m = max(m, lead_exp(src.p[off + k]));
      m = __reduce_max_sync(0xffffffffu, m);
      if (lane == 0) {
        ex[2 * warp + h] = m;
        if (r < rows) E[r] = m;
      }
    }
    __syncthreads();
  }
  const int r = r0 + (lane >> 1), half = lane & 1;
  if (r >= prows) return;
  long long off = 0;
  const bool on = src_row(src, r, rows, off);
  const int lead = LEAD ? ex[lane >> 1] : (r < rows ? E[r] : kEmuNoLead);
  const double* x = src.p + off;
  const int nk = (K + 15) / 16;
  for (int s = blockIdx.y * 8 + warp; s < nk; s += gridDim.y * 8) {
    const int k = s * 16 + half * 8;
    double v[8];
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = (on && k + i < K) ? x[k + i] : 0.0;
    put8<F>(v, lead, out + (size_t)s * F::S * 16 * prows, rb, r, half);
  }
}

// Rows strided in k (consecutive rows adjacent in memory): 32 rows per CTA,
// lanes along the rows for the reads, transposed through shared memory.  LEAD
// and blockIdx.y as in k_emu_slice_rows.
template <class F, bool LEAD>
__global__ void __launch_bounds__(256) k_emu_slice_cols(EmuSource src, int rows, int K,
                                                        int* __restrict__ E, __half* __restrict__ out,
                                                        int rb, int prows) {
  __shared__ double tile[64][33];  // [k][r]
  __shared__ int red[8][32];
  const int r0 = blockIdx.x * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  long long off = 0;
  const bool on = src_row(src, r0 + tx, rows, off);
  const double* x = src.p + off;
  if (LEAD) {
    int m = kEmuNoLead;
    if (on)
#pragma unroll 4
      for (int k = ty; k < K; k += 8) m = max(m, lead_exp(x[(size_t)k * src.ks]));
    red[ty][tx] = m;
    __syncthreads();
    if (ty == 0) {
      for (int y = 1; y < 8; y++) m = max(m, red[y][tx]);
      red[0][tx] = m;
      if (r0 + tx < rows) E[r0 + tx] = m;
    }
  } else if (ty == 0) {
    red[0][tx] = r0 + tx < rows ? E[r0 + tx] : kEmuNoLead;
  }
  // warp = (K step of the tile, rows 0-15 / 16-31), lane = (row, half of the K step)
  const int rr = (ty & 1) * 16 + (tx >> 1), ks = ty >> 1, half = tx & 1;
  const int nk = (K + 15) / 16;
  for (int s0 = blockIdx.y * 4; s0 < nk; s0 += gridDim.y * 4) {
    __syncthreads();
#pragma unroll
    for (int kk = ty; kk < 64; kk += 8)
      tile[kk][tx] = (on && s0 * 16 + kk < K) ? x[(size_t)(s0 * 16 + kk) * src.ks] : 0.0;
    __syncthreads();
    if (s0 + ks >= nk || r0 + rr >= prows) continue;
    double v[8];
#pragma unroll
    for (int i = 0; i < 8; i++) v[i] = tile[ks * 16 + half * 8 + i][rr];
    put8<F>(v, red[0][rr], out + (size_t)(s0 + ks) * F::S * 16 * prows, rb, r0 + rr, half);
  }
}

template <class F>
void slice_form(const EmuSource& src, int rows, int K, EmuOperand& op, cudaStream_t st, bool have_lead) {
  const int nk = cdiv(K, 16), prows = (int)op.blocks * op.rb;  // padded rows are cut as zeros
  if (src.ks != 1) {
    if (have_lead) {
      const int ny = std::min(cdiv(nk, 4), std::max(1, cdiv(8 * 152, cdiv(prows, 32))));
      k_emu_slice_cols<F, false><<<dim3(cdiv(prows, 32), ny), 256, 0, st>>>(src, rows, K, op.e, op.s, op.rb, prows);
    } else {
      k_emu_slice_cols<F, true><<<cdiv(prows, 32), 256, 0, st>>>(src, rows, K, op.e, op.s, op.rb, prows);
    }
  } else if (have_lead || K >= 2048) {
    // few long rows: exponents first, one row per CTA, so that a few hundred
    // rows fill the device
    if (!have_lead) {
      k_emu_lead<<<rows, 256, 0, st>>>(src, rows, K, op.e);
      RIS_CHECK_LAUNCH();
    }
    const int ny = std::min(cdiv(nk, 8), std::max(1, cdiv(8 * 152, cdiv(prows, 16))));
    k_emu_slice_rows<F, false><<<dim3(cdiv(prows, 16), ny), 256, 0, st>>>(src, rows, K, op.e, op.s, op.rb, prows);
  } else {
    k_emu_slice_rows<F, true><<<cdiv(prows, 16), 256, 0, st>>>(src, rows, K, op.e, op.s, op.rb, prows);
  }
  RIS_CHECK_LAUNCH();
}

template <class F>
void gemm_pass(int M, int N, const EmuOperand& A, const EmuOperand& B, const EmuEpilogue& ep,
               int* d_err, cudaStream_t st, const EmuBatch& bt) {
  EmuArgs a;
  a.M = M;
  a.N = N;
  a.K = A.K;
  const int bn = B.rb;
  a.ntn = cdiv(N, bn);
  a.nchunk = cdiv(A.K, F::kChunk);
  RIS_REQUIRE((((uintptr_t)A.s | (uintptr_t)B.s) & 15) == 0, RIS_ERR_ARG, "emu_gemm: slices not 16-byte aligned");
  a.sa = A.s;
  a.sb = B.s;
  a.pa = A.blocks * A.rb * (16 * F::S);
  a.pb = B.blocks * B.rb * (16 * F::S);
  a.ea = A.e;
  a.eb = B.e;
  a.ws = nullptr;
  a.ep = ep;
  a.mode = ep.beta != 0.0 ? 2 : ep.alpha != 1.0 ? 1 : 0;
  a.ashift = a.aneg = 0;
  int ax = 0;
  if (F::kBalanced && a.mode == 1 && std::fabs(std::frexp(ep.alpha, &ax)) == 0.5 && std::abs(ax) < 256) {
    a.mode = 0;
    a.ashift = ax - 1;
    a.aneg = ep.alpha < 0.0;
  }
  a.err = d_err;
  a.bt = bt;
  a.tiles1 = a.ntn * cdiv(M, EBM);
  const long long tiles = (long long)a.ntn * cdiv(M, EBM) * bt.n;
  RIS_REQUIRE(tiles * 64 < (1LL << 31), RIS_ERR_ARG, "emu_gemm: too many tiles");
  a.tiles = (int)tiles;
  // slices of a long contraction: the number of chunk rounds of the busiest
  // SM, plus about a chunk's time for each CTA's start and end
  int ns = 1;
  if (F::kBalanced && a.nchunk > 1) {
    long long best = -1;
    for (int s = 1; s <= std::min(a.nchunk, 64); s++) {
      const int cps = cdiv(a.nchunk, s);
      if (cdiv(a.nchunk, cps) != s) continue;
      if (s > 1 && (double)s * M * N * bt.n * sizeof(longlong2) > 1e9) break;
      const long long cost = (long long)cdiv(tiles * s, 152) * (2 * cps + 1);
      if (best < 0 || cost < best) {
        best = cost;
        ns = s;
      }
    }
  }
  a.cps = cdiv(a.nchunk, ns);
  a.ns = ns;
  MemTrack* tr = nullptr;
  const size_t wsb = (size_t)ns * M * N * bt.n * sizeof(longlong2);
  if (ns > 1) a.ws = (longlong2*)dev_alloc(wsb, st, &tr);
  auto kern = bn == 48 ? k_emu_gemm<F, 48> : bn == 32 ? k_emu_gemm<F, 32> : k_emu_gemm<F, 16>;
  ensure_smem_attr((const void*)kern, Tile<F>::kSmem);
  kern<<<(unsigned)std::min<long long>(tiles * ns, 152), ETHREADS, Tile<F>::kSmem, st>>>(a);
  RIS_CHECK_LAUNCH();
  if (ns > 1) {
    k_emu_finish<<<cdiv((long long)M * N * bt.n, 256), 256, 0, st>>>(a, ns);
    RIS_CHECK_LAUNCH();
    dev_free(a.ws, wsb, st, tr);
  }
}

// Contractions beyond kPassChunks chunks (the 64-bit sums hold 2^10 of them)
// run as passes added in FP64 through the output.
constexpr int kPassChunks = 512;
template <class F>
void gemm_form(int M, int N, const EmuOperand& A, const EmuOperand& B, const EmuEpilogue& ep,
               int* d_err, cudaStream_t st, const EmuBatch& bt) {
  prof_begin(kProfEmuGemm, st);
  constexpr int kPass = kPassChunks * F::kChunk;
  for (int k0 = 0; k0 < A.K; k0 += kPass) {
    EmuOperand a = A, b = B;
    EmuEpilogue e = ep;
    a.s = A.s + (size_t)(k0 / EBK) * F::S * 16 * A.blocks * A.rb;
    b.s = B.s + (size_t)(k0 / EBK) * F::S * 16 * B.blocks * B.rb;
    a.K = b.K = std::min(kPass, A.K - k0);
    if (k0 > 0) e.beta = 1.0;
    gemm_pass<F>(M, N, a, b, e, d_err, st, bt);
  }
  prof_end(kProfEmuGemm, st, 2.0 * M * N * (double)A.K * bt.n);
}

}  // namespace

// Tile width for N columns: a stage brings (128 + BN) rows of digits through
// shared memory whatever the products, so the total over the column tiles is
// taken least; ties go to the wider tile.
int emu_cols(int N) {
  int bn = 48;
  for (int c = 48; c >= 16; c -= 16)
    if ((long long)cdiv(N, c) * (EBM + c) < (long long)cdiv(N, bn) * (EBM + bn)) bn = c;
  return bn;
}

void emu_slice(EmuForm f, const EmuSource& src, int rows, int K, EmuOperand& op, cudaStream_t st,
               bool have_lead) {
  RIS_REQUIRE(rows > 0 && K > 0 && op.s && op.e, RIS_ERR_ARG, "emu_slice: bad operand");
  op.rows = rows;
  op.K = K;
  RIS_REQUIRE(op.rb > 0 && op.rb % 8 == 0, RIS_ERR_ARG, "emu_slice: row block");
  op.blocks = cdiv(rows, op.rb);
  op.slices = emu_slices(f);
  if (f == kEmu10x6)
    slice_form<Form10x6>(src, rows, K, op, st, have_lead);
  else
    slice_form<Form9x7>(src, rows, K, op, st, have_lead);
}

void emu_gemm(EmuForm f, int M, int N, const EmuOperand& A, const EmuOperand& B,
              const EmuEpilogue& ep, int* d_err, cudaStream_t st, const EmuBatch& bt) {
  if (M <= 0 || N <= 0) return;
  RIS_REQUIRE(A.K == B.K && A.K > 0, RIS_ERR_ARG, "emu_gemm: contraction lengths differ");
  RIS_REQUIRE(bt.n >= 1 && bt.n <= 8 && (bt.n == 1 || !ep.lead), RIS_ERR_ARG, "emu_gemm: batch");
  // `lead` takes the exponents of A B^T itself, of one pass
  RIS_REQUIRE(!ep.lead || (ep.alpha == 1.0 && ep.beta == 0.0 && A.K <= kPassChunks * Form9x7::kChunk), RIS_ERR_ARG,
              "emu_gemm: row exponents of a scaled, summed or very long product");
  for (int p = 0; p < bt.n; p++) {
    RIS_REQUIRE(A.rows - bt.a[p] >= M && B.rows - bt.b[p] >= N, RIS_ERR_ARG, "emu_gemm: operand rows");
    RIS_REQUIRE(bt.a[p] % kEmuRowsA == 0 && bt.b[p] % B.rb == 0, RIS_ERR_ARG, "emu_gemm: batch rows");
  }
  RIS_REQUIRE(A.rb == kEmuRowsA && (B.rb == 48 || B.rb == 32 || B.rb == 16), RIS_ERR_ARG,
              "emu_gemm: operand row blocks");
  RIS_REQUIRE(A.slices == emu_slices(f) && B.slices == A.slices, RIS_ERR_ARG, "emu_gemm: operand form");
  if (f == kEmu10x6)
    gemm_form<Form10x6>(M, N, A, B, ep, d_err, st, bt);
  else
    gemm_form<Form9x7>(M, N, A, B, ep, d_err, st, bt);
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
    a.rb = kEmuRowsA;
    b.rb = emu_cols(N);
    RIS_ALLOC(cudaMalloc(&a.s, sizeof(__half) * emu_size(f, M, K, a.rb)));
    RIS_ALLOC(cudaMalloc(&b.s, sizeof(__half) * emu_size(f, N, K, b.rb)));
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
