// FP64-accurate matrix products on the FP16 tensor cores of sm_103a by exact
// splitting of the operands into small-integer slices (Ozaki's scheme).
#pragma once
#include <cuda_fp16.h>

#include "common.cuh"

namespace ris {

// Slicing forms.  A row r of an operand (contraction index k) is written in
// one fixed-point frame per row, 2^(E_r) above its largest magnitude, and cut
// into digits:
//   kEmu10x6  ten 6-bit slices, digits 0 .. 63 with the element's sign (60
//             bits, truncated): the Coulomb transforms of the mixed form
//   kEmu9x7   nine 7-bit slices, balanced digits -64 .. 64 (62 bits and sign,
//             rounded to nearest): the exchange products of the FP64 form.
//             45 slice products instead of 55, and a frame 9 bits finer than
//             an FP64 significand, so that a row's small elements beside one
//             nine bits larger still keep FP64's relative precision.  Below
//             that an element keeps fewer than 53 bits (none from 2^-62 of the
//             row's largest on), and products of digits p + q >= 9 are
//             dropped: normwise, against max_k|A_rk| max_k|B_ck|, errors are
//             below FP64's, element by element (a row whose large elements
//             meet zeros) they are not
enum EmuForm { kEmu10x6 = 0, kEmu9x7 = 1 };
constexpr int emu_slices(EmuForm f) { return f == kEmu10x6 ? 10 : 9; }

// A sliced operand: FP16 integer digits in the layout in which the GEMM's
// stages lie in shared memory, so that a stage is one contiguous copy per
// operand:
//   [K step of 16][block of rb rows][slice][group of 8 rows][8 rows x 32 bytes]
// with the two 16-byte halves of rows 4..7 of a group exchanged (the 32-byte
// swizzle of the tensor core's operand tiles), zero past K and past the rows;
// and per row the exponent of its largest magnitude (kEmuNoLead for a row of
// zeros; at least kEmuLeadBad for a row that holds an infinity or a NaN: every
// product with it is NaN).  rb is the GEMM's tile edge: kEmuRowsA for the left
// operand, emu_cols(N) for the right one.
constexpr int kEmuNoLead = (int)0x80808080;  // set by a byte fill of 0x80
constexpr int kEmuLeadBad = 1024;
constexpr int kEmuRowsA = 128;
int emu_cols(int N);
struct EmuOperand {
  __half* s = nullptr;
  int* e = nullptr;
  int rows = 0, K = 0;
  int rb = 0;
  long long blocks = 0;  // row blocks
  int slices = 0;
};

inline int emu_pad(int n, int rb) { return (n + rb - 1) / rb * rb; }
// halves an operand of the form needs (ints: rows)
inline size_t emu_size(EmuForm f, long long rows, int K, int rb) {
  return (size_t)((K + 15) / 16) * emu_slices(f) * ((rows + rb - 1) / rb * rb) * 16;
}

// Source placement: element (r, k) of an operand at src[row(r) + k * ks] with
// row(r) = (r / rin) * rld + (r % rin) * rs (rin = 0: r * rs); rows with
// r % rin >= rvalid are zero (rvalid = 0: none).  With bin > 0 the rows come in
// blocks of bin: block r / bin starts at (r / bin) * bld, its rows from bvalid
// on are zero and the others are placed as above.
struct EmuSource {
  const double* p = nullptr;
  long long rs = 0, ks = 1;
  int rin = 0;
  long long rld = 0;
  int rvalid = 0;
  int bin = 0, bvalid = 0;
  long long bld = 0;
};

// Slices src (rows x K) into op (op.rb set; op.s / op.e hold emu_size / rows
// elements).
// have_lead: op.e already holds the row exponents (EmuEpilogue::lead).
void emu_slice(EmuForm f, const EmuSource& src, int rows, int K, EmuOperand& op, cudaStream_t st,
               bool have_lead = false);

// Output placement: element (r, c) goes to
//   c64[(r / rin) * rld + (r % rin) * rs + (c / cin) * cld + (c % cin) * cs]
// (rin, cin = 0: no blocking), as alpha * (A B^T)_rc + beta * c64[...].
struct EmuEpilogue {
  double* c64 = nullptr;
  int rin = 0, cin = 0;
  long long rld = 0, rs = 0, cld = 0, cs = 1;
  double alpha = 1.0, beta = 0.0;
  // lead: also the largest exponent of the outputs that the next product reads
  // as one row, by atomic maximum into
  //   lead[((r / lrd) % lrm) * lrs + ((c / lcd) % lcm) * lcs]
  // (filled with kEmuNoLead before), so that slicing them needs no pass of its
  // own for the row exponents; alpha 1, beta 0 and K of one pass only (229376)
  int* lead = nullptr;
  int lrd = 1, lrm = 1, lrs = 0, lcd = 1, lcm = 1, lcs = 0;
  void lead_rows(int d, int m, int s) { lrd = d; lrm = m; lrs = s; }
  void lead_cols(int d, int m, int s) { lcd = d; lcm = m; lcs = s; }
};

// Products that share a launch: product p takes A from row a[p] (a multiple of
// kEmuRowsA), B from row b[p] (a multiple of its rb) and writes at c64 + c[p]
// (without `lead`).
struct EmuBatch {
  int n = 1;
  int a[8] = {0}, b[8] = {0};
  long long c[8] = {0};
};

// C (M x N) = A (M x K) . B (N x K)^T from operands sliced in form f; *d_err
// (device int) is set non-zero if a pipeline wait timed out.
void emu_gemm(EmuForm f, int M, int N, const EmuOperand& A, const EmuOperand& B,
              const EmuEpilogue& ep, int* d_err, cudaStream_t st, const EmuBatch& bt = EmuBatch());

}  // namespace ris
