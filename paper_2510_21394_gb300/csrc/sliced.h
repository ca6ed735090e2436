// Sliced mu-mode products (Sec. 3.2): FP64 and precise FP32 matrix products
// computed on the bf16 tensor cores from exact integer slices (sliced.cu).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include "common.h"

namespace fcgle {

// Slices per operand: x = 2^E sum_a d_a 2^{RB (NS - 1 - a)} with integer digits
// |d_a| <= 2^{RB - 1} (the top one <= 64), exact in bf16, and one exponent E per row
// (a fiber of the contracted index); what is cut off is at most a unit of the last
// digit.  BITS counts the sum's bits and its sign.  NLEV levels of digit products are
// kept, NT output indices make a tile, NSTAGE chunks are in flight (sliced.cu).
//
// The cut is relative to the fiber's largest entry, so the bits exceed those of the
// type by as much as fibers are uneven: the spectrum of a smooth field is a few large
// entries and a long fall-off, and the cuts of all its entries enter every result; the
// entries of e^{theta K} fall off by many orders from the diagonal.  Measured against
// products in FP64 and FP32:
//  * FP64, 62 bits: the errors of f(theta K) v are 0.2 to 1.05 times theirs (near 1 those
//    of the eigenvalues, common to both, prevail).  With 7 digits
//    (55 bits, 28 products of digits instead of 36, 8 to 10 % less time per product)
//    the maximum error on the box (-1, 1)^2 was up to 1.5 times theirs, the median error
//    of an entry of e^{theta K} v, relative to the entry, up to 1.3 times.
//  * FP32, 30 bits: three LBDF2 steps at 300 x 200 x 150 and 300 x 310 end with 0.5 to
//    0.95 times their error.  With 3 digits of 9 (25 bits, 8 products instead of 10, 277
//    instead of 340 us at 432 x 432 x 100) the maximum error was 1.2 to 1.9 times theirs.
struct Slices64 {
  using T = double;
  static constexpr int NS = 8, RB = 8, BITS = 63, NLEV = 8, NT = 64, NSTAGE = 2;
};
struct Slices32 {
  using T = float;
  static constexpr int NS = 4, RB = 8, BITS = 31, NLEV = 4, NT = 128, NSTAGE = 3;
};

inline int slice_pitch(int K) { return (K + 7) & ~7; }   // 16-byte bf16 rows

// The digits of one operand, [NS][rows][pitch] bf16, and the exponent of every row.
struct Sliced {
  __nv_bfloat16* dig = nullptr;
  int* ex = nullptr;
  long long rows = 0;
  int K = 0;
  int seg = 0;      // matrix operand: terms of the contraction whose leading levels are summed exactly
  CUtensorMap tm;   // boxes of (32 k, 128 rows or the matrix tile) of one slice
};

// bytes of a digit buffer and of its exponents
template <class C>
inline size_t slice_bytes(long long rows, int K) {
  return (size_t)C::NS * (size_t)rows * (size_t)slice_pitch(K) * 2;
}

// exponents of a matrix operand: the product reads them by whole tiles
inline size_t slice_exponents(long long rows) { return (size_t)((rows + 127) / 128 * 128); }

// Fills s.tm for s.dig / s.rows / s.K.  matrix: the box of the matrix operand
// (M rows), else of the data operand.
template <class C>
void slice_map(Sliced& s, bool matrix);

// Terms of a segment of the contraction with M (rows x K, host): a multiple of 32.
template <class C>
int slice_segment(const typename C::T* M, int rows, int K);

// Where the product of a data operand goes: the matrix (m x K, row-major, finite)
// and Y, R, plane of sliced_gemm.  M == nullptr: a matrix operand.
template <typename T>
struct SliceOut {
  const T* M = nullptr;
  T* Y = nullptr;
  long long R = 1, plane = 0;
  int m = 0;
};

// Slices the rows of X: row r is nseg segments of seg_len contiguous elements,
// segment c at X + c * seg_stride + r * seg_len; s.K = nseg * seg_len.  Rows with
// an Inf have no digits: their results are written here, to o.Y (not X).
template <class C>
void slice_rows(const typename C::T* X, const Sliced& s, int nseg, int seg_len, long long seg_stride,
                const SliceOut<typename C::T>& o, cudaStream_t st, long long& nl);

// Y[c][i][r] = sum_k M[i][k] X[(c, r)][k] for the sliced operands x (rows =
// planes * R) and m (rows = output indices i), c = row / R; plane: elements
// between the planes of Y.
template <class C>
void sliced_gemm(const Sliced& x, const Sliced& m, typename C::T* Y, long long R, long long plane, int* err,
                 cudaStream_t st, long long& nl);

}  // namespace fcgle
