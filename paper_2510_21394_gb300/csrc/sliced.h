// Sliced mu-mode products (Sec. 3.2): FP64 and precise FP32 matrix products
// computed on the bf16 tensor cores from exact integer slices (sliced.cu).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include "common.h"

namespace fcgle {

// Slices per operand: x = 2^E sum_a d_a 2^{RB (NS - 1 - a)} with integer digits
// |d_a| <= 2^{RB - 1} (the top one <= 128), exact in bf16, and one exponent E
// per row (a fiber of the contracted index); what is cut off is at most half a
// unit of the last digit.  BITS counts the sum's bits and its sign: FP64 7 digits of 8
// bits, 55 and the sign against the 53 of the type; FP32 3 digits of 9 bits, 25 against 24
// (26 would fit, but then the top digits reach 256 and their products pass 2^24
// after 256 terms instead of 1024).
template <typename T>
struct SliceCfg;
template <>
struct SliceCfg<double> {
  static constexpr int NS = 7, RB = 8, BITS = 56;
};
template <>
struct SliceCfg<float> {
  static constexpr int NS = 3, RB = 9, BITS = 26;
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
template <typename T>
inline size_t slice_bytes(long long rows, int K) {
  return (size_t)SliceCfg<T>::NS * (size_t)rows * (size_t)slice_pitch(K) * 2;
}

// exponents of a matrix operand: the product reads them by whole tiles
inline size_t slice_exponents(long long rows) { return (size_t)((rows + 127) / 128 * 128); }

// Fills s.tm for s.dig / s.rows / s.K.  matrix: the box of the matrix operand
// (M rows), else of the data operand.
template <typename T>
void slice_map(Sliced& s, bool matrix);

// Terms of a segment of the contraction with M (rows x K, host): a multiple of 32.
template <typename T>
int slice_segment(const T* M, int rows, int K);

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
template <typename T>
void slice_rows(const T* X, const Sliced& s, int nseg, int seg_len, long long seg_stride, const SliceOut<T>& o,
                cudaStream_t st, long long& nl);

// Y[c][i][r] = sum_k M[i][k] X[(c, r)][k] for the sliced operands x (rows =
// planes * R) and m (rows = output indices i), c = row / R; plane: elements
// between the planes of Y.
template <typename T>
void sliced_gemm(const Sliced& x, const Sliced& m, T* Y, long long R, long long plane, int* err, cudaStream_t st,
                 long long& nl);

}  // namespace fcgle
