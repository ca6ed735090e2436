// Mode products in FP64 and in precise FP32 on the bf16 tensor cores.
//
// An FP64 multiply-add on GB300's CUDA cores runs at about 1.1 TFLOP/s per
// GPU, the bf16 tensor cores at 1.9 PFLOP/s: 36 bf16 products of integer
// slices (the error-free splitting of Ozaki, Ogita, Oishi and Rump, Numer.
// Algorithms 59 (2012)) are far cheaper than one FP64 product.  Both operands
// are written as fixed-point numbers with one exponent per row (per fiber of
// the contracted index), cut into NS balanced digits of RB bits, which bf16
// holds exactly, and
//     Y[i][r] = 2^{E_i + E_r} sum_s 2^{RB (2 NS - 2 - s)} P_s,
//     P_s = sum_{a + b = s} sum_k m_a[i][k] x_b[r][k],   s < NLEV,
// each P_s summed as integers in the FP32 accumulator.  The epilogue adds the
// levels as 64-bit integers (FP64 arithmetic would cost more than the product)
// and rounds once.
//
// What the accumulator holds exactly: integers up to 2^24.  Level s takes s + 1
// products per k of digits |d| <= 128, the top ones <= 64.  A unit lost in P_s is
// 2^{-8 s - 12} of a full-size term max|x| max|M_i|, and an FP64 product rounds by up to
// 2^-53 K of one: levels 0 .. 4 have to be exact, and are, whatever the data:
// contractions go in segments short enough for the digits of the matrix at hand
// (slice_segment; 256 terms always do, and 350 to 500 with eigenvector matrices, whose
// digits average half the largest).  Levels 5 .. 7 may lose units of 2^-52 and less
// when hundreds of their digits are in line.  FP32: P_0 and P_1 are exact over 1024
// terms (2^12 and 2^14 per k); a unit lost in P_2 is 2^-28 of a full-size term.
//
// Cut off: a unit of an operand's last digit at most, and the levels s >= NLEV, for an
// error per entry of about 2^-60 sqrt(K) max|x| max|M_i| (FP32: 2^-29), relative to the
// largest entries of the two fibers, not to the entry's own terms.
//
// Orientation: the data rows (c, r) are the MMA's M (TMEM lanes), so that a
// warp stores 32 consecutive r of one output index i; 64 (FP64) or 128 (FP32)
// output indices are the N of one level.  The digits b of one data row block
// follow each other in shared memory, and so do those of the matrix: one MMA
// takes slice a of the data against several slices b of the matrix (N up to
// 256) and adds into the neighbouring levels a + b, which lie side by side in
// tensor memory.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <stdexcept>
#include <string>
#include <vector>

#include "b3_kernel.cuh"
#include "sliced.h"
#include "tma_host.h"

namespace fcgle {

namespace {

using namespace b3;

// exponents of rows that digits cannot hold: a NaN among the entries (the product
// writes NaN), an Inf but no NaN (the slicing pass writes the row's results)
constexpr int kSliceNaN = 0x40000000, kSliceInf = 0x40000001;
__device__ __forceinline__ bool unsliced(int e) { return e >= kSliceNaN; }

// ------------------------------------------------------------ slicing pass
// HBM-bound (FP64: 8 bytes read and 14 written per element), so one pass: a
// group of 8, 16 or 32 lanes owns a row, finds its largest exponent, and cuts
// the elements (read again, from L1 or L2) with integer shifts; no FP64
// arithmetic.
template <typename T>
struct Bits;
template <>
struct Bits<double> {
  using U = unsigned long long;
  static constexpr int kMant = 52, kExpMask = 0x7ff;
};
template <>
struct Bits<float> {
  using U = unsigned int;
  static constexpr int kMant = 23, kExpMask = 0xff;
};

template <typename T>
__device__ __forceinline__ void load4(const T* p, typename Bits<T>::U (&u)[4]) {
  if constexpr (sizeof(T) == 8) {
    const ulonglong2 a = reinterpret_cast<const ulonglong2*>(p)[0], b = reinterpret_cast<const ulonglong2*>(p)[1];
    u[0] = a.x; u[1] = a.y; u[2] = b.x; u[3] = b.y;
  } else {
    const uint4 a = *reinterpret_cast<const uint4*>(p);
    u[0] = a.x; u[1] = a.y; u[2] = a.z; u[3] = a.w;
  }
}

// The digits of one element as a balanced number: half a digit added at every
// place but the top one, so that place a is (w >> RB (NS - 1 - a)) mod 2^RB - 2^{RB - 1}.
template <typename T>
struct Balanced;
template <>
struct Balanced<double> {
  using W = long long;
};
template <>
struct Balanced<float> {
  using W = int;
};
template <class C>
__host__ __device__ __forceinline__ typename Balanced<typename C::T>::W balanced(typename Bits<typename C::T>::U u,
                                                                                 int emax, bool bad) {
  using T = typename C::T;
  using U = typename Bits<T>::U;
  using W = typename Balanced<T>::W;
  constexpr int NS = C::NS, RB = C::RB, MB = Bits<T>::kMant, UP = C::BITS - MB - 2;
  const int e = (int)((u >> MB) & Bits<T>::kExpMask);
  const U mant = ((u & ((U(1) << MB) - 1)) | (e ? U(1) << MB : U(0))) << UP;
  const int s = emax - (e > 1 ? e : 1);
  const U m = s < (int)(8 * sizeof(U)) - 2 ? (mant + ((U(1) << s) >> 1)) >> s : U(0);
  W x = (u >> (8 * sizeof(U) - 1)) ? -(W)m : (W)m;
  if (bad) x = 0;
  W off = 0;
#pragma unroll
  for (int j = 0; j + 1 < NS; ++j) off += W(1) << (RB * j + RB - 1);
  return x + off;
}

// After a block's rows are cut, by the lanes that found a row with an Inf or a NaN
// among theirs: rows whose only non-finite entries are infinities get their
// results here, M[i][k] (+-Inf) summed over these, which is what the sum over all
// entries comes to.  Apart from the loop over the rows, which it would cost registers.
template <typename T>
__device__ __noinline__ void infinite_rows(const T* X, long long rows, int nseg, int seg_len, long long seg_stride,
                                           int group, int* ex, const SliceOut<T>& o) {
  if (!o.M) return;
  const int per_block = 256 / group, lig = threadIdx.x % group, K = nseg * seg_len;
  for (long long row = (long long)blockIdx.x * per_block + threadIdx.x / group; row < rows;
       row += (long long)gridDim.x * per_block) {
    const T* src = X + row * seg_len;
    bool nan = false, inf = false;
    for (int k = 0; k < K && !nan; ++k) {
      const T x = src[(k / seg_len) * seg_stride + k % seg_len];
      nan = isnan(x);
      inf |= isinf(x);
    }
    if (nan || !inf) continue;
    const long long c = row / o.R;
    T* dst = o.Y + c * o.plane + (row - c * o.R);
    for (int i = lig; i < o.m; i += group) {
      T sum = 0;
      for (int k = 0; k < K && !isnan(sum); ++k) {
        const T x = src[(k / seg_len) * seg_stride + k % seg_len];
        if (isinf(x)) sum += o.M[(size_t)i * K + k] * x;
      }
      dst[(long long)i * o.R] = sum;
    }
    if (lig == 0) ex[row] = kSliceInf;   // the same lane wrote kSliceNaN
  }
}

template <class C, typename T = typename C::T>
__global__ void __launch_bounds__(256) slice_kernel(const T* X, long long rows, int nseg, int seg_len,
                                                    long long seg_stride, int pitch, int group,
                                                    __nv_bfloat16* __restrict__ dig, int* __restrict__ ex,
                             const __grid_constant__ SliceOut<T> o) {
  using U = typename Bits<T>::U;
  constexpr int NS = C::NS, RB = C::RB, MB = Bits<T>::kMant;
  constexpr int UP = C::BITS - MB - 2;   // spare bits below the last one of the largest entry
  pdl_trigger();
  pdl_wait();
  const int per_block = 256 / group;
  const int lig = threadIdx.x % group;
  const int quads = seg_len / 4;
  bool any_bad = false;
  for (long long row0 = (long long)blockIdx.x * per_block; row0 < rows; row0 += (long long)gridDim.x * per_block) {
    const long long row = row0 + threadIdx.x / group;
    const bool live = row < rows;
    int emax = 1;
    if (live)
      for (int c = 0; c < nseg; ++c) {
        const T* src = X + c * seg_stride + row * seg_len;
        for (int q = lig; q < quads; q += group) {
          U u[4];
          load4<T>(src + 4 * q, u);
#pragma unroll
          for (int v = 0; v < 4; ++v) emax = max(emax, (int)((u[v] >> MB) & Bits<T>::kExpMask));
        }
      }
    for (int o = group / 2; o > 0; o >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
    if (!live) continue;
    const bool bad = emax == Bits<T>::kExpMask;
    any_bad |= bad;
    // x = mant 2^{e - bias - MB}; v = (mant << UP) >> (emax - e): unit 2^{emax - bias - MB - UP}
    if (lig == 0) ex[row] = bad ? kSliceNaN : emax - (Bits<T>::kExpMask >> 1) - MB - UP;
    for (int c = 0; c < nseg; ++c) {
      const T* src = X + c * seg_stride + row * seg_len;
      __nv_bfloat16* dst = dig + row * pitch + c * seg_len;
      for (int q = lig; q < quads; q += group) {
        U u[4];
        load4<T>(src + 4 * q, u);
        typename Balanced<T>::W w[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) w[v] = balanced<C>(u[v], emax, bad);
#pragma unroll
        for (int a = 0; a < NS; ++a) {
          uint32_t h[4];
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            // digit as a small integer, exact in bf16 (at most 8 significant bits)
            const int d = a == 0 ? (int)(w[v] >> (RB * (NS - 1)))
                                 : ((int)(w[v] >> (RB * (NS - 1 - a))) & ((1 << RB) - 1)) - (1 << (RB - 1));
            h[v] = __float_as_uint((float)d);
          }
          uint2 d2;
          d2.x = (h[0] >> 16) | (h[1] & 0xFFFF0000u);
          d2.y = (h[2] >> 16) | (h[3] & 0xFFFF0000u);
          *reinterpret_cast<uint2*>(dst + (size_t)a * rows * pitch + 4 * q) = d2;
        }
      }
    }
  }
  if (any_bad) infinite_rows<T>(X, rows, nseg, seg_len, seg_stride, group, ex, o);
}

// The same pass for rows of up to 8 x 32 x IT elements in segments of a multiple
// of 8: a lane keeps its 8-element pieces in registers between the two halves
// and stores 16 bytes per digit (FP32 at 432^3 with 3 digits: 473 us with 4-element
// pieces read twice, 303 this way = 5.3 TB/s).
template <class C, int IT, typename T = typename C::T>
__global__ void __launch_bounds__(256) slice8_kernel(const T* X, long long rows, int nseg, int seg_len,
                                                     long long seg_stride, int pitch, int group,
                                                     __nv_bfloat16* __restrict__ dig, int* __restrict__ ex,
                             const __grid_constant__ SliceOut<T> o) {
  using U = typename Bits<T>::U;
  using W = typename Balanced<T>::W;
  constexpr int NS = C::NS, RB = C::RB, MB = Bits<T>::kMant, UP = C::BITS - MB - 2;
  pdl_trigger();
  pdl_wait();
  const int per_block = 256 / group, lig = threadIdx.x % group;
  const int cps = seg_len / 8, chunks = nseg * cps;
  bool any_bad = false;
  for (long long row0 = (long long)blockIdx.x * per_block; row0 < rows; row0 += (long long)gridDim.x * per_block) {
    const long long row = row0 + threadIdx.x / group;
    const bool live = row < rows;
    U u[IT][8];
    int emax = 1;
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const int c = lig + group * it;
      if (live && c < chunks) {
        const int seg = c >= cps ? 1 : 0;
        const T* src = X + seg * seg_stride + row * seg_len + 8 * (c - seg * cps);
        U h[4];
        load4<T>(src, h);
#pragma unroll
        for (int v = 0; v < 4; ++v) u[it][v] = h[v];
        load4<T>(src + 4, h);
#pragma unroll
        for (int v = 0; v < 4; ++v) u[it][4 + v] = h[v];
#pragma unroll
        for (int v = 0; v < 8; ++v) emax = max(emax, (int)((u[it][v] >> MB) & Bits<T>::kExpMask));
      }
    }
    for (int o = group / 2; o > 0; o >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
    if (!live) continue;
    const bool bad = emax == Bits<T>::kExpMask;
    any_bad |= bad;
    if (lig == 0) ex[row] = bad ? kSliceNaN : emax - (Bits<T>::kExpMask >> 1) - MB - UP;
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const int c = lig + group * it;
      if (c < chunks) {
        W w[8];
#pragma unroll
        for (int v = 0; v < 8; ++v) w[v] = balanced<C>(u[it][v], emax, bad);
        __nv_bfloat16* dst = dig + row * pitch + 8 * c;
#pragma unroll
        for (int a = 0; a < NS; ++a) {
          uint32_t h[8];
#pragma unroll
          for (int v = 0; v < 8; ++v) {
            const int d = a == 0 ? (int)(w[v] >> (RB * (NS - 1)))
                                 : ((int)(w[v] >> (RB * (NS - 1 - a))) & ((1 << RB) - 1)) - (1 << (RB - 1));
            h[v] = __float_as_uint((float)d);
          }
          uint4 d4;
          d4.x = __byte_perm(h[0], h[1], 0x7632);
          d4.y = __byte_perm(h[2], h[3], 0x7632);
          d4.z = __byte_perm(h[4], h[5], 0x7632);
          d4.w = __byte_perm(h[6], h[7], 0x7632);
          *reinterpret_cast<uint4*>(dst + (size_t)a * rows * pitch) = d4;
        }
      }
    }
  }
  if (any_bad) infinite_rows<T>(X, rows, nseg, seg_len, seg_stride, group, ex, o);
}

// ------------------------------------------------------------ product
// Measured with the slicing pass (one real product, GB300, L2 flushed): FP64 128 x
// 120 x 136 68 us (900 us on the CUDA cores, whose FP64 rate is 1.1 TFLOP/s), 400 x
// 400 40 (412), 1023 x 1024 138 (4090), 432 x 432 x 100 945 (27014).  FP32 1023 x
// 1024 44 us (150), 432 x 432 x 100 337 (1080).
// What bounds it: the bf16 tensor cores and, close behind, the operand bytes
// an SM pulls from L2 (FP64: 96 KB per 32 k against 2304 MMA clocks, 43 bytes
// per clock).  All levels of a tile share tensor memory (FP64 8 x 64, FP32
// 4 x 128 columns), so the accumulators are single-buffered and the MMAs of
// the next tile wait while the epilogue reads them.  16 epilogue warps therefore
// only add the levels up to integer sums (16 or 32 columns each), hand tensor
// memory back, and round and store while the next tile runs (8 warps that rounded
// first: 1125 against 754 us for FP32 at 432^3, 67 against 51 for FP64 at
// 128 x 120 x 136).
constexpr int kSegK = 1024;     // longest contraction whose levels 0 and 1 stay exact (within 2^24)
constexpr int kGK = 32;         // k per stage: 64-byte bf16 rows, 64-byte swizzle
constexpr int kGM = 128;        // data rows per tile
constexpr int kGEpi = 16;       // epilogue warps
constexpr int kGThreads = 32 * (4 + kGEpi);   // producer, MMA issuer, two idle ones
// registers: 128 x 40 + 512 x 104 = 58368 of the 640 x 96 = 61440 at launch (checked by the host)
constexpr int kGRegCtl = 40, kGRegEpi = 104, kGRegLaunch = 96;

template <class C>
struct GemmLayout {
  static constexpr int NS = C::NS;
  static constexpr uint32_t kA = kGM * 64, kB = C::NT * 64;   // bytes of one slice of a chunk
  static constexpr uint32_t kStage = NS * (kA + kB);
  static constexpr uint32_t kOffBar = C::NSTAGE * kStage;
  static constexpr uint32_t kSmem = kOffBar + 256 + 1024;
  static_assert(kSmem <= 232448, "shared memory budget");
  static_assert(C::NLEV * C::NT <= 512, "tensor memory columns");
  static_assert(kStage % 1024 == 0 && kA % 1024 == 0 && kB % 1024 == 0, "slices start on swizzle atoms");
};

struct GemmParams {
  long long rows;    // data rows
  long long R;       // rows per plane of the output
  long long plane;   // elements between the planes of Y
  int m;             // output indices
  int m_tiles, k_chunks;
  long long units;
  int seg;           // k-chunks of a segment
  int* err;
};

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&v)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(taddr));
}
// K-major, SWIZZLE_64B: rows of 64 bytes, 8-row groups 512 bytes apart
__device__ __forceinline__ uint64_t desc64(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(512 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)4 << 61);
}

// The levels of one output, added up exactly: FP64 as V = 2^32 hi + lo (levels 0 .. 3
// and 4 .. 7), FP32 from the smallest level up.  add() takes the levels of one segment of the
// contraction, get() gives the sum times 2^e.
template <class C, typename T = typename C::T>
struct Sum {   // FP64, RB = 8
  static_assert(C::NLEV == 8 && C::RB == 8, "sums of eight 8-bit levels");
  long long hi = 0, lo = 0;
  __device__ __forceinline__ void add(const float (&P)[C::NLEV]) {
    hi += ((long long)__float2int_rn(P[0]) << 24) + ((long long)__float2int_rn(P[1]) << 16) +
          ((long long)__float2int_rn(P[2]) << 8) + (long long)__float2int_rn(P[3]);
    lo += ((long long)__float2int_rn(P[4]) << 24) + ((long long)__float2int_rn(P[5]) << 16) +
          ((long long)__float2int_rn(P[6]) << 8) + (long long)__float2int_rn(P[7]);
  }
  // |hi| < 2^37 K: rounded to 53 bits through a 63-bit integer t = V / 2^s, s the
  // smallest shift that makes it fit, so that t is V itself or has 62 bits.  To
  // double by integer arithmetic: FP64 additions and the conversion instruction run on
  // the FP64 pipe at two lanes per clock and SM.
  __device__ __forceinline__ double get(int e) const {
    const int s = max(0, 34 - __clzll(hi ^ (hi >> 63))), up = 32 - s;   // bits of |hi| beyond 30; K <= 2^24: s <= 32
    const unsigned long long tu =
        ((unsigned long long)hi << up) + (unsigned long long)((lo + ((1ll << s) >> 1)) >> s);
    const long long t = (long long)tu;
    const int k = e + 8 * (2 * C::NS - 1 - C::NLEV) + s;
    if (k <= -1000 || k >= 900) return ldexp((double)t, k);
    // normalise to 64 bits, round to nearest even, fill in sign and exponent
    const uint32_t sg = (uint32_t)((int)(tu >> 32) >> 31);
    const unsigned long long mag = (tu ^ (((unsigned long long)sg << 32) | sg)) + (sg & 1u);
    const uint32_t m1 = (uint32_t)(mag >> 32), m0 = (uint32_t)mag;
    const uint32_t x1 = m1 ? m1 : m0, x0 = m1 ? m0 : 0u;
    const int lz = __clz((int)x1);
    const uint32_t n1 = __funnelshift_l(x0, x1, lz), n0 = x0 << lz;   // lz < 32 unless t == 0
    const uint32_t up1 = (n0 >> 10) & (uint32_t)((n0 & 0x3FFu) != 0u || (n0 & 0x800u)) & 1u;
    const uint32_t field = (uint32_t)(1022 + 63 - lz - (m1 ? 0 : 32) + k);
    const unsigned long long bits = (((unsigned long long)((n1 >> 11) + (field << 20)) << 32) |
                                     __funnelshift_r(n0, n1, 11)) + up1;
    return tu == 0ull ? 0.0 : __longlong_as_double((long long)(bits | ((unsigned long long)(sg & 0x80000000u) << 32)));
  }
};
template <class C>
struct Sum<C, float> {
  float t = 0.f;
  __device__ __forceinline__ void add(const float (&P)[4]) {
    constexpr float u = 1.f / (1 << C::RB);
    t += fmaf(fmaf(fmaf(P[3], u, P[2]), u, P[1]), u, P[0]);
  }
  __device__ __forceinline__ float get(int e) const {
    const int k = e + C::RB * (2 * C::NS - 2);
    if (k >= -126 && k <= 127) return t * __int_as_float((k + 127) << 23);
    return ldexpf(t, k);
  }
};

template <class C, typename T = typename C::T>
__device__ __forceinline__ T finish(const Sum<C>& s, int er, int ei) {
  return unsliced(er) || unsliced(ei) ? (T)NAN : s.get(er + ei);
}

// SEG: the contraction goes in segments of gp.seg chunks, each drained from tensor
// memory into the integer sums before the next begins.
template <class C, bool SEG, typename T = typename C::T>
__global__ void __launch_bounds__(kGThreads, 1)
    sliced_gemm_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_m,
                       const int* ex, const int* __restrict__ em, T* __restrict__ Y,
                       const GemmParams gp) {
  using L = GemmLayout<C>;
  constexpr int NS = C::NS, NLEV = C::NLEV, NT = C::NT, NSTAGE = C::NSTAGE;
  extern __shared__ uint8_t smem_raw[];
  pdl_trigger();
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::kOffBar);
  auto full_bar = [&](int s) { return smem_u32(&bars[s]); };
  auto empty_bar = [&](int s) { return smem_u32(&bars[NSTAGE + s]); };
  const uint32_t acc_full = smem_u32(&bars[2 * NSTAGE]);
  const uint32_t acc_empty = smem_u32(&bars[2 * NSTAGE + 1]);
  const uint32_t fin_bar = smem_u32(&bars[2 * NSTAGE + 2]);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::kOffBar + 192);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::kOffBar + 200);
  static_assert((2 * NSTAGE + 3) * 8 <= 192, "barrier area");

  if (threadIdx.x == 0) {
    for (int s = 0; s < NSTAGE; ++s) {
      mbar_init(full_bar(s), 1);
      mbar_init(empty_bar(s), 1);
    }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, kGEpi);
    mbar_init(fin_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  pdl_wait();

  if (warp < 4) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kGRegCtl));
  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      uint32_t g = 0;
      bool ok = true;
      for (long long u = blockIdx.x; u < gp.units && ok; u += gridDim.x) {
        const int row0 = (int)(u / gp.m_tiles) * kGM;
        const int i0 = (int)(u % gp.m_tiles) * NT;
        for (int kc = 0; kc < gp.k_chunks; ++kc, ++g) {
          const int s = (int)(g % NSTAGE);
          if (!mbar_wait(empty_bar(s), ((g / NSTAGE) & 1) ^ 1, abort_flag, gp.err, 51)) { ok = false; break; }
          const uint32_t st = sbase + s * L::kStage;
          mbar_arrive_tx(full_bar(s), L::kStage);
#pragma unroll
          for (int a = 0; a < NS; ++a) {
            tma_load_3d(st + a * L::kA, &tm_x, kc * kGK, row0, a, full_bar(s));
            tma_load_3d(st + NS * L::kA + a * L::kB, &tm_m, kc * kGK, i0, a, full_bar(s));
          }
        }
      }
      // drain: every issued stage must have landed before the CTA may exit
      const uint32_t issued = g;
      for (uint32_t q = issued >= (uint32_t)NSTAGE ? issued - NSTAGE : 0; q < issued; ++q)
        mbar_wait(full_bar(q % NSTAGE), (q / NSTAGE) & 1, abort_flag, gp.err, 57, true);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kGM >> 4) << 24);
      uint32_t g = 0, t = 0;
      bool ok = true;
      for (long long u = blockIdx.x; u < gp.units && ok; u += gridDim.x) {
        for (int kc = 0; kc < gp.k_chunks; ++kc, ++g) {
          const bool begin = SEG ? kc % gp.seg == 0 : kc == 0;
          if (begin) {
            if (!mbar_wait(acc_empty, (t & 1) ^ 1, abort_flag, gp.err, 52)) { ok = false; break; }
            tc_fence_after();
          }
          const int s = (int)(g % NSTAGE);
          if (!mbar_wait(full_bar(s), (g / NSTAGE) & 1, abort_flag, gp.err, 53)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sa = sbase + s * L::kStage, sb = sa + NS * L::kA;
#pragma unroll
          for (int ks = 0; ks < 2; ++ks) {
            const uint32_t off = ks * 32;
            const bool first = begin && ks == 0;
#pragma unroll
            for (int a = 0; a < NS; ++a) {
              // slice a against slices 0 .. nb - 1, at most 256 columns per MMA; a piece
              // starts its levels where no earlier piece of the tile has added to them
              constexpr int kPer = 256 / NT;
              const int nb = NS < NLEV - a ? NS : NLEV - a;
#pragma unroll
              for (int b = 0; b < nb; b += kPer) {
                const int w = nb - b < kPer ? nb - b : kPer;
                const int seen = a == 0 ? b : (NS < NLEV - a + 1 ? NS : NLEV - a + 1) + a - 1;   // levels begun so far
                const uint32_t acc = (first && a + b >= seen) ? 0u : 1u;
                mma_bf16(tmem_base + (a + b) * NT, desc64(sa + a * L::kA + off), desc64(sb + b * L::kB + off),
                         idesc0 | ((uint32_t)(w * NT >> 3) << 17), acc);
              }
            }
          }
          mma_commit(empty_bar(s));
          if (kc + 1 == gp.k_chunks || (SEG && (kc + 1) % gp.seg == 0)) {
            mma_commit(acc_full);
            ++t;
          }
        }
      }
      // drain: all issued MMAs complete before TMEM is released
      mma_commit(fin_bar);
      mbar_wait(fin_bar, 0, abort_flag, gp.err, 58, true);
    }
  }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kGRegEpi));
    // ------------------------------------------------------------ epilogue
    // lane = data row, NC columns per warp: the levels into integer (FP32: float)
    // sums, tensor memory back to the MMA warp, then rounding and stores
    constexpr int NC = NT / 4;
    const int q = warp & 3, cg = (warp - 4) >> 2;
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;
    uint32_t t = 0;
    bool ok = true;
    const int segs = SEG ? (gp.k_chunks + gp.seg - 1) / gp.seg : 1;
    for (long long u = blockIdx.x; u < gp.units && ok; u += gridDim.x) {
      const long long row = (u / gp.m_tiles) * kGM + q * 32 + lane;
      const int i0 = (int)(u % gp.m_tiles) * NT + cg * NC;
      const bool live = row < gp.rows;
      const int er = live ? ex[row] : 0;
      Sum<C> sum[NC];
      for (int sg = 0; sg < segs; ++sg, ++t) {
        if (!mbar_wait(acc_full, t & 1, abort_flag, gp.err, 59)) { ok = false; break; }
        tc_fence_after();
#pragma unroll
        for (int c0 = 0; c0 < NC; c0 += 4) {
          uint32_t v[NLEV][4];
#pragma unroll
          for (int l = 0; l < NLEV; ++l) tmem_ld4(tmem_base + lane_off + l * NT + cg * NC + c0, v[l]);
          tmem_wait_ld();
#pragma unroll
          for (int l = 0; l < NLEV; ++l) tmem_loaded(v[l]);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float P[NLEV];
#pragma unroll
            for (int l = 0; l < NLEV; ++l) P[l] = __uint_as_float(v[l][j]);
            sum[c0 + j].add(P);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty);
      }
      if (!ok) break;
      if (live && er != kSliceInf) {   // rows with an Inf are the slicing pass's
        const long long c = row / gp.R;
        T* dst = Y + c * gp.plane + (row - c * gp.R) + (long long)i0 * gp.R;
        const int4* e4 = reinterpret_cast<const int4*>(em + i0);   // readable up to a whole tile
#pragma unroll
        for (int j4 = 0; j4 < NC / 4; ++j4) {
          const int4 x = __ldg(e4 + j4);
          const int ei[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (i0 + 4 * j4 + j < gp.m) dst[(long long)(4 * j4 + j) * gp.R] = finish<C>(sum[4 * j4 + j], er, ei[j]);
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512));
}

}  // namespace

// The levels that have to be exact are summed in the worst case, with the data's
// digits at their largest and in line with the matrix's: sum over a < s of 128 |m_a|
// plus 64 |m_s| for every row and segment, most for s = 4 (FP32: levels 0 and 1,
// within 2^24 over kSegK terms whatever the digits).
template <class C>
int slice_segment(const typename C::T* M, int rows, int K) {
  using T = typename C::T;
  constexpr int NS = C::NS, RB = C::RB;
  const int chunks = (K + kGK - 1) / kGK;
  int seg = std::min(chunks, kSegK / kGK);
  if (sizeof(T) == 8) {
    constexpr int kExact = 5;   // levels 0 .. 4
    // per row and chunk: that sum for s = 4, which bounds the levels before it too
    std::vector<int> sum((size_t)rows * chunks, 0);
    for (int i = 0; i < rows; ++i) {
      const T* row = M + (size_t)i * K;
      int emax = 1;
      auto bits = [](T x) {
        typename Bits<T>::U u;
        std::memcpy(&u, &x, sizeof(u));
        return u;
      };
      for (int k = 0; k < K; ++k) emax = std::max(emax, (int)((bits(row[k]) >> Bits<T>::kMant) & Bits<T>::kExpMask));
      const bool bad = emax == Bits<T>::kExpMask;
      for (int k = 0; k < K; ++k) {
        const auto w = balanced<C>(bits(row[k]), emax, bad);
        for (int a = 0; a < kExact; ++a) {
          const int dig = a == 0 ? (int)(w >> (RB * (NS - 1)))
                                 : ((int)(w >> (RB * (NS - 1 - a))) & ((1 << RB) - 1)) - (1 << (RB - 1));
          sum[(size_t)i * chunks + k / kGK] += (a + 1 < kExact ? 128 : 64) * std::abs(dig);
        }
      }
    }
    for (int n = (chunks + seg - 1) / seg;; ++n) {
      seg = (chunks + n - 1) / n;
      bool fits = true;
      for (int i = 0; i < rows && fits; ++i)
        for (int c0 = 0; c0 < chunks && fits; c0 += seg) {
          long long level = 0;
          for (int c = c0; c < std::min(c0 + seg, chunks); ++c) level += sum[(size_t)i * chunks + c];
          fits = level <= (1ll << 24);
        }
      if (fits) break;   // at the latest with 8 chunks = 256 terms: (64 + 3 x 128 + 64) x 128 x 256 = 2^24
    }
  }
  return seg * kGK;
}

template <class C>
void slice_map(Sliced& s, bool matrix) {
  const cuuint64_t pitch = (cuuint64_t)slice_pitch(s.K);
  cuuint64_t dims[3] = {(cuuint64_t)s.K, (cuuint64_t)s.rows, (cuuint64_t)C::NS};
  cuuint64_t strides[2] = {pitch * 2, pitch * 2 * (cuuint64_t)s.rows};
  cuuint32_t box[3] = {kGK, (cuuint32_t)(matrix ? C::NT : kGM), 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = encode_fn()(&s.tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, s.dig, dims, strides, box, estr,
                           CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) throw std::runtime_error("cuTensorMapEncodeTiled (slices) failed (" + std::to_string((int)r) + ")");
}

template <class C>
void slice_rows(const typename C::T* X, const Sliced& s, int nseg, int seg_len, long long seg_stride,
                const SliceOut<typename C::T>& o, cudaStream_t st, long long& nl) {
  const int chunks = nseg * seg_len / 8;
  if (seg_len % 8 == 0 && chunks <= 128) {
    int group = 1;
    while (group < 32 && group < chunks) group *= 2;
    const long long per_block = 256 / group;
    const int blocks = (int)std::min<long long>((s.rows + per_block - 1) / per_block, (long long)num_sms() * 32);
    const int it = (chunks + group - 1) / group;
    launch_pdl(it == 1   ? slice8_kernel<C, 1>
               : it == 2 ? slice8_kernel<C, 2>
               : it == 3 ? slice8_kernel<C, 3>
                         : slice8_kernel<C, 4>,
               blocks, 256, 0, st, X, s.rows, nseg, seg_len, seg_stride, slice_pitch(s.K), group, s.dig, s.ex, o);
    FCGLE_LAUNCHED(nl);
    return;
  }
  const int quads = seg_len / 4;
  const int group = quads <= 8 ? 8 : (quads <= 16 ? 16 : 32);
  const long long per_block = 256 / group;
  const long long blocks = std::min<long long>((s.rows + per_block - 1) / per_block, (long long)num_sms() * 16);
  launch_pdl(slice_kernel<C>, (int)blocks, 256, 0, st, X, s.rows, nseg, seg_len, seg_stride, slice_pitch(s.K), group,
             s.dig, s.ex, o);
  FCGLE_LAUNCHED(nl);
}

template <class C>
void sliced_gemm(const Sliced& x, const Sliced& m, typename C::T* Y, long long R, long long plane, int* err,
                 cudaStream_t st, long long& nl) {
  static std::once_flag attr;
  std::call_once(attr, [] {
    for (auto* k : {sliced_gemm_kernel<C, false>, sliced_gemm_kernel<C, true>}) {
      cudaFuncAttributes a;
      FCGLE_CUDA(cudaFuncGetAttributes(&a, k));
      if (a.numRegs < kGRegLaunch)
        throw std::logic_error("sliced product built with " + std::to_string(a.numRegs) + " registers");
    }
    FCGLE_CUDA(cudaFuncSetAttribute(sliced_gemm_kernel<C, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)GemmLayout<C>::kSmem));
    FCGLE_CUDA(cudaFuncSetAttribute(sliced_gemm_kernel<C, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    (int)GemmLayout<C>::kSmem));
  });
  GemmParams gp;
  gp.rows = x.rows;
  gp.R = R;
  gp.plane = plane;
  gp.m = (int)m.rows;
  gp.m_tiles = (gp.m + C::NT - 1) / C::NT;
  gp.k_chunks = (x.K + kGK - 1) / kGK;
  gp.units = (x.rows + kGM - 1) / kGM * gp.m_tiles;
  gp.seg = m.seg / kGK;
  gp.err = err;
  launch_pdl(gp.k_chunks <= gp.seg ? sliced_gemm_kernel<C, false> : sliced_gemm_kernel<C, true>,
             (int)std::min<long long>(gp.units, num_sms()), kGThreads, GemmLayout<C>::kSmem, st, x.tm, m.tm,
             (const int*)x.ex, (const int*)m.ex, Y, gp);
  FCGLE_LAUNCHED(nl);
}

#define INST(C)                                                                                                    \
  template int slice_segment<C>(const C::T*, int, int);                                                            \
  template void slice_map<C>(Sliced&, bool);                                                                       \
  template void slice_rows<C>(const C::T*, const Sliced&, int, int, long long, const SliceOut<C::T>&, cudaStream_t, \
                              long long&);                                                                         \
  template void sliced_gemm<C>(const Sliced&, const Sliced&, C::T*, long long, long long, int*, cudaStream_t, long long&);
INST(Slices32)
INST(Slices64)
#undef INST

}  // namespace fcgle
