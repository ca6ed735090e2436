// Split-BF16 mu-mode product on the sm_103a tensor cores (tcgen05 + TMEM + TMA)
// with a fused pointwise epilogue (the last mode product of a Tucker operator
// that carries a scheme's pointwise stage).
//
// One launch computes, in the rotating layout of common.h,
//     acc[c][i][r] = sum_k M[i][k] X[c][r][k]              (Sec. 3.2, one mode product)
// where every operand arrives pre-split into two bf16 numbers, x = x_hi + x_lo,
// and the product is M_hi X_hi + M_hi X_lo + M_lo X_hi with FP32 accumulation
// in tensor memory (the dropped M_lo X_lo term is below 2^-16 relative).
// The FP32 result is handed, element by element as a complex number
// (acc[0][i][r], acc[1][i][r]), to an epilogue functor `Epi` that may read
// other standard-order tensors, evaluate the nonlinearity or the stage
// combinations of a scheme and write any outputs, split or FP32.
//
// GEMM orientation: D[i][col] = sum_k A[i][k] B[col][k] with A = M (MMA M =
// 128 output indices i per block) and B = 128 data rows: the same 64 indices
// r0..r0+63 of the real plane (columns 0..63) and of the imaginary plane
// (columns 64..127), so each epilogue thread sees complete complex values.
//
// Warp roles (one CTA per SM, persistent over (r-tile, i-block)):
//   warp 0      X producer: X_hi, X_lo (2 x 64 x 64) bf16 chunks by TMA,
//               SWIZZLE_128B, straight into the MMA layout.
//   warp 1      TMEM allocator and single-thread MMA issuer (3 MMAs per k-step).
//   warp 2      M producer: M_hi, M_lo (128 x 64) chunks (idle when M is in TMEM).
//   warp 3      idle (fills the control warpgroup).
//   warps 4-19  epilogue: TMEM -> registers -> the functor, on 4 consecutive r
//               of one output index per lane.  Warp w reads TMEM lane quarter
//               w % 4, 16 rows x 32 columns of each plane.
// Every mbarrier wait is bounded by a wall-clock limit; on expiry the CTA
// records an error code in *err, drains its own TMA and MMA work, frees its
// TMEM and returns.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>

#include "b3_epilogues.cuh"
#include "common.h"
#include "pdl.cuh"

namespace fcgle {
namespace b3 {

constexpr int BM = 128;     // output indices i per MMA
constexpr int BR = 64;      // r indices per tile (x 2 planes = MMA N)
constexpr int BN = 2 * BR;  // MMA N
constexpr int BK = 64;      // k per chunk (one 128-byte bf16 row)

// Launch shape of the fused-epilogue kernel: 16 epilogue warps share a tile (4
// TMEM lane quarters x 2 halves of 16 rows x 2 halves of 32 columns).
//
// What bounds it: not the arithmetic (leaving out the phi functions changes
// nothing) but the number of L2 requests and sectors per element; removing any
// stream of operands or results shortens it in proportion.  Hence:
//  * Operands are fetched ahead with cp.async, a warp copying blocks of 8 rows
//    x 128 bytes per plane (4 whole lines per instruction) into its own ring in
//    shared memory, across tile boundaries; sources of g travel the same way.
//    Loads of 64-byte pieces by the lanes that use them: 164 against 134 us for
//    EpiKrog3 at 256^3; a ring of 8 x 64-byte blocks twice as deep: 1337 against
//    1143 us for EpiLBDF2S at 432^3.
//  * Split results of two neighbouring pieces are exchanged between lanes, so
//    that a row is stored as 64 bytes per plane at once (EpiLBDF2S 1143 -> 975,
//    EpiExtrapG 898 -> 714 us at 432^3).
//  * Accumulator columns reach the functor without a pass through shared memory:
//    tcgen05.ld 16x256b gives each lane 2 + 2 columns of one row, and one
//    exchange between neighbouring lanes makes that 4 consecutive r.
//  * M in tensor memory (MT, p <= 256, single-problem real form): the grid is a
//    multiple of m_blocks, so a CTA keeps one i-block for the whole launch, and
//    its 128 x p block of M_hi and M_lo fits 256 TMEM columns.  Streamed through
//    shared memory, M = N = 128 MMAs read 8 KB of operands for 64 clocks of work
//    while TMA writes 64 KB per 12 of them: 127 clocks per MMA in the issue
//    loop.  M is constant, so it is loaded before the wait on the previous
//    kernel.  (EpiUpdateG 91 -> 73 us at 256^3.)
//  * setmaxnreg moves registers from the control warps to the epilogue (104,
//    grouped 112, instead of 96), which then does not spill.
// Per launch at 256^3, before -> now, us: EpiStageD 85 -> 78, EpiUpdateG 91 ->
// 80, EpiFhat 123 -> 104, EpiKrog2 124 -> 103, EpiKrog3 164 -> 123,
// EpiKrogFinal 154 -> 122 (5.1 .. 5.5 TB/s of 6.8).
//
// Complex form (CX = true, the Kronecker-product exponential of Eq. Neudeckerd):
// M = E = Er + i Ei is complex, so an M stage also carries the Ei_hi, Ei_lo chunks.
constexpr int kMtMaxP = 256;
constexpr uint32_t kFuXStage = 32768;   // X_hi (re | im) 16K | X_lo (re | im) 16K
template <class Epi, bool CX = false, bool MT = false>
struct Cfg {
  static constexpr int kEpi = 16;
  static constexpr int kThreads = 32 * (4 + kEpi);   // 3 control warps, one idle
  // registers per thread of the control warpgroup and of the four epilogue ones, out of the
  // 640 x 96 the block is launched with (checked by the host: a split beyond that would
  // wait for registers forever).  Grouped launches: the control warps do with 32
  static constexpr int kRegCtl = 40, kRegEpi = 104, kRegCtlG = 32, kRegEpiG = 112, kRegLaunch = 96;
  static_assert(128 * kRegCtl + (kThreads - 128) * kRegEpi <= kThreads * kRegLaunch, "register split");
  static_assert(128 * kRegCtlG + (kThreads - 128) * kRegEpiG <= kThreads * kRegLaunch, "register split");
  static constexpr bool kRing = Epi::kIn > 0 || Epi::kG;   // fetches operands or source terms
  // X and M ring depths
  static constexpr int kNX = CX ? 2 : (MT ? (kRing ? 3 : 6) : (Epi::kIn == 4 ? 2 : (kRing ? 3 : 4)));
  static constexpr int kNM = MT ? 0 : 2;
  static constexpr uint32_t kMStage = CX ? 65536 : 32768;   // M_hi 16K | M_lo 16K (| Ei_hi | Ei_lo)
  static constexpr uint32_t kOffM = kNX * kFuXStage;
  static constexpr uint32_t kOffEpi = kOffM + kNM * kMStage;
  // operand ring of a warp: slots of one block, 8 rows x 128 bytes per plane
  static constexpr uint32_t kEpiWarp = !kRing ? 0 : (CX ? 2048 : (MT ? 8192 : (Epi::kIn == 4 ? 6144 : 4096)));
  static constexpr int kPlanes = (int)(kEpiWarp / 1024);   // planes the ring can hold
  static_assert(kPlanes >= Epi::kIn, "one block of operands");
  static constexpr uint32_t kOffBar = kOffEpi + kEpi * kEpiWarp;
  static constexpr uint32_t kSmemBytes = kOffBar + 256 + 1024;   // + barriers + alignment slack
  static constexpr int kTmemCols = MT ? 512 : 2 * BN;
  static constexpr uint32_t kSmemGrouped = kSmemBytes + kEpi * (uint32_t)sizeof(PhiPoly);   // after the barriers
  static_assert(kSmemGrouped <= 232448 || MT, "shared memory budget");
  static_assert(kSmemBytes <= 232448, "shared memory budget");
  static_assert(!(CX && MT), "the complex block does not fit tensor memory");
};

constexpr unsigned long long kTimeoutNs = 2000000000ull;   // 2 s per wait

struct KParams {
  long long R;      // rows per plane of X; row length of the output planes
  int p;            // extent of the contracted / produced index (rows of M)
  int m_blocks;     // ceil(p / 128)
  int k_chunks;     // ceil(p / 64)
  long long tiles;  // ceil(R / 64)
  int* err;
  int ei_row = 0;   // complex forms: row of Ei in the stacked [Er; Ei] matrix maps
  // M in tensor memory: the padded matrices themselves (rows of k_pad elements)
  const __nv_bfloat16* mhi = nullptr;
  const __nv_bfloat16* mlo = nullptr;
  int k_pad = 0;
};

// Complex mode product (Eq. Neudecker): with M = Er + i Ei and the tile's
// columns 0..63 = re rows, 64..127 = im rows of X,
//   D[:, 0:64]   = Er Xre - Ei Xim   (re part)
//   D[:, 64:128] = Er Xim + Ei Xre   (im part)
// as one N = 128 product with Er over both planes plus two N = 64 products
// with Ei: negated on the im rows into columns 0..63, plain on the re rows
// into columns 64..127 (instruction-descriptor bit 13 negates A).  Each of the
// three is split hi.hi + hi.lo + lo.hi.
constexpr uint32_t kNegA = 1u << 13;

// -------------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait; returns false (and raises the CTA abort flag) on timeout or,
// unless `drain` is set, as soon as another role has aborted.  Drain waits
// (for this CTA's own TMA / MMA work before exit) only stop at the time limit.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* err,
                                          int code, bool drain = false) {
  if (mbar_try(bar, parity)) return true;
  const unsigned long long t0 = now_ns();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try(bar, parity)) return true;
    if ((it & 63) == 0) {
      if (!drain && *abort_flag) return false;
      if (now_ns() - t0 > kTimeoutNs) {
        *abort_flag = 1;
        atomicExch(err, code);
        return false;
      }
    }
  }
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}
__device__ __forceinline__ uint64_t sw128_desc(uint32_t addr) {
  // K-major, SWIZZLE_128B: rows of 128 bytes, 8-row groups 1024 bytes apart.
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
// MN-major, SWIZZLE_128B: every k is a 128-byte row of 64 consecutive n, 8-row
// (k) groups 1024 bytes apart (stride byte offset); the next 64 n start
// `mn_stride` bytes further (leading byte offset).  Used with the instruction
// descriptor's transpose-B bit.
__device__ __forceinline__ uint64_t sw128_mn_desc(uint32_t addr, uint32_t mn_stride) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((mn_stride >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}
constexpr uint32_t kTransB = 1u << 16;   // instruction descriptor: B is MN-major
__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                         uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum)
      : "memory");
}
// tcgen05.mma with the A operand in tensor memory
__device__ __forceinline__ void mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc,
                                            uint32_t accum) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accum)
      : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&v)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void cp_async16(uint32_t dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}
// 16 TMEM lanes x 16 columns: lane l of the warp gets rows l / 4 (v[0], v[1], v[4],
// v[5]) and l / 4 + 8 (v[2], v[3], v[6], v[7]) of columns 2 (l % 4) + {0, 1} and,
// in the second half of v, of the same columns + 8
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr));
}
// row l / 4 + 8 g of such a fragment: 4 consecutive columns from frag_col(l) on
__device__ __forceinline__ void frag_row(const uint32_t (&v)[8], int g, int lane, float (&o)[4]) {
  const bool odd = lane & 1;
  const uint32_t a0 = g ? v[2] : v[0], a1 = g ? v[3] : v[1], b0 = g ? v[6] : v[4], b1 = g ? v[7] : v[5];
  const uint32_t r0 = __shfl_xor_sync(0xffffffffu, odd ? a0 : b0, 1);
  const uint32_t r1 = __shfl_xor_sync(0xffffffffu, odd ? a1 : b1, 1);
  o[0] = __uint_as_float(odd ? r0 : a0);
  o[1] = __uint_as_float(odd ? r1 : a1);
  o[2] = __uint_as_float(odd ? b0 : r0);
  o[3] = __uint_as_float(odd ? b1 : r1);
}
__device__ __forceinline__ int frag_col(int lane) { return ((lane & 1) << 3) | ((lane & 2) << 1); }
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// orders every use of the loaded registers after the preceding tmem_wait_ld
template <int N>
__device__ __forceinline__ void tmem_loaded(uint32_t (&v)[N]) {
#pragma unroll
  for (int j = 0; j < N; ++j) asm volatile("" : "+r"(v[j]));
}

// ------------------------------------------------------------------ kernel
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, uint32_t src, int x, int y, int z) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(src), "r"(x), "r"(y), "r"(z)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait0() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ uint32_t split_pair(float a, float b, uint32_t& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  const float2 hf = __bfloat1622float2(h);
  const __nv_bfloat162 l = __floats2bfloat162_rn(a - hf.x, b - hf.y);
  lo = *reinterpret_cast<const uint32_t*>(&l);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// Grouped launches: problem k of a descriptor array owns the global units
// [gd[k].ubegin, gd[k + 1].ubegin); every warp role walks its units in
// increasing order, so a forward-only cursor finds the problem of a unit.
template <class D>
__device__ __forceinline__ long long locate(const D* gd, int n, long long u, int& pid) {
  while (pid + 1 < n && u >= gd[pid + 1].ubegin) ++pid;
  return u - gd[pid].ubegin;
}

// the phi polynomial of a functor that has one
template <class Epi>
__device__ __forceinline__ auto poly_of(const Epi& e, int) -> decltype(&e.ph) {
  return &e.ph;
}
template <class Epi>
__device__ __forceinline__ const PhiPoly* poly_of(const Epi&, long) {
  return nullptr;
}

// one problem of a grouped fused launch (aligned as its tensor maps)
template <class Epi>
struct FusedDesc {
  CUtensorMap xhi, xlo, mhi, mlo;
  KParams kp;
  long long ubegin;
  Epi epi;
};

// Grouped form (G = true): one persistent launch serves the last mode
// product of several independent problems; maps, sizes and the epilogue
// functor of problem k come from gd[k].  Same arithmetic per unit.
//
// Natural-order input (MN = true): X holds the contracted index as its
// SLOWEST index, X[c][k][r], the layout the slab-fused mode-1+2 product
// (b3_slab.cuh) leaves behind, so no rotation precedes this product.  The X
// tensor maps are 3D (r, k, plane) with 64 x 64 boxes (64 r of one k per
// 128-byte row), and the B operand is read MN-major; the accumulator, the
// epilogue and the output layout Y[c][i][r] are those of the K-major form.
template <class Epi, bool G = false, bool CX = false, bool MN = false, bool MT = false>
__global__ void __launch_bounds__(Cfg<Epi, CX, MT>::kThreads, 1)
    mp_b3_kernel(const __grid_constant__ CUtensorMap tm_xhi, const __grid_constant__ CUtensorMap tm_xlo,
                 const __grid_constant__ CUtensorMap tm_mhi, const __grid_constant__ CUtensorMap tm_mlo,
                 const KParams kp, const __grid_constant__ Epi epi, const FusedDesc<Epi>* __restrict__ gd, int ngd,
                 long long gunits) {
  static_assert(!(G && CX), "the complex form has no grouped variant");
  static_assert(!(MN && (G || CX)), "the natural-order form is single-problem and real");
  static_assert(!(MT && (G || CX)), "M in tensor memory: single-problem and real");
  using C = Cfg<Epi, CX, MT>;
  constexpr int NX = C::kNX, NM = C::kNM, NEPI = C::kEpi;
  constexpr uint32_t kMSt = C::kMStage, kOffM = C::kOffM, kOffBar = C::kOffBar;
  constexpr uint32_t kColM = 2 * BN;   // MT: per 16 k, 8 columns of M_hi and 8 of M_lo from here on
  extern __shared__ uint8_t smem_raw[];
  pdl_trigger();
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const uint32_t sbase = smem_u32(smem);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kOffBar);
  auto full_x = [&](int s) { return smem_u32(&bars[s]); };
  auto empty_x = [&](int s) { return smem_u32(&bars[NX + s]); };
  auto full_m = [&](int s) { return smem_u32(&bars[2 * NX + s]); };
  auto empty_m = [&](int s) { return smem_u32(&bars[2 * NX + NM + s]); };
  auto acc_full = [&](int a) { return smem_u32(&bars[2 * (NX + NM) + a]); };
  auto acc_empty = [&](int a) { return smem_u32(&bars[2 * (NX + NM) + 2 + a]); };
  const uint32_t fin_bar = smem_u32(&bars[2 * (NX + NM) + 4]);
  const uint32_t m_ready = smem_u32(&bars[2 * (NX + NM) + 5]);
  static_assert((2 * (NX + NM) + 6) * 8 <= 192, "barrier area");
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + kOffBar + 192);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + kOffBar + 200);

  if (threadIdx.x == 0) {
    for (int s = 0; s < NX; ++s) {
      mbar_init(full_x(s), 1);
      mbar_init(empty_x(s), 1);
    }
    for (int s = 0; s < NM; ++s) {
      mbar_init(full_m(s), 1);
      mbar_init(empty_m(s), 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(acc_full(a), 1);
      mbar_init(acc_empty(a), NEPI);
    }
    mbar_init(fin_bar, 1);
    mbar_init(m_ready, NEPI);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(C::kTmemCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  if constexpr (MT) {
    // this CTA's block of M into tensor memory: lane = row, two bf16 per column
    if (warp >= 4) {
      const int q = warp & 3, nk = 4 * kp.k_chunks;
      const size_t row = (size_t)(blockIdx.x % kp.m_blocks) * BM + q * 32 + lane;
      const uint32_t dst = tmem_base + ((uint32_t)(q * 32) << 16) + kColM;
      for (int kk = (warp - 4) >> 2; kk < nk; kk += NEPI / 4) {
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          const uint4* src = reinterpret_cast<const uint4*>((part ? kp.mlo : kp.mhi) + row * kp.k_pad + 16 * kk);
          const uint4 x = __ldg(src), y = __ldg(src + 1);
          const uint32_t v[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
          tmem_st8(dst + 16 * kk + 8 * part, v);
        }
      }
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(m_ready);
    }
  }
  pdl_wait();

  long long units;
  int* err;
  if constexpr (G) {
    units = gunits;
    err = gd[0].kp.err;
  } else {
    units = kp.tiles * kp.m_blocks;
    err = kp.err;
  }

  if (warp < 4) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(G ? C::kRegCtlG : C::kRegCtl));
  if (warp == 0) {
    // ------------------------------------------------------------ X producer
    if (lane == 0) {
      uint32_t g = 0;
      bool ok = true;
      int pid = 0;
      for (long long u = blockIdx.x; u < units && ok; u += gridDim.x) {
        long long lu = u, R = kp.R;
        int mbk = kp.m_blocks, KC = kp.k_chunks;
        const CUtensorMap *mxh = &tm_xhi, *mxl = &tm_xlo;
        if constexpr (G) {
          lu = locate(gd, ngd, u, pid);
          R = gd[pid].kp.R;
          mbk = gd[pid].kp.m_blocks;
          KC = gd[pid].kp.k_chunks;
          mxh = &gd[pid].xhi;
          mxl = &gd[pid].xlo;
        }
        const long long tile = lu / mbk;
        const int r0 = (int)(tile * BR);
        const int r1 = (int)(R + tile * BR);   // same r in the imaginary plane
        for (int kc = 0; kc < KC; ++kc, ++g) {
          const int s = (int)(g % NX);
          if (!mbar_wait(empty_x(s), ((g / NX) & 1) ^ 1, abort_flag, err, 1)) { ok = false; break; }
          const uint32_t st = sbase + s * kFuXStage;
          mbar_arrive_tx(full_x(s), kFuXStage);
          if constexpr (MN) {
            // 64 k-rows of 64 r, real plane then imaginary plane
            tma_load_3d(st, mxh, r0, kc * BK, 0, full_x(s));
            tma_load_3d(st + 8192, mxh, r0, kc * BK, 1, full_x(s));
            tma_load_3d(st + 16384, mxl, r0, kc * BK, 0, full_x(s));
            tma_load_3d(st + 16384 + 8192, mxl, r0, kc * BK, 1, full_x(s));
          } else {
            tma_load_2d(st, mxh, kc * BK, r0, full_x(s));
            tma_load_2d(st + 8192, mxh, kc * BK, r1, full_x(s));
            tma_load_2d(st + 16384, mxl, kc * BK, r0, full_x(s));
            tma_load_2d(st + 16384 + 8192, mxl, kc * BK, r1, full_x(s));
          }
        }
      }
      // drain: every issued stage must have landed before the CTA may exit
      const uint32_t issued = g;
      for (uint32_t q = issued >= NX ? issued - NX : 0; q < issued; ++q)
        mbar_wait(full_x(q % NX), (q / NX) & 1, abort_flag, err, 7, true);
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------ M producer
    if (!MT && lane == 0) {
      uint32_t g = 0;
      bool ok = true;
      int pid = 0;
      for (long long u = blockIdx.x; u < units && ok; u += gridDim.x) {
        long long lu = u;
        int mbk = kp.m_blocks, KC = kp.k_chunks;
        const CUtensorMap *mmh = &tm_mhi, *mml = &tm_mlo;
        if constexpr (G) {
          lu = locate(gd, ngd, u, pid);
          mbk = gd[pid].kp.m_blocks;
          KC = gd[pid].kp.k_chunks;
          mmh = &gd[pid].mhi;
          mml = &gd[pid].mlo;
        }
        const int mb = (int)(lu % mbk);
        for (int kc = 0; kc < KC; ++kc, ++g) {
          constexpr int ND = MT ? 1 : NM;
          const int s = (int)(g % ND);
          if (!mbar_wait(empty_m(s), ((g / ND) & 1) ^ 1, abort_flag, err, 4)) { ok = false; break; }
          const uint32_t st = sbase + kOffM + s * kMSt;
          mbar_arrive_tx(full_m(s), kMSt);
          tma_load_2d(st, mmh, kc * BK, mb * BM, full_m(s));
          tma_load_2d(st + 16384, mml, kc * BK, mb * BM, full_m(s));
          if constexpr (CX) {
            tma_load_2d(st + 32768, mmh, kc * BK, kp.ei_row + mb * BM, full_m(s));
            tma_load_2d(st + 49152, mml, kc * BK, kp.ei_row + mb * BM, full_m(s));
          }
        }
      }
      constexpr int ND = MT ? 1 : NM;
      const uint32_t issued = g;
      for (uint32_t q = issued >= ND ? issued - ND : 0; q < issued; ++q)
        mbar_wait(full_m(q % ND), (q / ND) & 1, abort_flag, err, 5, true);
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) |
                                 ((uint32_t)(BM >> 4) << 24) | (MN ? kTransB : 0u);
      constexpr uint32_t idesc64 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BR >> 3) << 17) |
                                   ((uint32_t)(BM >> 4) << 24);
      uint32_t g = 0, t = 0;
      bool ok = true;
      int pid = 0;
      if (MT) ok = mbar_wait(m_ready, 0, abort_flag, err, 10);
      for (long long u = blockIdx.x; u < units && ok; u += gridDim.x, ++t) {
        int KC = kp.k_chunks;
        if constexpr (G) {
          locate(gd, ngd, u, pid);
          KC = gd[pid].kp.k_chunks;
        }
        const int a = t & 1;
        if (!mbar_wait(acc_empty(a), ((t >> 1) & 1) ^ 1, abort_flag, err, 2)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + a * BN;
        for (int kc = 0; kc < KC; ++kc, ++g) {
          constexpr int ND = MT ? 1 : NM;
          const int sx = (int)(g % NX), sm = (int)(g % ND);
          if (!MT && !mbar_wait(full_m(sm), (g / ND) & 1, abort_flag, err, 6)) { ok = false; break; }
          if (!mbar_wait(full_x(sx), (g / NX) & 1, abort_flag, err, 3)) { ok = false; break; }
          tc_fence_after();
          const uint32_t ahi = sbase + kOffM + sm * kMSt, alo = ahi + 16384;
          const uint32_t bhi = sbase + sx * kFuXStage, blo = bhi + 16384;
#pragma unroll
          for (int ks = 0; ks < BK / 16; ++ks) {
            const uint32_t off = ks * 32;
            const uint32_t acc0 = (kc > 0 || ks > 0) ? 1u : 0u;
            // MN: k-step ks = k-rows 16 ks .. 16 ks + 15 (2048 bytes in); the
            // imaginary plane's 64 r follow 8 KB after the real plane's
            const uint64_t bh = MN ? sw128_mn_desc(bhi + ks * 2048, 8192) : sw128_desc(bhi + off);
            const uint64_t bl = MN ? sw128_mn_desc(blo + ks * 2048, 8192) : sw128_desc(blo + off);
            if constexpr (MT) {
              const uint32_t mh = tmem_base + kColM + 16 * (4 * kc + ks), ml = mh + 8;
              mma_bf16_ts(d_tmem, mh, bh, idesc, acc0);
              mma_bf16_ts(d_tmem, mh, bl, idesc, 1u);
              mma_bf16_ts(d_tmem, ml, bh, idesc, 1u);
            } else {
              mma_bf16(d_tmem, sw128_desc(ahi + off), bh, idesc, acc0);
              mma_bf16(d_tmem, sw128_desc(ahi + off), bl, idesc, 1u);
              mma_bf16(d_tmem, sw128_desc(alo + off), bh, idesc, 1u);
            }
            if constexpr (CX) {
              // Ei chunks at +32 KB (hi) and +48 KB (lo); X re rows at bhi, im rows at bhi + 8 KB
              const uint32_t eh = ahi + 32768, el = ahi + 49152;
              mma_bf16(d_tmem, sw128_desc(eh + off), sw128_desc(bhi + 8192 + off), idesc64 | kNegA, 1u);
              mma_bf16(d_tmem, sw128_desc(eh + off), sw128_desc(blo + 8192 + off), idesc64 | kNegA, 1u);
              mma_bf16(d_tmem, sw128_desc(el + off), sw128_desc(bhi + 8192 + off), idesc64 | kNegA, 1u);
              mma_bf16(d_tmem + BR, sw128_desc(eh + off), sw128_desc(bhi + off), idesc64, 1u);
              mma_bf16(d_tmem + BR, sw128_desc(eh + off), sw128_desc(blo + off), idesc64, 1u);
              mma_bf16(d_tmem + BR, sw128_desc(el + off), sw128_desc(bhi + off), idesc64, 1u);
            }
          }
          mma_commit(empty_x(sx));
          if (!MT) mma_commit(empty_m(sm));
        }
        if (!ok) break;
        mma_commit(acc_full(a));
      }
      // drain: all issued MMAs complete before TMEM is released
      mma_commit(fin_bar);
      mbar_wait(fin_bar, 0, abort_flag, err, 8, true);
    }
  }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(G ? C::kRegEpiG : C::kRegEpi));
    // ------------------------------------------------------------ epilogue
    // warp: TMEM lane quarter q, 16 rows (half) x 32 columns of each plane (the
    // 32-column half hc), walked as four pieces j of 8 rows x 16 columns: a lane
    // has 4 consecutive r of one row, and the two pieces of a row follow each
    // other, so that every 128-byte line is touched at once
    const int q = warp & 3, half = ((warp - 4) >> 2) & 1, hc = (warp - 4) >> 3;
    const int row = q * 32 + 16 * half + (lane >> 2), col = 32 * hc + frag_col(lane);
    constexpr int NI = Epi::kIn > 0 ? Epi::kIn : 1, NOP = Epi::kIn / 2;
    // position of a walk over this CTA's units: piece j of unit u is output
    // index i0 + 8 (j / 2), columns r + 16 (j % 2) .. + 3
    struct Walk {
      uint32_t u;
      int j = 0, pid = 0;
      int i0, pl;
      uint32_t r, R;
    };
    const uint32_t nunits = (uint32_t)units;   // 2 P < 2^32, so units and r fit 32 bits
    auto place = [&](Walk& w) {
      if (w.u >= nunits) return;
      uint32_t lu = w.u, mbk = (uint32_t)kp.m_blocks;
      w.R = (uint32_t)kp.R;
      w.pl = kp.p;
      if constexpr (G) {
        lu = (uint32_t)locate(gd, ngd, (long long)w.u, w.pid);
        w.R = (uint32_t)gd[w.pid].kp.R;
        mbk = (uint32_t)gd[w.pid].kp.m_blocks;
        w.pl = gd[w.pid].kp.p;
      }
      w.i0 = (int)(lu % mbk) * BM + row;
      w.r = lu / mbk * BR + col;
    };
    const Epi* const single = &epi;
    auto functor = [&](const Walk& w) { return G ? &gd[w.pid].epi : single; };
    const uint32_t ring = sbase + C::kOffEpi + (warp - 4) * C::kEpiWarp;
    // source terms fetched with the operands (single-problem forms), as many as fit one slot
    int nsf = 0;
    if constexpr (Epi::kG && !G) nsf = min(epi.g.nsrc, (C::kPlanes - Epi::kIn) / 2);
    const int planes = Epi::kIn + 2 * nsf;
    const bool ringed = planes > 0;
    const uint32_t slot = 1024u * planes;
    const int depth = ringed ? min(4, C::kPlanes / planes) : 1, ahead = depth > 1 ? depth - 1 : 1;
    Walk f;            // the block (8 rows x 32 columns) fetched next
    int fs = 0, rs = 0;   // ring slots fetched into and read from
    // two copies of 4 rows x 128 bytes per plane; 16-byte piece c of row k lands at
    // c ^ 4 (k & 1): the reads of two neighbouring rows use different banks
    const int frow = lane >> 3, fcol = 4 * (lane & 7);
    const uint32_t fdst = ring + frow * 128 + 16 * ((lane & 7) ^ (4 * (frow & 1)));
    auto fetch = [&]() {
      if (f.u < nunits) {
        const Epi& E = *functor(f);
#pragma unroll
        for (int n = 0; n < 2; ++n) {
          const int i = f.i0 - (lane >> 2) + 8 * f.j + 4 * n + frow;
          const uint32_t r = f.r - frag_col(lane) + fcol;
          if (i < f.pl && r < f.R && (f.R & 7u) == 0) {
            const uint32_t e = (uint32_t)i * f.R + r, d = fdst + fs * slot + 512 * n;
#pragma unroll
            for (int k = 0; k < NOP; ++k) {
              cp_async16(d + (2 * k) * 1024, E.src(k) + e);
              cp_async16(d + (2 * k + 1) * 1024, E.src(k) + E.P + e);
            }
            if constexpr (Epi::kG && !G) {
              for (int k = 0; k < nsf; ++k) {
                cp_async16(d + (Epi::kIn + 2 * k) * 1024, E.g.S[k] + e);
                cp_async16(d + (Epi::kIn + 2 * k + 1) * 1024, E.g.S[k] + E.P + e);
              }
            }
          }
        }
        if (++f.j == 2) {
          f.j = 0;
          f.u += gridDim.x;
          place(f);
        }
      }
      cp_async_commit();
      fs = fs + 1 == depth ? 0 : fs + 1;
    };
    if (C::kRing && ringed) {
      f.u = blockIdx.x;
      place(f);
      for (int d = 0; d < ahead; ++d) fetch();
    }
    // this lane's 16-byte piece of a block: row lane / 4, columns frag_col .. + 3 (+ 16)
    const int prow = lane >> 2, pcol = frag_col(lane) >> 2;
    Walk w;
    w.u = blockIdx.x;
    // Grouped: the descriptor's phi polynomial is no kernel parameter.  Read from global
    // memory for every element, its 24 words held up the functors with eigenvalue sums
    // (96 instances: EpiFhat 917, EpiKrog2 911 us, against 785 and 765 before the epilogue
    // took two pieces of a row at a time; ETD2RK step 4.20 against 4.09 ms).  Each warp
    // keeps a copy in shared memory: 747 and 657 us, 3.87 ms.
    const uint32_t sph = G ? sbase + kOffBar + 256 + (warp - 4) * (uint32_t)sizeof(PhiPoly) : 0u;
    int sph_pid = -1;
    uint32_t t = 0;
    for (; w.u < nunits; w.u += gridDim.x, ++t) {
      place(w);
      const int a = t & 1;
      const uint32_t tl = tmem_base + ((uint32_t)(q * 32 + 16 * half) << 16) + a * BN + 32 * hc;
      const Epi& E = *functor(w);
      if constexpr (G) {
        if (const PhiPoly* ph = poly_of(E, 0); ph && w.pid != sph_pid) {
          sph_pid = w.pid;
          __syncwarp();
          if (lane < (int)(sizeof(PhiPoly) / 4))
            asm volatile("st.shared.f32 [%0], %1;" ::"r"(sph + 4 * lane), "f"(reinterpret_cast<const float*>(ph)[lane])
                         : "memory");
          __syncwarp();
        }
      }
      // eigenvalue sums of the tile: the part of r, and lam_d of this lane's rows
      LamR<4> lr[2];
      float ld[2] = {0.f, 0.f};
      if constexpr (Epi::kLam) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (w.r + 16 * h < w.R && (w.R & 7u) == 0) lam_r<4>(E.L, w.r + 16 * h, lr[h]);
          if (w.i0 + 8 * h < w.pl) ld[h] = __ldg(E.L.lam[E.L.d - 1] + w.i0 + 8 * h);
        }
      }
      if (!mbar_wait(acc_full(a), (t >> 1) & 1, abort_flag, err, 9)) break;
      tc_fence_after();
      uint32_t vr[2][8], vi[2][8];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        tmem_ld_frag(tl + 16 * h, vr[h]);
        tmem_ld_frag(tl + 16 * h + BR, vi[h]);
      }
      tmem_wait_ld();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        tmem_loaded(vr[h]);
        tmem_loaded(vi[h]);
      }
      // the accumulator goes back to the MMA warp
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty(a));
      SplitVal em[2];   // split results of the two pieces of a block
      // a loop, not two copies of a block's code, except for the functors with most operands
      constexpr int kUnrollG = Epi::kIn == 4 ? 2 : 1;
#pragma unroll kUnrollG
      for (int g = 0; g < 2; ++g)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int i = w.i0 + 8 * g;
        const uint32_t r = w.r + 16 * h, e = (uint32_t)i * w.R + r;
        const bool live = i < w.pl && r < w.R;
        float re[4], im[4];
        frag_row(vr[h], g, lane, re);
        frag_row(vi[h], g, lane, im);
        if (C::kRing && ringed && h == 0) {
          if (ahead == 1) cp_async_wait<0>();
          else if (ahead == 2) cp_async_wait<1>();
          else cp_async_wait<2>();
          __syncwarp();              // the block has landed, and every lane is done with the one before it
          if (depth > 1) fetch();
        }
        if (live && (w.R & 7u) == 0) {
          float in[NI][4];
          const uint32_t piece = ring + rs * slot + prow * 128 + 16 * ((pcol + 4 * h) ^ (4 * (prow & 1)));
#pragma unroll
          for (int k = 0; k < 2 * NOP; ++k) lds16(piece + k * 1024, in[k]);
          float sv[4] = {0.f, 0.f, 0.f, 0.f};
          if constexpr (Epi::kLam) lam_s<4>(lr[h], g ? ld[1] : ld[0], sv);
          E.template store<4, G>(e, sv, re, im, in, SrcIn{piece + Epi::kIn * 1024, nsf, sph}, em[h]);
        } else if (live) {   // rows of odd length (d = 1): element by element
#pragma unroll 1
          for (int v = 0; v < 4; ++v) {
            if (r + v < w.R) {
              float in[NI][1];
#pragma unroll
              for (int k = 0; k < NOP; ++k) {
                in[2 * k][0] = E.src(k)[e + v];
                in[2 * k + 1][0] = E.src(k)[E.P + e + v];
              }
              const float re1[1] = {v == 0 ? re[0] : v == 1 ? re[1] : v == 2 ? re[2] : re[3]};
              const float im1[1] = {v == 0 ? im[0] : v == 1 ? im[1] : v == 2 ? im[2] : im[3]};
              float sv[1] = {0.f};
              if constexpr (Epi::kLam) {
                LamR<1> l1;
                lam_r<1>(E.L, r + v, l1);
                lam_s<1>(l1, g ? ld[1] : ld[0], sv);
              }
              E.template store<1>(e + v, sv, re1, im1, in, SrcIn{}, em[h]);
            }
          }
        }
        if (h == 1 && (w.R & 7u) == 0 && E.split().hi) {
          // 8 consecutive columns per lane: lanes 0, 1 of a quad take those of the first
          // piece, lanes 2, 3 of the second, i.e. 64 bytes per row and plane at once
          const bool high = lane & 2;
          const uint32_t c = w.r - frag_col(lane) + 16 * (high ? 1 : 0) + 8 * (lane & 1);
          const uint32_t o = (uint32_t)i * w.R + c;
          const SplitOut so = E.split();
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint2 a0 = em[0].v[k], b0 = em[1].v[k];
            const uint32_t x = __shfl_xor_sync(0xffffffffu, high ? a0.x : b0.x, 2);
            const uint32_t y = __shfl_xor_sync(0xffffffffu, high ? a0.y : b0.y, 2);
            const uint4 val = high ? make_uint4(x, y, b0.x, b0.y) : make_uint4(a0.x, a0.y, x, y);
            if (i < w.pl && c < w.R)
              *reinterpret_cast<uint4*>(((k & 1) ? so.lo : so.hi) + (k < 2 ? 0u : E.P) + o) = val;
          }
        }
        if (C::kRing && ringed && h == 1) {
          rs = rs + 1 == depth ? 0 : rs + 1;
          if (depth == 1) {
            __syncwarp();
            fetch();
          }
        }
      }
    }
    if constexpr (C::kRing) cp_async_wait<0>();   // nothing in flight when the CTA leaves
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::kTmemCols));
}

}  // namespace b3
}  // namespace fcgle
