// Definitions of the fused-epilogue launchers (b3_launch.h).
#pragma once

#include <algorithm>
#include <cstring>
#include <mutex>
#include <stdexcept>
#include <string>

#include "b3_launch.h"
#include "tma_host.h"

namespace fcgle {

// Shared memory of a fused kernel, and the registers it is launched with, which its
// setmaxnreg split relies on.
template <class K>
void set_smem(K* kernel, uint32_t bytes) {
  FCGLE_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  cudaFuncAttributes a;
  FCGLE_CUDA(cudaFuncGetAttributes(&a, kernel));
  if (a.numRegs < b3::Cfg<b3::EpiStoreF32>::kRegLaunch)
    throw std::logic_error("fused kernel built with " + std::to_string(a.numRegs) + " registers");
}

template <class Epi>
void FusedLaunch<Epi>::attributes() {
  set_smem(b3::mp_b3_kernel<Epi, false, false, false, false>, b3::Cfg<Epi>::kSmemBytes);
  set_smem(b3::mp_b3_kernel<Epi, false, false, true, false>, b3::Cfg<Epi>::kSmemBytes);
  set_smem(b3::mp_b3_kernel<Epi, false, false, false, true>, b3::Cfg<Epi, false, true>::kSmemBytes);
  set_smem(b3::mp_b3_kernel<Epi, false, false, true, true>, b3::Cfg<Epi, false, true>::kSmemBytes);
}

template <class Epi>
void FusedLaunch<Epi>::single(bool natural_order, const FusedMaps& m, const b3::KParams& kp, const Epi& epi,
                              cudaStream_t st) {
  const long long units = kp.tiles * kp.m_blocks;
  const b3::FusedDesc<Epi>* none = nullptr;
  if (kp.p <= b3::kMtMaxP) {
    // M in tensor memory: every CTA keeps one i-block, so the grid is a multiple of m_blocks
    using C = b3::Cfg<Epi, false, true>;
    const int sms = num_sms() - num_sms() % kp.m_blocks;
    launch_pdl(natural_order ? b3::mp_b3_kernel<Epi, false, false, true, true>
                             : b3::mp_b3_kernel<Epi, false, false, false, true>,
               (int)std::min<long long>(units, sms), C::kThreads, C::kSmemBytes, st, m.xhi, m.xlo, m.mhi, m.mlo, kp,
               epi, none, 0, 0LL);
  } else {
    using C = b3::Cfg<Epi>;
    launch_pdl(natural_order ? b3::mp_b3_kernel<Epi, false, false, true, false>
                             : b3::mp_b3_kernel<Epi, false, false, false, false>,
               (int)std::min<long long>(units, num_sms()), C::kThreads, C::kSmemBytes, st, m.xhi, m.xlo, m.mhi, m.mlo,
               kp, epi, none, 0, 0LL);
  }
}

template <class Epi>
void FusedLaunch<Epi>::grouped(const void* descs, int n, long long units, cudaStream_t st) {
  static std::once_flag attr;
  std::call_once(attr, [] { set_smem(b3::mp_b3_kernel<Epi, true>, b3::Cfg<Epi>::kSmemGrouped); });
  CUtensorMap z;
  std::memset(&z, 0, sizeof(z));
  b3::KParams kp{};
  launch_pdl(b3::mp_b3_kernel<Epi, true>, (int)std::min<long long>(units, num_sms()), b3::Cfg<Epi>::kThreads,
             b3::Cfg<Epi>::kSmemGrouped, st, z, z, z, z, kp, Epi{}, static_cast<const b3::FusedDesc<Epi>*>(descs), n,
             units);
}

template <class Epi>
void FusedLaunchCx<Epi>::attributes() {
  set_smem(b3::mp_b3_kernel<Epi, false, true>, b3::Cfg<Epi, true>::kSmemBytes);
}

template <class Epi>
void FusedLaunchCx<Epi>::single(const FusedMaps& m, const b3::KParams& kp, const Epi& epi, cudaStream_t st) {
  using C = b3::Cfg<Epi, true>;
  const long long units = kp.tiles * kp.m_blocks;
  const b3::FusedDesc<Epi>* none = nullptr;
  launch_pdl(b3::mp_b3_kernel<Epi, false, true>, (int)std::min<long long>(units, num_sms()), C::kThreads,
             C::kSmemBytes, st, m.xhi, m.xlo, m.mhi, m.mlo, kp, epi, none, 0, 0LL);
}

}  // namespace fcgle
