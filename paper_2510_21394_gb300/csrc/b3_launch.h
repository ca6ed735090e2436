// Launchers of the fused-epilogue mode products (b3_kernel.cuh), one struct per
// epilogue functor.  Their definitions (b3_launch.cuh) are instantiated in
// fused_*.cu, a few functors each, so that the kernels compile in parallel.
#pragma once

#include "b3_epilogues.cuh"
#include "b3_kernel.cuh"

namespace fcgle {

// X and M tensor maps of one launch
struct FusedMaps {
  CUtensorMap xhi, xlo, mhi, mlo;
};

template <class Epi>
struct FusedLaunch {
  static void attributes();   // shared memory of the kernels below, once per process
  // one product; natural_order: X[c][k][r] instead of X[c][r][k]
  static void single(bool natural_order, const FusedMaps& m, const b3::KParams& kp, const Epi& epi, cudaStream_t st);
  // one persistent launch over n descriptors (b3::FusedDesc<Epi>) with `units` units in all
  static void grouped(const void* descs, int n, long long units, cudaStream_t st);
};

// the complex products of the Kronecker-product exponential
template <class Epi>
struct FusedLaunchCx {
  static void attributes();
  static void single(const FusedMaps& m, const b3::KParams& kp, const Epi& epi, cudaStream_t st);
};

}  // namespace fcgle
