// Host helpers shared by the tensor-core translation units: tensor-map
// encoding through the driver entry point, programmatic dependent launch, the
// SM count.
#pragma once

#include <cuda.h>
#include <cudaTypedefs.h>

#include <cstdlib>
#include <stdexcept>
#include <utility>

#include "common.h"

namespace fcgle {

// Programmatic dependent launch of the mode-product kernels (on unless the
// environment sets FCGLE_PDL=0): the kernel may be scheduled while the previous
// kernel of the stream drains and runs its prologue meanwhile; it waits for
// that kernel's completion (griddepcontrol.wait) before any global access.
inline bool pdl_enabled() {
  static const bool on = [] {
    const char* e = std::getenv("FCGLE_PDL");
    return !(e && e[0] == '0');
  }();
  return on;
}

template <class... P, class... A>
void launch_pdl(void (*kernel)(P...), int grid, int threads, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 1 : 0;
  FCGLE_CUDA(cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...));
}

inline int num_sms() {
  static const int sms = [] {   // thread-safe one-time initialisation
    int dev = 0, m = 0;
    FCGLE_CUDA(cudaGetDevice(&dev));
    FCGLE_CUDA(cudaDeviceGetAttribute(&m, cudaDevAttrMultiProcessorCount, dev));
    return m;
  }();
  return sms;
}

inline PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = [] {
    cudaDriverEntryPointQueryResult q;
    void* p = nullptr;
    FCGLE_CUDA(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q));
    if (q != cudaDriverEntryPointSuccess || !p) throw std::runtime_error("cuTensorMapEncodeTiled unavailable");
    return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }();
  return fn;
}

}  // namespace fcgle
