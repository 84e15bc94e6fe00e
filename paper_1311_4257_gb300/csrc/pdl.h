// Programmatic dependent launch of the apply's kernels: a kernel may be placed
// on the SMs while the one before it on the stream still drains, and waits in
// pdl_begin for that one's results.  Every kernel that launch_pdl starts calls
// pdl_begin before its first access to global memory; what an earlier kernel of the apply
// wrote is read with ordinary loads (not through the read-only path, which a
// compiler may move above the wait).
//
// Back-to-back kernels are 2 to 3 us apart otherwise, and the last blocks of each
// drain alone: sphere of 4 wavelengths (15 kernels) 100 -> 77 us, of 32 1.40 -> 1.36
// ms.  A stream's `early` says whether to: applies of over a million points x
// right-hand sides lose by it (sphere of 64 wavelengths 4.29 -> 4.36 ms).
#pragma once
#include <utility>

#include "common.h"

namespace dfmm {

// A stream and whether its kernels may be placed early.
struct LaunchStream {
  cudaStream_t s;
  bool early;
  LaunchStream(cudaStream_t st, bool e = false) : s(st), early(e) {}
  operator cudaStream_t() const { return s; }
};

#ifdef __CUDACC__
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <class... KArgs, class... Args>
void launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, LaunchStream s, Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s.s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = s.early ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  DFMM_CUDA(cudaLaunchKernelEx(&cfg, kernel, KArgs(std::forward<Args>(args))...));
}
#endif

}  // namespace dfmm
