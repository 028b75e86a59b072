// Programmatic dependent launches: a chained launch is set up, down to resident
// CTAs, while the kernel before it in the stream drains.
//
// What a chained kernel may read, and how: the launch is signalled before the
// wait, so on a small grid the kernel after next can be resident while this
// one still reads the buffer that the next one writes.  The wait returns when
// the kernel before has ended and its writes are visible, to coherent loads.
// Data that any kernel in the stream writes (states, lambda, dL/dF) is
// therefore read after the wait, by ordinary loads alone: no ld.global.nc,
// no __ldg and no __restrict__ from which the compiler may make one, all of
// which promise data unchanged for the kernel's whole life.  Work items and
// masks are written once, before the first launch, and may be read either way.
#pragma once
#include <cuda_runtime.h>

namespace lbm {

// First statement of a kernel that may be chained: lets the next launch come
// up, and holds every thread until the kernel before has ended and its writes
// are visible (a launch without the attribute passes at once).
__device__ __forceinline__ void begin_chained() {
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <class Args>
cudaError_t launch_chained(void (*kernel)(const Args), int grid, int tpb, const Args& a, bool chained, cudaStream_t st) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(grid));
  cfg.blockDim = dim3(unsigned(tpb));
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, a);
}

}  // namespace lbm
