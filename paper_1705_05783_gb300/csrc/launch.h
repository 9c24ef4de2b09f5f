// Launches that may begin while the kernel before them drains (programmatic
// dependent launch): the CTAs are placed early and wait in pdl_enter until
// that kernel has completed and its writes are visible.
#pragma once

#include "cams_internal.h"

namespace cams {

// Grids whose iteration is a chain of kernels of a few microseconds, where the
// gaps between them count (five steps at 40x40: 21.4 -> 20.7 ms).  On larger
// ones the waiting CTAs hold SMs that the kernel before them, or other members
// of an ensemble, could use: with every grid launched so a 64^3 step took 18.2
// ms instead of 17.3 and 16 members 110 instead of 91.
inline bool pdl_grid(const Geo& g) { return g.N <= 20000; }

#ifdef __CUDACC__
// At the top of a kernel that is launched so, before any access to memory
// (both are no-ops in an ordinary launch).
__device__ __forceinline__ void pdl_enter() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

inline cudaLaunchAttribute pdl_attribute() {
  cudaLaunchAttribute a{};
  a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  a.val.programmaticStreamSerializationAllowed = 1;
  return a;
}

// Whether the device can hold a cluster of `ctas` such CTAs at all (a part of it
// may not: a partition, a limit on its SMs).
template <class... P>
bool cluster_fits(void (*kern)(P...), int ctas, int threads, int smem) {
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3((unsigned)ctas);
  c.blockDim = dim3((unsigned)threads);
  c.dynamicSmemBytes = (size_t)smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)ctas;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  c.attrs = at;
  c.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &c) != cudaSuccess) n = 0;
  cudaGetLastError();
  return n > 0;
}

template <class... P, class... A>
cudaError_t launch_after(bool pdl, void (*kern)(P...), dim3 grid, int threads, int smem, cudaStream_t s,
                         A&&... args) {
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = dim3((unsigned)threads);
  c.dynamicSmemBytes = (size_t)smem;
  c.stream = s;
  cudaLaunchAttribute at[1] = {pdl_attribute()};
  c.attrs = at;
  c.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&c, kern, static_cast<P>(args)...);
}
#endif

}  // namespace cams
