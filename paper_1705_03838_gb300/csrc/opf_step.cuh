// Helpers shared by the kernels of a time step: programmatic dependent launch
// and the per-trajectory offsets of a batched launch.
#pragma once
#include <cuda_runtime.h>

#include <utility>

#include "opf_internal.h"

namespace opf {

// Programmatic dependent launch between the kernels of a step: each step
// kernel lets its successor launch once all of its own blocks have reached
// the trigger (d.pdl = 1: at the top; 2: before the final store phase), and
// waits for its predecessor grid to complete -- with its memory visible --
// before it reads or writes any buffer another kernel of the step touches
// (grid_dep_wait after a prologue that reads only setup data: twiddles,
// stencils, factors).  Every step kernel waits, so the ordering is
// transitive along the stream.  Without a programmatic launch both are
// no-ops.
__device__ __forceinline__ void grid_dep_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_trigger_at(const Dims& d, int where) {
  if (d.pdl == where) grid_dep_trigger();
}
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch with the programmatic-serialisation attribute when d.pdl is set
// (captured into a graph, the edge to the previous kernel becomes a
// programmatic dependency), plainly otherwise.
template <typename... KArgs, typename... Args>
void launch_step_kernel(const Dims& d, void (*kern)(KArgs...), dim3 g, dim3 b, size_t sm, cudaStream_t st,
                        Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = g;
  cfg.blockDim = b;
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = d.pdl ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
}

// FP64 <-> FP32 by integer operations: the conversion instructions run on the
// FP64 unit at its two lanes per clock, these at 64 a clock.  Same results;
// FP32 subnormals, infinities and NaN take the instruction.  Narrowing only
// sets *rare for them: where the FP64 unit is the bound, the caller converts
// several values again in one branch (a branch per value becomes a predicated
// instruction, which occupies the unit all the same).
__device__ __forceinline__ float to_float(double x, bool* rare) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const unsigned e = (hi >> 20) & 0x7ffu, sign = hi & 0x80000000u;
  unsigned f = __funnelshift_r(lo, hi, 29) + 0x40000000u;      // exponent less 896 (mod 512)
  f += ((lo & 0x1fffffffu) + 0x0fffffffu + (f & 1u)) >> 29;    // to nearest, ties to even
  f = e < 873u ? sign : (f & 0x7fffffffu) | sign;              // (below half of the least subnormal: zero)
  *rare |= e - 873u < 24u || e > 1150u;
  return __uint_as_float(f);
}
__device__ __forceinline__ double to_double(float x) {
  const unsigned f = __float_as_uint(x), e = (f >> 23) & 0xffu;
  unsigned hi = ((f & 0x7fffffffu) >> 3) + 0x38000000u, lo = f << 29;
  if (e - 1u > 253u) {
    if (f << 1) return (double)x;
    hi = lo = 0u;
  }
  return __hiloint2double((int)(hi | (f & 0x80000000u)), (int)lo);
}

// x / 2 by its exponent (a multiplication takes the FP64 unit as long as an
// addition).
__device__ __forceinline__ double halved(double x) {
  const int hi = __double2hiint(x);
  const unsigned e = ((unsigned)hi >> 20) & 0x7ffu;
  return e - 2u < 0x7fdu ? __hiloint2double(hi - 0x100000, __double2loint(x)) : 0.5 * x;
}

// Batched launches: trajectory b = blockIdx.z; its buffers sit `stride` bytes
// after trajectory b-1's (stride 0: shared).  Null stays null.
template <typename P>
__device__ __forceinline__ P* bofs(P* p, long stride) {
  return p ? (P*)((char*)p + (long)blockIdx.z * stride) : p;
}

inline int device_sms() {
  static const int sms = [] {
    int dev = 0, n = 152;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 152;
  }();
  return sms;
}

}  // namespace opf
