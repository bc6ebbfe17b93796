// Pieces shared by the hot-path kernel files: stage time, dependent launch, staged tile copies, the
// SSP-RK3 combination and the programmatic launch.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>
#include <utility>

#include "internal.h"

namespace rdg {
namespace dev {

__device__ __forceinline__ double tau_of(int kind, double omega, double t) {
  return kind == RDG_TAU_COS ? cos(omega * t) : (kind == RDG_TAU_SIN ? sin(omega * t) : 1.0);
}

__device__ __forceinline__ double stage_time(const TimeArg& ta) {
  const double t0 = ta.ts ? ta.ts->t0 : ta.t0, n = ta.ts ? (double)ta.ts->n : ta.n;
  return t0 + (n + ta.off) * ta.dt;
}

// Programmatic dependent launch: a kernel launched with programmatic stream serialization may
// start while its predecessor in the stream finishes; it must wait here before touching any
// data the predecessor reads or writes (a no-op for an ordinary launch).
__device__ __forceinline__ void wait_for_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Lets the next kernel in the stream launch once every block of this grid has executed it
// (or exited); the next kernel still waits for this grid's completion and memory before it
// reads anything this grid writes.
__device__ __forceinline__ void allow_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ void report(int* err, int bit) {
  if (err) atomicOr(err, bit);
}

// Convex combination of SSP-RK3 stages 2 and 3: (1 - c) u_n + c v with c = 1/4 or 2/3,
// evaluated as u_n + c (v - u_n).  Written as c1 u_n + c2 v with the coefficients rounded to
// FP32, c1 + c2 = 1 + 3e-8 for c = 2/3 and every step would scale the state by that factor
// (a 1.5e-5 drift over 500 steps); here the rounding of c only touches the increment.
template <typename T, int MODE>
__device__ __forceinline__ T rk_combine(T un, T v) {
  const T c = MODE == 2 ? T(0.25) : T(2.0 / 3.0);
  return fma(c, v - un, un);
}

// Batched staging: every thread first issues all of its 16-byte loads of a block's rows
// (n values, n <= BLK * NP, 16-byte aligned start) into registers, and only then stores them
// to shared memory, so a tile costs one memory round trip instead of one per loop trip.
template <typename T, int BLK, int NP>
struct Staged {
  static constexpr int V = 16 / (int)sizeof(T);
  static constexpr int IT = ((BLK * NP + V - 1) / V + BLK - 1) / BLK;
  float4 r[IT];
  T tail0;
  __device__ __forceinline__ void load(const T* g, int n) {
    const int nv = n / V;
    const float4* g4 = reinterpret_cast<const float4*>(g);
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const int i = threadIdx.x + it * BLK;
      if (i < nv) r[it] = __ldcs(g4 + i);
    }
    const int i = nv * V + threadIdx.x;
    if (threadIdx.x < V && i < n) tail0 = g[i];
  }
  __device__ __forceinline__ void store(T* sh, int n) const {
    const int nv = n / V;
    float4* s4 = reinterpret_cast<float4*>(sh);
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const int i = threadIdx.x + it * BLK;
      if (i < nv) s4[i] = r[it];
    }
    const int i = nv * V + threadIdx.x;
    if (threadIdx.x < V && i < n) sh[i] = tail0;
  }
};

template <typename T>
__device__ __forceinline__ void stage_out(T* g, const T* sh, int n) {
  constexpr int V = 16 / sizeof(T);
  const int nv = n / V;
  float4* g4 = reinterpret_cast<float4*>(g);
  const float4* s4 = reinterpret_cast<const float4*>(sh);
  for (int i = threadIdx.x; i < nv; i += blockDim.x) __stcs(g4 + i, s4[i]);
  for (int i = nv * V + threadIdx.x; i < n; i += blockDim.x) g[i] = sh[i];
}

}  // namespace dev

// Launch with programmatic stream serialization (the kernel waits for its predecessor with
// griddepcontrol.wait), so its launch and block scheduling overlap the predecessor's tail.
template <typename... KArgs, typename... Args>
inline int launch_pdl(void (*kernel)(KArgs...), unsigned grid, unsigned block, cudaStream_t s, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...) == cudaSuccess ? RDG_OK : RDG_ECUDA;
}

inline int sm_count() {
  static int cached[64] = {0};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return 1;
  if (!cached[dev]) {
    int n = 0;
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    cached[dev] = n > 0 ? n : 1;
  }
  return cached[dev];
}

}  // namespace rdg
