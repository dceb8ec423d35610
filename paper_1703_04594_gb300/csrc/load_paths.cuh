// Load paths of the pull gathers: ordinary cached loads, or L2 only inside a persistent kernel whose
// source buffers were written earlier in the same launch.
//
// A kernel launched by launch_dependent is resident while the kernel before it still writes what it is
// about to read.  pdl_wait() orders its later ordinary loads after those writes; read-only loads (__ldg,
// or a const __restrict__ kernel parameter) are defined only for data that nobody writes while the
// kernel is resident, so these kernels use none on states, lambda or partial sums.
#pragma once
#include "collide_fp64.cuh"
#include "kernels.h"

namespace d2q37 {

// kL1: the loads may be served from L1 (sources written by earlier launches only), which
// also allows staging through L1-cached asynchronous copies.
struct LdCached {
  static constexpr bool kL1 = true;
  template <class T>
  __device__ __forceinline__ T operator()(const T* p) const { return *p; }
};
struct LdL2 {
  static constexpr bool kL1 = false;
  template <class T>
  __device__ __forceinline__ T operator()(const T* p) const { return __ldcg(p); }
};

__device__ __forceinline__ int wrap_index(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

}  // namespace d2q37
