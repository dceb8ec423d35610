// Load paths of the pull gathers: read-only cache, or L2 only inside a persistent kernel whose
// source buffers were written earlier in the same launch.
#pragma once
#include "collide_fp64.cuh"
#include "kernels.h"

namespace d2q37 {

// kL1: the loads may be served from L1 (sources written by earlier launches only), which
// also allows staging through L1-cached asynchronous copies.
struct LdReadOnly {
  static constexpr bool kL1 = true;
  template <class T>
  __device__ __forceinline__ T operator()(const T* p) const { return __ldg(p); }
};
struct LdL2 {
  static constexpr bool kL1 = false;
  template <class T>
  __device__ __forceinline__ T operator()(const T* p) const { return __ldcg(p); }
};

__device__ __forceinline__ int wrap_index(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

}  // namespace d2q37
