// Kernels of float64 states: fused pull step, the separate propagate / bc / collide kernels,
// equilibrium initialisation, moments and the kinetic-energy reduction.
//
// Thread mapping: block = 32 x 4 threads (the fused step: step_block); threadIdx.x runs along y
// (the contiguous axis, Sec. 4 "column-major, Y innermost"), so each warp owns 32
// consecutive sites of one column x and every population load/store of a warp is one
// contiguous 256-byte run (shifted by the hop's vy for loads).
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "kernels.h"
#include "step_fix64.cuh"

namespace d2q37 {

namespace {

constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ int wrap(int v, int n) { return wrap_index(v, n); }

// Source column offsets x_s * pitch for hops vx = -3..3 (index vx + 3), x periodic.
__device__ __forceinline__ void source_columns(int x, const StepArgs& a, long long (&col)[7]) {
#pragma unroll
  for (int d = 0; d < 7; ++d) col[d] = (long long)wrap(x - (d - 3), a.lx) * a.pitch;
}

}  // namespace

// ---------------------------------------------------------------------------------------
// Fused step of float64 states: gather (propagate + bc) -> collide -> streaming store
// (step_fix64.cuh).  4096 x 8192: 3.65 ms, 5.4 TB/s (0.81 of the copy rate); colliding in float64, bound by
// that pipe, 15.4 ms.  Bound now by latency at 20 warps per SM with the multiply-add, ALU and float64
// pipes and issue each 55 to 58 % busy: 96 registers, and 9.5 KB of staging per warp.  24 warps
// (80 registers, the largest carveout) left too little L1 for the gather: 4.35 -> 5.41 ms for
// 2160 x 8192, 2 steps.
#ifndef LBM_FIX64_MIN_BLOCKS
#define LBM_FIX64_MIN_BLOCKS 5
#endif
extern __shared__ double step_staged[];  // 37 populations x 32 sites per warp
// The sites outside the fixed-point range, by a function that forms its indices itself and is not
// inlined, so that the kernel keeps neither its float64 values nor its arguments in registers (4096 x
// 8192, 2 steps, of ordinary strips: 7.30 ms; with the vote before the relaxation, and a second copy of
// that for mixed strips, 7.40; with the arguments kept, which spills, 7.52; no vote 7.26).
template <bool PERIODIC>
__device__ __noinline__ void step_float64_sites(const double* fin, double* fout, const StepArgs& a, bool left) {
  const int x = blockIdx.y * blockDim.y + threadIdx.y;
  collide_strip_float64<PERIODIC, LdCached>(fin, fout, a, a, x, blockIdx.x * 32, step_staged + threadIdx.y * (Q * 32),
                                            left);
}

template <bool PERIODIC>
__global__ void __launch_bounds__(128, LBM_FIX64_MIN_BLOCKS) k_step_fix64(const double* fin, double* fout, StepArgs a) {
  pdl_trigger();
  pdl_wait();
  const int x = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= a.lx) return;  // uniform per warp
  const bool left = step_strip_fix64<PERIODIC>(fin, fout, a, a, x, blockIdx.x * 32, LdCached(),
                                               step_staged + threadIdx.y * (Q * 32));
  if (__any_sync(FULL, left)) step_float64_sites<PERIODIC>(fin, fout, a, left);
}

// ---------------------------------------------------------------------------------------
// Separate kernels (the paper's propagate -> bc -> collide sequence, Sec. 5).
template <bool PERIODIC>
__global__ void __launch_bounds__(128) k_propagate_fp64(const double* __restrict__ fin,
                                                        double* __restrict__ ftmp, StepArgs a) {
  const int x = blockIdx.y * 4 + threadIdx.y;
  const int y = blockIdx.x * 32 + threadIdx.x;
  if (x >= a.lx || y >= a.ly) return;
  long long col[7];
  source_columns(x, a, col);
  double* dst = ftmp + (long long)x * a.pitch + y;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    int ys = y - vy(i);
    if (PERIODIC) ys = wrap(ys, a.ly);
    else if (ys < 0 || ys >= a.ly) continue;  // left for bc
    __stcs(dst + i * a.pop, __ldg(fin + i * a.pop + col[vx(i) + 3] + ys));
  }
}

// Push form of propagate: site (x, y) sends each of its populations to (x + vx, y + vy).
// A warp reads 32 consecutive y of one population (one aligned 256-byte run) and writes
// them shifted by the hop, so the writes are the unaligned side.  Moves that leave the fluid
// in y are dropped; the entries they would have fed from outside are left for bc.
template <bool PERIODIC>
__global__ void __launch_bounds__(128) k_propagate_push_fp64(const double* __restrict__ fin,
                                                             double* __restrict__ ftmp, StepArgs a) {
  const int x = blockIdx.y * 4 + threadIdx.y;
  const int y = blockIdx.x * 32 + threadIdx.x;
  if (x >= a.lx || y >= a.ly) return;
  long long col[7];  // destination column offsets for vx = -3..3
#pragma unroll
  for (int d = 0; d < 7; ++d) col[d] = (long long)wrap(x + (d - 3), a.lx) * a.pitch;
  const double* src = fin + (long long)x * a.pitch + y;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    int yd = y + vy(i);
    if (PERIODIC) yd = wrap(yd, a.ly);
    else if (yd < 0 || yd >= a.ly) continue;  // leaves the fluid
    __stcs(ftmp + i * a.pop + col[vx(i) + 3] + yd, __ldg(src + i * a.pop));
  }
}

// One thread per (column x, wall row r in 0..5): rows 0,1,2 and ly-3, ly-2, ly-1.
__global__ void __launch_bounds__(128) k_bc_fp64(const double* __restrict__ fin, double* __restrict__ ftmp,
                                                 StepArgs a) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= a.lx * 6) return;
  const int x = t / 6, r = t % 6;
  const bool bottom = r < 3;
  const int y = bottom ? r : a.ly - 6 + r;
  const int wall_row = bottom ? 0 : a.ly - 1;
  double* dst = ftmp + (long long)x * a.pitch + y;
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int ys = y - vy(i);
    const bool outside = bottom ? (ys < 0) : (ys >= a.ly);
    if (!outside) continue;
    const double* src = fin + (long long)wrap(x - vx(i), a.lx) * a.pitch + wall_row;
    double rw = 0.0;
#pragma unroll
    for (int j = 0; j < Q; ++j) rw += __ldg(src + j * a.pop);
    dst[i * a.pop] = rw * (bottom ? a.wall_b[i] : a.wall_t[i]);
  }
}

__global__ void __launch_bounds__(128) k_collide_fp64(const double* __restrict__ ftmp, double* __restrict__ fout,
                                                      StepArgs a) {
  const int x = blockIdx.y * 4 + threadIdx.y;
  const int y = blockIdx.x * 32 + threadIdx.x;
  if (x >= a.lx || y >= a.ly) return;
  const long long o = (long long)x * a.pitch + y;
  double f[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) f[i] = __ldg(ftmp + o + i * a.pop);
  double* dst = fout + o;
  collide_site(f, a.cc, [&](int i, double v) { __stcs(dst + i * a.pop, v); });
}

// ---------------------------------------------------------------------------------------
// f_i = f_i^eq(rho, u, T) from [lx][ly] fields: the fixed-point equilibrium of site_fix64.cuh (the
// float64 pipe converts the 37 results and little else; a float64 equilibrium's ~250 operations of
// it took 5.5 times as long), float64 for fields outside its range.
__device__ __noinline__ void init_site_float64(double rho, double X, double Y, double t, double* __restrict__ dst,
                                               long long pop) {
  double f[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) f[i] = 0.0;
  relax_site(f, 0.0, rho, X, Y, t, [&](int i, double v) { dst[i * pop] = v; });
}

__global__ void __launch_bounds__(128, 4) k_init_fp64(const double* __restrict__ rho, const double* __restrict__ ux,
                                                   const double* __restrict__ uy, const double* __restrict__ T,
                                                   double* __restrict__ fout, StepArgs a) {
  const int x = blockIdx.y * 4 + threadIdx.y;
  const int y = blockIdx.x * 32 + threadIdx.x;
  if (x >= a.lx || y >= a.ly) return;
  const long long fi = (long long)x * a.ly + y;
  double* dst = fout + (long long)x * a.pitch + y;
  const double r = rho[fi], u = ux[fi], v = uy[fi], t = T[fi];
  int kb;
  const FixScalars s = fix_scalars_of(r, u, v, t, kb);
  if (s.ok) fix_relax<true>(s, FxHalves{0, 0}, StepIo{nullptr, dst, a.pop, kb});
  else init_site_float64(r, C * u, C * v, t - 1.0, dst, a.pop);
}

// The moments (integer velocity units) of a site outside the range of fix_moments' sums: sums in integers
// at the exponent of its largest population.  Terms round to 2^-54 of that or less, so that the sums are
// closer to exact than float64 ones, whose 126 operations of the float64 pipe took 1.89 ms for the fields of
// 2048 x 4096 such sites and 2.11 for the energy (now 0.83 and 0.85), and which are left to sites with an
// infinity or a NaN and to the ends of the exponent range.
__device__ __noinline__ void moments_block(const double* __restrict__ f, long long pop, double& rho, double& jx,
                                           double& jy, double& e) {
  double g[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) g[i] = __ldg(f + i * pop);
  unsigned top = 0;
#pragma unroll
  for (int i = 0; i < Q; ++i) top = max(top, fx_hi_word(g[i]) & 0x7fffffffu);
  const int E = (int)(top >> 20), k = 1077 - E;  // |g_i| 2^k < 2^55, and sum |v|^2 |g_i| 2^k < 216 2^55 < 2^63
  if (E < 55 || E > 2037) {                      // k within fix_to_double_rn's range otherwise
    moments_float64([&](int i) { return g[i]; }, rho, jx, jy, e);
    return;
  }
  bool unused = false;
  const auto fix = [&](int i) { return fx_from_double(g[i], k, 64, unused); };
  long long R = fix(0), En = 0, X = 0, Y = 0;
#pragma unroll
  for (int i = 1; i <= NPAIR; ++i) {
    const long long a = fix(i), b = fix(i + NPAIR), P = a + b, M = a - b;
    R += P;
    En += (long long)v2(i) * P;
    if (rep_vx(i) != 0) X += (long long)rep_vx(i) * M;
    if (rep_vy(i) != 0) Y += (long long)rep_vy(i) * M;
  }
  rho = fix_to_double_rn(R, k), jx = fix_to_double_rn(X, k), jy = fix_to_double_rn(Y, k), e = fix_to_double_rn(En, k);
}

// rho, c u and T of a site by the fixed-point moments and scalars of site_fix64.cuh: exact sums, four
// conversions on the float64 pipe.  The kernels below then run at the
// copy rate, given the 128 registers that keep a site's 37 loads in flight (left to itself the
// compiler took 66 and 0.48 ms): k_moments_fp64 reads and writes 2.75 GB (2048 x 4096) in 0.395 ms, 7.0 TB/s; with
// rounding sums and float64 scalars it took ~0.85 ms.  Outside the scalars' range the result is false, and
// in their places stand rho, jx, jy and e: from the same sums (T = 1.5 everywhere: 0.43 ms for the
// fields, 0.44 for the energy) or from moments_block.
__device__ __forceinline__ bool site_fields_fix(const double* __restrict__ f, long long pop, double& rho, double& x,
                                                double& y, double& T) {
  double g[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) g[i] = __ldg(f + i * pop);
  const FixMoments m = fix_moments([&](int i) { return g[i]; }, [](int, FxHalves) {});
  const FixConsts no_force = {1, {0, 0}, {0, 1 << 30}, {0, 0}, {0, 0}, 0, 0, 0};  // omega = 1, g = 0
  const FixScalars v = fix_scalars(m, no_force);
  if (!v.ok) {
    if (m.sums_ok) {  // 2 <= 60 - k <= 951
      const int k = 60 - m.kb / (1 << 20);
      rho = fix_to_double_rn(m.R, k), x = fix_to_double_rn(m.X, k), y = fix_to_double_rn(m.Y, k),
      T = fix_to_double_rn(m.E, k);
    } else {
      moments_block(f, pop, rho, x, y, T);
    }
    return false;
  }
  rho = fx_lower_exponent(m.R, (60 << 20) - m.kb);
  x = fx_lower_exponent(v.X, 64 << 20);
  y = fx_lower_exponent(v.Y, 64 << 20);
  T = fx_lower_exponent((1LL << 60) + (v.t >> 4), 60 << 20);
  return true;
}

__global__ void __launch_bounds__(128, 4) k_moments_fp64(const double* __restrict__ fin, double* __restrict__ rho,
                                                      double* __restrict__ ux, double* __restrict__ uy,
                                                      double* __restrict__ T, StepArgs a) {
  const int x = blockIdx.y * 4 + threadIdx.y;
  const int y = blockIdx.x * 32 + threadIdx.x;
  if (x >= a.lx || y >= a.ly) return;
  const long long fi = (long long)x * a.ly + y;
  double r, u, v, t;
  if (site_fields_fix(fin + (long long)x * a.pitch + y, a.pop, r, u, v, t)) {
    u *= 1.0 / C;
    v *= 1.0 / C;
  } else {
    const double inv_rho = 1.0 / r;
    u = C * u * inv_rho;
    v = C * v * inv_rho;
    t = (C2 * t * inv_rho - fma(u, u, v * v)) / D;
  }
  rho[fi] = r;
  ux[fi] = u;
  uy[fi] = v;
  T[fi] = t;
}

// Kinetic energy: per-block partial sums (fixed order), then k_reduce_sum adds the partials.
__global__ void __launch_bounds__(128, 4) k_ke_partial_fp64(const double* __restrict__ fin, double* __restrict__ part,
                                                         StepArgs a) {
  const int x = blockIdx.y * 4 + threadIdx.y;
  const int y = blockIdx.x * 32 + threadIdx.x;
  double ke = 0.0;
  if (x < a.lx && y < a.ly) {
    double rho, u, v, T;
    if (site_fields_fix(fin + (long long)x * a.pitch + y, a.pop, rho, u, v, T)) {
      ke = (0.5 / C2) * (rho * fma(u, u, v * v));
    } else {
      const double inv_rho = 1.0 / rho;
      u = C * u * inv_rho;
      v = C * v * inv_rho;
      ke = 0.5 * rho * fma(u, u, v * v);
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) ke += __shfl_down_sync(FULL, ke, off);
  __shared__ double warp_sum[4];
  if (threadIdx.x == 0) warp_sum[threadIdx.y] = ke;
  __syncthreads();
  if (threadIdx.x == 0 && threadIdx.y == 0)
    part[blockIdx.y * gridDim.x + blockIdx.x] = (warp_sum[0] + warp_sum[1]) + (warp_sum[2] + warp_sum[3]);
}

// Sum of part[0..n) over one block of 1024 threads in a fixed order, valid in thread 0: eight
// independent sums per thread keep as many loads in flight.
__device__ __forceinline__ double block_sum_1024(const double* __restrict__ part, long long n) {
  double v[8] = {};
  for (long long i = threadIdx.x; i < n; i += 8 * 1024) {
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (i + j * 1024 < n) v[j] += part[i + j * 1024];
  }
  double s = ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(FULL, s, off);
  __shared__ double ws[32];
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
  __syncthreads();
  double t = threadIdx.x < 32 ? ws[threadIdx.x] : 0.0;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) t += __shfl_down_sync(FULL, t, off);
  return t;
}

// One cluster of CLUSTER blocks, each summing its part of the array; block 0 adds their sums in order
// through distributed shared memory, which may be written once every block of the cluster has started
// (the first barrier: arrived at on entry, waited for after the loads).
template <int CLUSTER>
__global__ void __launch_bounds__(1024) k_reduce_sum(const double* __restrict__ part, long long n,
                                                    double* __restrict__ out) {
  if constexpr (CLUSTER == 1) {
    const double t = block_sum_1024(part, n);
    if (threadIdx.x == 0) *out = t;
  } else {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    cluster.barrier_arrive();
    __shared__ double sums[CLUSTER];
    const long long each = (n + CLUSTER - 1) / CLUSTER, begin = each * blockIdx.x;
    const double t = block_sum_1024(part + begin, begin < n ? (n - begin < each ? n - begin : each) : 0);
    cluster.barrier_wait();
    if (threadIdx.x == 0) cluster.map_shared_rank(sums, 0)[blockIdx.x] = t;
    cluster.sync();
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      double s = 0.0;
      for (int c = 0; c < CLUSTER; ++c) s += sums[c];
      *out = s;
    }
  }
}

// ---------------------------------------------------------------------------------------
// Host-side launchers.
static inline dim3 site_grid(const StepArgs& a) { return dim3((a.ly + 31) / 32, (a.lx + 3) / 4); }
static const dim3 kSiteBlock(32, 4);

cudaError_t launch_step_fix64(const double* fin, double* fout, const StepArgs& a, cudaStream_t s) {
  const dim3 block = step_block(a);
  const size_t smem = block.y * Q * 32 * sizeof(double);
  return launch_dependent(a.periodic ? k_step_fix64<true> : k_step_fix64<false>, step_grid(a), block, smem, s, fin, fout,
                          a);
}

cudaError_t launch_propagate_fp64(const double* fin, double* ftmp, const StepArgs& a, cudaStream_t s) {
  if (a.periodic) k_propagate_fp64<true><<<site_grid(a), kSiteBlock, 0, s>>>(fin, ftmp, a);
  else k_propagate_fp64<false><<<site_grid(a), kSiteBlock, 0, s>>>(fin, ftmp, a);
  return cudaGetLastError();
}

cudaError_t launch_propagate_push_fp64(const double* fin, double* ftmp, const StepArgs& a, cudaStream_t s) {
  if (a.periodic) k_propagate_push_fp64<true><<<site_grid(a), kSiteBlock, 0, s>>>(fin, ftmp, a);
  else k_propagate_push_fp64<false><<<site_grid(a), kSiteBlock, 0, s>>>(fin, ftmp, a);
  return cudaGetLastError();
}

cudaError_t launch_bc_fp64(const double* fin, double* ftmp, const StepArgs& a, cudaStream_t s) {
  if (a.periodic) return cudaSuccess;
  const int n = a.lx * 6;
  k_bc_fp64<<<(n + 127) / 128, 128, 0, s>>>(fin, ftmp, a);
  return cudaGetLastError();
}

cudaError_t launch_collide_fp64(const double* ftmp, double* fout, const StepArgs& a, cudaStream_t s) {
  k_collide_fp64<<<site_grid(a), kSiteBlock, 0, s>>>(ftmp, fout, a);
  return cudaGetLastError();
}

cudaError_t launch_init_fp64(const double* rho, const double* ux, const double* uy, const double* T, double* f,
                             const StepArgs& a, cudaStream_t s) {
  k_init_fp64<<<site_grid(a), kSiteBlock, 0, s>>>(rho, ux, uy, T, f, a);
  return cudaGetLastError();
}

cudaError_t launch_moments_fp64(const double* f, double* rho, double* ux, double* uy, double* T,
                                const StepArgs& a, cudaStream_t s) {
  k_moments_fp64<<<site_grid(a), kSiteBlock, 0, s>>>(f, rho, ux, uy, T, a);
  return cudaGetLastError();
}

long long ke_partial_count(const StepArgs& a) {
  const dim3 g = site_grid(a);
  return (long long)g.x * g.y;
}

// One block reads at most ~60 GB/s: from 8192 partials (one round of its loads) on, a cluster of eight
// (65536 partials: 26 -> 11 us).
cudaError_t launch_reduce_sum(const double* part, long long n, double* out, cudaStream_t s) {
  if (n <= 8192) {
    k_reduce_sum<1><<<1, 1024, 0, s>>>(part, n, out);
    return cudaGetLastError();
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(8);
  cfg.blockDim = dim3(1024);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 8;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_reduce_sum<8>, part, n, out);
  const cudaError_t last = cudaGetLastError();
  return e != cudaSuccess ? e : last;
}

cudaError_t launch_kinetic_energy_fp64(const double* f, double* out, double* part, const StepArgs& a,
                                       cudaStream_t s) {
  k_ke_partial_fp64<<<site_grid(a), kSiteBlock, 0, s>>>(f, part, a);
  return launch_reduce_sum(part, ke_partial_count(a), out, s);
}

}  // namespace d2q37
