// One warp-strip of the fused float64 step with the fixed-point collision of site_fix64.cuh.
#pragma once
#include "site_fix64.cuh"
#include "load_paths.cuh"

namespace d2q37 {

// 8-byte asynchronous global -> shared copy (sm_80+ LDGSTS), cached in L1.
__device__ __forceinline__ void cp_async8(double* smem_dst, const double* gmem_src) {
  const unsigned dst = (unsigned)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(dst), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// rho(x_s, row) of the seven source columns: lane l sums every fourth population of column
// l % 8, and two shuffles add the four parts (the same value in the column's four lanes).
template <class Ld>
__device__ __forceinline__ double wall_density_lane(const double* fin, int x, const StepScalars& a, int row,
                                                    Ld ld) {
  const int lane = threadIdx.x & 31;
  const int d = lane & 7, part = lane >> 3;
  double r = 0.0;
  if (d < 7) {
    const double* src = fin + (long long)wrap_index(x - (d - 3), a.lx) * a.pitch + row;
#pragma unroll
    for (int n = 0; n < 10; ++n) {
      const int i = 4 * n + part;
      if (i < Q) r += ld(src + i * a.pop);
    }
  }
  r += __shfl_xor_sync(0xffffffffu, r, 8);
  r += __shfl_xor_sync(0xffffffffu, r, 16);
  return r;
}

// Whether the strip at rows y0 .. y0 + 31 pulls from beyond the first or the last row.
__device__ __forceinline__ bool edge_strip(const StepScalars& a, int y0) { return y0 < 3 || y0 + 32 > a.ly - 3; }

// The pull-gather of a strip into its slots sf[i * 32] (sf: the lane's first slot), walls
// included; yc is the lane's row clamped into the lattice.  First the copies are issued
// (asynchronous when Ld caches in L1), then waited for and the ghosts of wall strips written over
// the clamped rows; in between the caller can issue other loads.
template <bool PERIODIC, class Ld>
__device__ __forceinline__ void stage_issue(const double* fin, const StepScalars& a, int x, int y0, int yc,
                                            double* __restrict__ sf, Ld ld) {
  // one pointer per source column (planes < 2^32 elements); a plane's stride and a hop in y are then
  // an addition and an immediate
  const double* col[7];
#pragma unroll
  for (int d = 0; d < 7; ++d) col[d] = fin + (unsigned)wrap_index(x - (d - 3), a.lx) * (unsigned)a.pitch;
  if (edge_strip(a, y0)) {
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const int ys = PERIODIC ? wrap_index(yc - vy(i), a.ly) : min(max(yc - vy(i), 0), a.ly - 1);
      const double* src = col[vx(i) + 3] + i * a.pop + (unsigned)ys;
      if (Ld::kL1) cp_async8(sf + i * 32, src);
      else sf[i * 32] = ld(src);
    }
  } else {
#pragma unroll
    for (int d = 0; d < 7; ++d) col[d] += (unsigned)yc;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
      const double* src = col[vx(i) + 3] + i * a.pop - vy(i);
      if (Ld::kL1) cp_async8(sf + i * 32, src);
      else sf[i * 32] = ld(src);
    }
  }
}
// The ghosts a wall gives one column: population i of the k-th row from the bottom wall, k < vy_i
// (the opposite population from the top one), from source column d.
struct WallGhost {
  unsigned char i, k, opposite, d;
};
struct WallGhosts {
  WallGhost g[32];
  int n;
};
constexpr WallGhosts wall_ghosts() {
  WallGhosts r = {};
  for (int i = 0; i < Q; ++i)
    for (int k = 0; k < vy(i); ++k) {
      r.g[r.n++] = {(unsigned char)i, (unsigned char)k, (unsigned char)(i > NPAIR ? i - NPAIR : i + NPAIR),
                    (unsigned char)(vx(i) + 3)};
    }
  return r;
}
static_assert(wall_ghosts().n <= 32, "one lane per ghost");
static __constant__ WallGhosts c_wall_ghosts = wall_ghosts();

// The wall sums are formed while the copies arrive, and one product per lane then gives all of a
// wall's 26 ghosts (in the threads that pull them it took 15, at 64 cycles of the float64 pipe each).
template <bool PERIODIC, class Ld>
__device__ __forceinline__ void stage_finish(const double* fin, const StepScalars& a, const StepWalls& w,
                                             int x, int y0, int yc, double* __restrict__ sf, Ld ld) {
  if (!PERIODIC && edge_strip(a, y0)) {
    const int lane = threadIdx.x & 31;
    double rho[2] = {};  // each wall only where the strip reaches it
    if (y0 < 3) rho[0] = wall_density_lane(fin, x, a, 0, ld);
    if (y0 + 32 > a.ly - 3) rho[1] = wall_density_lane(fin, x, a, a.ly - 1, ld);
    if (Ld::kL1) cp_async_wait_all();
    __syncwarp();
    const bool ghost = lane < wall_ghosts().n;
    const WallGhost g = c_wall_ghosts.g[ghost ? lane : 0];
    const double r0 = __shfl_sync(0xffffffffu, rho[0], g.d), r1 = __shfl_sync(0xffffffffu, rho[1], 6 - g.d);
    if (ghost && y0 < 3) sf[g.i * 32 + (g.k - lane)] = r0 * w.wall_b[g.i];
    const int top = a.ly - 1 - g.k - y0;  // the ghost's row in the strip
    if (ghost && top >= 0 && top < 32) sf[g.opposite * 32 + (top - lane)] = r1 * w.wall_t[g.opposite];
    __syncwarp();
  } else if (Ld::kL1) {
    cp_async_wait_all();
  }
}

// The relaxation's view of a site: its slots, and its column of the output state.
struct StepIo {
  const FxHalves* slots;
  double* out;
  long long pop;
  int kb;
  struct At {
    const FxHalves* f;
    double* out;
  };
  __device__ __forceinline__ At at(int i) const { return At{slots + i * 32, out + i * pop}; }
  __device__ __forceinline__ FxHalves fixed(At h, int k) const { return h.f[k * (NPAIR * 32)]; }
  __device__ __forceinline__ void put(At h, int k, long long v, int s) const {
    __stcs(k ? h.out + NPAIR * pop : h.out, fx_lower_exponent(v, ((57 + shell_exp(s)) << 20) - kb));
  }
};

// Returns whether the lane's site is still to be collided, in float64 (collide_strip_float64).
template <bool PERIODIC, class Ld>
__device__ __forceinline__ bool step_strip_fix64(const double* fin, double* __restrict__ fout, const StepScalars& a,
                                                 const StepWalls& w, int x, int y0, Ld ld, double* __restrict__ sf) {
  const int lane = threadIdx.x & 31;
  const int y = y0 + lane;
  const bool active = y < a.ly;  // the other lanes work on the last row's data and store nothing
  const int yc = active ? y : a.ly - 1;
  sf += lane;
  const int usable = a.fx.usable;  // read under the copies (48 lattices of a batch: 2.048 ms after them, 2.026 here)
  stage_issue<PERIODIC>(fin, a, x, y0, yc, sf, ld);
  stage_finish<PERIODIC>(fin, a, w, x, y0, yc, sf, ld);
  if (!usable) return active;  // uniform: the lattice's constants are outside the formats
  FxHalves* const sx = reinterpret_cast<FxHalves*>(sf);  // the same slots, as fixed point
  const FixMoments m = fix_moments([&](int i) { return sf[i * 32]; }, [&](int i, FxHalves q) { sx[i * 32] = q; });
  const FixScalars v = fix_scalars(m, a.fx);
  if (!active) return false;
  if (!v.ok) return true;
  fix_relax(v, a.fx.om1, StepIo{sx, fout + (long long)x * a.pitch + (unsigned)y, a.pop, m.kb});
  return false;
}

// The float64 collision of the lanes that step_strip_fix64 left: the whole warp gathers the strip once
// more, walls included, over the fixed-point forms.  T = 1.5 everywhere: 64 x 128 18.3 us, 501 x 1003
// 267 us, 2048 x 4096 3.87 ms a step; with each lane gathering its own site, and summing 37 wall values
// per ghost, 74, 374 and 4.26; a kernel of the float64 collision alone 18.6, 258 and 3.88.
template <bool PERIODIC, class Ld>
__device__ __forceinline__ void collide_strip_float64(const double* fin, double* fout, const StepScalars& a,
                                                      const StepWalls& w, int x, int y0, double* sf, bool left) {
  const int y = y0 + (threadIdx.x & 31), yc = min(y, a.ly - 1);
  sf += threadIdx.x & 31;
  __syncwarp();
  if (a.fx.usable) {  // else the populations are still in the slots
    stage_issue<PERIODIC>(fin, a, x, y0, yc, sf, Ld());
    stage_finish<PERIODIC>(fin, a, w, x, y0, yc, sf, Ld());
  }
  if (!left) return;
  const auto f = [&](int i) { return sf[i * 32]; };
  const SiteScalars v = site_scalars(f, a.cc, [](int, int) {});
  double* const dst = fout + (long long)x * a.pitch + (unsigned)y;
  relax_site_get(f, a.cc.om1, v.R, v.Ux, v.Uy, v.t, [&](int i, double val) { __stcs(dst + i * a.pop, val); });
}

}  // namespace d2q37
