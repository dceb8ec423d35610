// Hand-written adjoint (vector-Jacobian product) of the FP64 fused step, and of the
// equilibrium initialisation and the kinetic-energy observable.
//
// The step is S = C o B o P: pull propagate P and wall bc B are linear in f (a ghost value
// is rho_w(x_s) * w_i P_i(T_wall), rho_w a sum of the source column's wall-row
// populations); collide C acts site by site (Sec. 3, eqs. "lbequation", "macro").  For
// lambda' = dL/df^{n+1}:
//   1. (k_adj_collide) at every site z, recompute f~ = B P f^n and its moments, then
//        mu_i = lambda'_i,
//        out_i = (1 - w) mu_i + w (nu_rho + nu_J . xi_i + nu_E |xi_i|^2),   w = 1/tau,
//      where nu = (d f^eq / d(rho, J, E))^T mu through u = J/rho,
//      T = (E/rho - |u|^2)/D, the gravity shift u_s = u + tau g, T_s = T + tau(1-tau)|g|^2/D
//      and the fourth-order Hermite polynomial; the site's contribution to dL/dtau is
//        sum_i mu_i d f_i'/d tau = -(1/tau^2) sum_i mu_i (f^eq_i - f~_i)
//                                   + w [G_u . g + G_t (1 - 2 tau) |g|^2 / D];
//      and the transpose of the pull is applied on the way out, as a push: out_i(z) is
//      the value of lambda_i(z - v_i) when z - v_i is a fluid site.  When it is a ghost
//      (z was fed from the wall), out_i(z) goes to a per-column slot of the wall's source
//      column instead; entries lambda_i(x) with no fluid source x + v_i are set to zero
//      by their own site;
//   2. (k_adj_walls) the wall rows: every population of (x_s, 0) receives the sum of the
//      bottom slots of column x_s, each times its ghost's weight w_i P_i(T_wall) (the
//      transpose of rho_w = sum_j f_j(x_s, 0)), and likewise at the top.
// dL/dtau partials are summed per block and then in a fixed order (deterministic).
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/lbm_d2q37.h"
#include "adjoint_fix64.cuh"
#include "kernels.h"
#include "step_fix64.cuh"

namespace d2q37 {

static_assert(D == 2.0, "nu_E = g_t / D is formed as an exact halving");

namespace {

// Vector-Jacobian product of the equilibrium f^eq_i = w_i rho P_i(s_i, U, t),
// s_i = xi_i . u_s, U = |u_s|^2, t = T_s - 1, against mu: returns
//   Grho = sum mu_i w_i P_i,            (d/d rho at fixed u_s, t)
//   Gu   = rho sum mu_i w_i (dP/ds xi_i + 2 dP/dU u_s),
//   Gt   = rho sum mu_i w_i dP/dt.
struct EqVjp {
  double Grho, Gux, Guy, Gt;
};

// Computed one opposite pair (v, -v) at a time: with s = xi_v . u_s,
// P(+-s) = E +- O, dP/ds(+-s) = Pse +- Pso, dP/dU(+-s) = PUe +- PUo, dP/dt(+-s) = Pte +- Pto,
// and S = mu_v + mu_-v, Dm = mu_v - mu_-v, the pair contributes
//   Grho: w (S E + Dm O);  Gu: w [xi (Dm Pse + S Pso) + 2 u_s (S PUe + Dm PUo)];
//   Gt: w (S Pte + Dm Pto)   (the factor rho of Gu, Gt applied at the end).
// `mu(i)` returns mu_i (read on demand, so the 37 values need not stay in registers).
template <class Mu>
__device__ __forceinline__ EqVjp eq_vjp_pairs(double rho, double usx, double usy, double t, Mu&& mu) {
  const double U = fma(usx, usx, usy * usy);
  const double Ux = C * usx, Uy = C * usy;  // s = v . (Ux, Uy)
  double Gr, Gx, Gy, Gt;
  {  // rest population: s = 0, xi = 0
    const double c0 = 1.0 - 0.5 * U - 0.5 * t * D + 0.125 * U * U + 0.25 * t * U * (D + 2.0) +
                      0.125 * t * t * D * (D + 2.0);
    const double pue = -0.5 + 0.25 * U + 0.25 * t * (D + 2.0);
    const double pt0 = -0.5 * D + 0.25 * U * (D + 2.0) + 0.25 * t * D * (D + 2.0);
    const double m = mu(0) * weight(0);
    Gr = m * c0;
    Gx = m * (2.0 * pue * usx);
    Gy = m * (2.0 * pue * usy);
    Gt = m * pt0;
  }
#pragma unroll
  for (int k = 1; k <= NPAIR; ++k) {
    const double q = C2 * (double)v2(k);
    const double xix = C * (double)rep_vx(k), xiy = C * (double)rep_vy(k);
    const double c2 = 0.5 - 0.25 * U + 0.25 * t * (q - D - 4.0);
    const double c1 = 1.0 - 0.5 * U + 0.5 * t * (q - D - 2.0);
    const double c0 = 1.0 - 0.5 * U + 0.5 * t * (q - D) + 0.125 * U * U + 0.25 * t * U * (D + 2.0 - q) +
                      0.125 * t * t * (q * q - 2.0 * (D + 2.0) * q + D * (D + 2.0));
    const double pue0 = -0.5 + 0.25 * U + 0.25 * t * (D + 2.0 - q);
    const double pt0 = 0.5 * (q - D) + 0.25 * U * (D + 2.0 - q) +
                       0.25 * t * (q * q - 2.0 * (D + 2.0) * q + D * (D + 2.0));
    const double s = fma((double)rep_vx(k), Ux, (double)rep_vy(k) * Uy);
    const double s2 = s * s;
    const double E = fma(s2, fma(s2, 1.0 / 24.0, c2), c0);
    const double O = s * fma(s2, 1.0 / 6.0, c1);
    const double Pse = fma(0.5, s2, c1);
    const double Pso = s * fma(s2, 1.0 / 6.0, 2.0 * c2);
    const double PUe = fma(-0.25, s2, pue0);
    const double PUo = -0.5 * s;
    const double Pte = fma(0.25 * (q - D - 4.0), s2, pt0);
    const double Pto = 0.5 * (q - D - 2.0) * s;
    const double w = weight(k);
    const double mp = mu(k), mm = mu(k + NPAIR);
    const double S = (mp + mm) * w, Dm = (mp - mm) * w;
    Gr = fma(S, E, fma(Dm, O, Gr));
    const double xiPart = fma(Dm, Pse, S * Pso);
    const double uPart = 2.0 * fma(S, PUe, Dm * PUo);
    Gx = fma(xix, xiPart, fma(uPart, usx, Gx));
    Gy = fma(xiy, xiPart, fma(uPart, usy, Gy));
    Gt = fma(S, Pte, fma(Dm, Pto, Gt));
  }
  return {Gr, rho * Gx, rho * Gy, rho * Gt};
}

// Ghost slots of one column: population i with vy_i > 0 fed rows 0 .. vy_i - 1 of column
// x_s + vx_i from the bottom ghosts of column x_s; those entries take bottom slots
// ghost_base(i, +1) + row of column x_s.  The top mirrors it with -vy_i and row ly - 1 - y.
__host__ __device__ constexpr int ghost_base_calc(int i, int sign) {
  int n = 0;
  for (int j = 0; j < i; ++j) n += sign * vy(j) > 0 ? sign * vy(j) : 0;
  return n;
}
constexpr int kGhostSlots = ghost_base_calc(Q, 1);  // 26 for D2Q37, the same at the top
static_assert(ghost_base_calc(Q, -1) == kGhostSlots, "the velocity set is symmetric in y");
__host__ __device__ constexpr int ghost_base(int i, int sign) {
  constexpr int b[Q] = {ghost_base_calc(0, 1),  ghost_base_calc(1, 1),  ghost_base_calc(2, 1),  ghost_base_calc(3, 1),
                        ghost_base_calc(4, 1),  ghost_base_calc(5, 1),  ghost_base_calc(6, 1),  ghost_base_calc(7, 1),
                        ghost_base_calc(8, 1),  ghost_base_calc(9, 1),  ghost_base_calc(10, 1), ghost_base_calc(11, 1),
                        ghost_base_calc(12, 1), ghost_base_calc(13, 1), ghost_base_calc(14, 1), ghost_base_calc(15, 1),
                        ghost_base_calc(16, 1), ghost_base_calc(17, 1), ghost_base_calc(18, 1), ghost_base_calc(19, 1),
                        ghost_base_calc(20, 1), ghost_base_calc(21, 1), ghost_base_calc(22, 1), ghost_base_calc(23, 1),
                        ghost_base_calc(24, 1), ghost_base_calc(25, 1), ghost_base_calc(26, 1), ghost_base_calc(27, 1),
                        ghost_base_calc(28, 1), ghost_base_calc(29, 1), ghost_base_calc(30, 1), ghost_base_calc(31, 1),
                        ghost_base_calc(32, 1), ghost_base_calc(33, 1), ghost_base_calc(34, 1), ghost_base_calc(35, 1),
                        ghost_base_calc(36, 1)};
  constexpr int t[Q] = {ghost_base_calc(0, -1),  ghost_base_calc(1, -1),  ghost_base_calc(2, -1),  ghost_base_calc(3, -1),
                        ghost_base_calc(4, -1),  ghost_base_calc(5, -1),  ghost_base_calc(6, -1),  ghost_base_calc(7, -1),
                        ghost_base_calc(8, -1),  ghost_base_calc(9, -1),  ghost_base_calc(10, -1), ghost_base_calc(11, -1),
                        ghost_base_calc(12, -1), ghost_base_calc(13, -1), ghost_base_calc(14, -1), ghost_base_calc(15, -1),
                        ghost_base_calc(16, -1), ghost_base_calc(17, -1), ghost_base_calc(18, -1), ghost_base_calc(19, -1),
                        ghost_base_calc(20, -1), ghost_base_calc(21, -1), ghost_base_calc(22, -1), ghost_base_calc(23, -1),
                        ghost_base_calc(24, -1), ghost_base_calc(25, -1), ghost_base_calc(26, -1), ghost_base_calc(27, -1),
                        ghost_base_calc(28, -1), ghost_base_calc(29, -1), ghost_base_calc(30, -1), ghost_base_calc(31, -1),
                        ghost_base_calc(32, -1), ghost_base_calc(33, -1), ghost_base_calc(34, -1), ghost_base_calc(35, -1),
                        ghost_base_calc(36, -1)};
  return sign > 0 ? b[i] : t[i];
}

// The population of each slot.
struct GhostSlots {
  unsigned char bottom[32], top[32];
};
constexpr GhostSlots ghost_slots() {
  GhostSlots r = {};
  int b = 0, t = 0;
  for (int i = 0; i < Q; ++i) {
    for (int k = 0; k < vy(i); ++k) r.bottom[b++] = (unsigned char)i;
    for (int k = 0; k < -vy(i); ++k) r.top[t++] = (unsigned char)i;
  }
  return r;
}
static_assert(kGhostSlots <= 32, "one lane per slot");
__constant__ GhostSlots c_ghost_slots = ghost_slots();

}  // namespace

// The lattice-wide scalars of the adjoint collision, formed once on the host.
struct AdjConsts {
  double om, om2;       // w = 1/tau, w^2
  double om1;           // 1 - w
  double om_c, om_c2;   // w c, w c^2
  double tgx, tgy;      // the gravity shift of the velocity, tau g
  double tshift;        // tau (1 - tau) |g|^2 / D - 1:  t = T + tshift
  double gx, gy;
  double dts_dtau;      // d T_s / d tau = (1 - 2 tau) |g|^2 / D
  AdjFixConsts fx;
};

// Scatter of a strip's outputs next to a wall or across the periodic seam.  out_i(z) is
// lambda_i(z - v_i) of the previous step (the transposed pull), or goes to the wall slot of its
// source column when z - v_i is a ghost; entries of the site whose source z + v_i lies beyond a
// wall get no push and are set to zero.
template <bool PERIODIC>
__device__ __noinline__ void push_strip_edge(const double* sf, double* __restrict__ lam_out, double* __restrict__ side,
                                             const StepArgs& a, int x, int y) {
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const int xs = wrap_index(x - vx(i), a.lx), yd = y - vy(i);
    const double val = sf[i * 32];
    if (!PERIODIC && yd < 0) {
      __stcs(side + ((long long)xs * kGhostSlots + ghost_base(i, 1) + y), val);
    } else if (!PERIODIC && yd >= a.ly) {
      __stcs(side + (((long long)a.lx + xs) * kGhostSlots + ghost_base(i, -1) + (a.ly - 1 - y)), val);
    } else {
      __stcs(lam_out + (i * a.pop + (long long)xs * a.pitch + (PERIODIC ? wrap_index(yd, a.ly) : yd)), val);
    }
    const int ys = y + vy(i);
    if (!PERIODIC && (ys < 0 || ys >= a.ly)) __stcs(lam_out + (i * a.pop + (long long)x * a.pitch + y), 0.0);
  }
}

extern __shared__ double adj_staged[];

// The adjoint collision, in float64, of the lanes of a strip that the fixed-point path left, called by
// the whole warp: their outputs to their slots and from there on, and their parts of dL/dtau returned.
// It forms its indices itself and is not inlined, so that neither they nor its arithmetic weigh on the
// register allocation of the fixed-point path.  The warp gathers the strip once more as a whole, as
// collide_strip_float64 does.  T = 1.5 everywhere: 64 x 128 56 us, 256 x 512 246, 512 x 1024 831 a step
// (each lane gathering its own site, and the fixed-point part run for nothing: 104, 344, 1069; a kernel
// that takes only the equilibrium's derivatives in float64: 54, 233, 824).
template <bool PERIODIC>
__device__ __noinline__ double adj_float64_sites(const double* fin, const double* lam_next, double* lam_out,
                                                 double* side, const StepArgs& a, const AdjConsts& k, bool left) {
  const int x = blockIdx.y * 4 + threadIdx.y, y0 = blockIdx.x * 32;
  const int y = y0 + threadIdx.x, yc = min(y, a.ly - 1);
  double* const sf = adj_staged + threadIdx.y * (Q * 32) + threadIdx.x;
  __syncwarp();
  if (a.fx.usable && k.fx.usable) {  // else the populations are still in the slots
    stage_issue<PERIODIC>(fin, a, x, y0, yc, sf, LdCached());
    stage_finish<PERIODIC>(fin, a, a, x, y0, yc, sf, LdCached());
  }
  if (!left) return 0.0;
  const double* const lam = lam_next + ((long long)x * a.pitch + (unsigned)y);
  double mu_ft = 0.0, rho, jx, jy, e;
  moments_get([&](int i) { return sf[i * 32]; }, rho, jx, jy, e, [](int, int) {});
#pragma unroll
  for (int i = 0; i < Q; ++i) {
    const double l = lam[i * a.pop];
    mu_ft = fma(l, sf[i * 32], mu_ft);
    sf[i * 32] = l;
  }
  const auto mu = [&](int i) { return sf[i * 32]; };
  const double inv = 1.0 / rho;
  const double Jx = C * jx, Jy = C * jy, E = C2 * e;  // xi-unit moments
  const double ux = Jx * inv, uy = Jy * inv;
  const double uu = fma(ux, ux, uy * uy);
  const double TD = fma(E, inv, -uu);  // D T
  const double t = fma(TD, 1.0 / D, k.tshift);
  const EqVjp G = eq_vjp_pairs(1.0, ux + k.tgx, uy + k.tgy, t, mu);  // per unit density
  // nu = (d f^eq / d(rho, J, E))^T mu through u = J / rho, T = (E / rho - |u|^2) / D:
  // the factors rho of G and 1 / rho of the chain rule cancel, and E / rho = D T + |u|^2
  const double nuE = pow2_scale(G.Gt, -1);      // gt / D, D = 2 (exact scalings on the integer pipe)
  const double m2nuE = pow2_scale(-nuE, 1);
  const double nuJx = fma(ux, m2nuE, G.Gux);
  const double nuJy = fma(uy, m2nuE, G.Guy);
  const double nuR = fma(nuE, uu - TD, G.Grho - fma(G.Gux, ux, G.Guy * uy));
  // out_{+-v} = (1-w) mu + A_s +- B_v with A_s = w (nuR + nuE c^2 |v|^2) (one per shell)
  // and B_v = w c nuJ . v (from the multiples of w c nuJ)
  const double om1 = k.om1;
  const double wR = k.om * nuR, wE = k.om_c2 * nuE;
  const Multiples wJ = make_multiples(k.om_c * nuJx, k.om_c * nuJy);
  sf[0] = fma(om1, mu(0), wR);
#pragma unroll
  for (int j = 1; j <= NPAIR; ++j) {
    const double A = fma(wE, (double)v2(j), wR);
    const double B = dot_v(wJ, rep_vx(j), rep_vy(j));
    sf[j * 32] = fma(om1, mu(j), A + B);
    sf[(j + NPAIR) * 32] = fma(om1, mu(j + NPAIR), A - B);
  }
  push_strip_edge<PERIODIC>(sf, lam_out, side, a, x, y);
  // sum_i mu_i f^eq_i = rho * Grho
  return fma(-k.om2, fma(rho, G.Grho, -mu_ft),
             (k.om * rho) * fma(G.Gux, k.gx, fma(G.Guy, k.gy, G.Gt * k.dts_dtau)));
}

// The fixed-point adjoint's view of a site: its slots, and its lambda (planes below 2^32 elements).
struct AdjIo {
  FxHalves* slots;
  const double* lam;
  unsigned pop;
  int K;  // exponent units of the outputs
  struct At {
    FxHalves* f;
    const double* lam;
  };
  __device__ __forceinline__ At at(int i) const { return At{slots + i * 32, lam + (unsigned long long)pop * (unsigned)i}; }
  __device__ __forceinline__ double mu(At h, int k) const { return *(k ? h.lam + (unsigned long long)pop * NPAIR : h.lam); }
  __device__ __forceinline__ FxHalves fixed(At h, int k) const { return h.f[k * (NPAIR * 32)]; }
  __device__ __forceinline__ void keep(At h, int k, FxHalves q) const { h.f[k * (NPAIR * 32)] = q; }
  __device__ __forceinline__ FxHalves held(int i) const { return slots[i * 32]; }
  __device__ __forceinline__ void out(int i, long long v) const {
    reinterpret_cast<double*>(slots)[i * 32] = fx_lower_exponent(v, K);
  }
};

// Step 1: per-site adjoint of the collision with the transposed propagate as its store.
// (block 32 x 4 as the forward kernels).  `side` holds 2 * lx * kGhostSlots doubles: the bottom slots of
// every column, then the top slots.  The strip's pull-gather is staged in shared memory (9.5 KB
// per warp); a slot holds f~_i, then its fixed-point form, then mu_i's, then the output.  What bounds
// it: latency at 16 warps per SM (128 registers), and 5.8 k instructions per strip, more code than
// the instruction cache holds unless the loops over populations are rolled and block barriers keep
// a block's four warps, one per scheduler, on the same code (512 x 1024: 0.236 ms without the
// barriers, 0.221 with, fully unrolled 0.247; blocks of 8 to 20 warps 0.238 to 0.338).  With lambda's
// scan under the gather's copies and each group's lambda loaded a group ahead 0.157 ms, 2.9 TB/s; the
// version in float64 and fixed point it replaces took 0.314.
template <bool PERIODIC>
__global__ void __launch_bounds__(128, 4) k_adj_collide(const double* fin, const double* lam_next, double* lam_out,
                                                     double* side, double* dtau_part, StepArgs a, AdjConsts k) {
  pdl_wait();
  const int x = blockIdx.y * 4 + threadIdx.y;
  if (x >= a.lx) return;  // uniform per warp
  const int y0 = blockIdx.x * 32;
  const int y = y0 + threadIdx.x;
  const bool active = y < a.ly;  // the other lanes work on the last row's data and store nothing
  const int yc = active ? y : a.ly - 1;
  double* const sf = adj_staged + threadIdx.y * (Q * 32) + threadIdx.x;
  FxHalves* const sx = reinterpret_cast<FxHalves*>(sf);
  const double* lam = lam_next + (long long)x * a.pitch + (unsigned)yc;
  stage_issue<PERIODIC>(fin, a, x, y0, yc, sf, LdCached());
  // the block exponent of lambda, from the high words alone (the values are loaded again below,
  // when their fixed-point forms can go to the slots at once)
  unsigned top = 0;
#pragma unroll
  for (int i = 0; i < Q; ++i)
    top = max(top, reinterpret_cast<const unsigned*>(lam + i * a.pop)[1] & 0x7fffffffu);
  stage_finish<PERIODIC>(fin, a, a, x, y0, yc, sf, LdCached());
  bool left = active;  // the lane's site is still to be taken in float64
  double contrib = 0.0;
  if (a.fx.usable && k.fx.usable) {  // uniform; else the lattice's constants are outside the formats
    __syncthreads();
    const FixMoments m = fix_moments_rolled(c_fix_groups, [&](int i) { return sf[i * 32]; }, [&](int i, FxHalves q) { sx[i * 32] = q; });
    const FixScalars v = fix_scalars(m, a.fx);
    const unsigned E = top == 0u ? 512u : top >> 20;  // all zero: any exponent
    __syncthreads();
    const int K = (1080 - (int)E) << 20;
    const bool ok = v.ok && E - 100u < 978u;
    const bool some = __any_sync(0xffffffffu, ok);  // else the rest is spared (831 against 947 us)
    const AdjIo io = {sx, lam, (unsigned)a.pop, K};
    FixMu mm = {};
    if (some) mm = fix_mu_moments(K + (1 << 20), c_fix_groups, io);
    __syncthreads();
    FixVjp r = {};
    if (some) r = fix_vjp(m, v, mm, a.fx, k.fx);
    if (top == 0u) r = FixVjp{};  // lambda = 0: no rounding residue
    __syncthreads();
    if (some) fix_adj_outputs(r, k.fx.om1, c_pair_fix, io);
    left = active && !ok;
    if (active && ok) {
      contrib = fix_dtau(r.D, k.om2, K, m.kb);
      if (edge_strip(a, y0)) {
        push_strip_edge<PERIODIC>(sf, lam_out, side, a, x, y);
      } else {
        double* col[7];  // row y of column x - vx
#pragma unroll
        for (int d = 0; d < 7; ++d)
          col[d] = lam_out + ((unsigned)wrap_index(x - (d - 3), a.lx) * (unsigned)a.pitch + (unsigned)y);
#pragma unroll
        for (int i = 0; i < Q; ++i) __stcs(col[vx(i) + 3] + i * a.pop - vy(i), sf[i * 32]);
      }
    }
  }
  if (__any_sync(0xffffffffu, left)) contrib += adj_float64_sites<PERIODIC>(fin, lam_next, lam_out, side, a, k, left);
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) contrib += __shfl_down_sync(0xffffffffu, contrib, off);
  __shared__ double warp_sum[4];
  if (threadIdx.x == 0) warp_sum[threadIdx.y] = contrib;
  __syncthreads();
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    double s = warp_sum[0];
    for (int w = 1; w < 4 && x + w < a.lx; ++w) s += warp_sum[w];  // the warps past lx have returned
    dtau_part[blockIdx.y * gridDim.x + blockIdx.x] = s;
  }
}

// Adds sum(part[0..n)) to *acc in a fixed order; one block of 256 threads.  Sixteen independent
// sums per thread keep as many loads in flight.
__device__ __forceinline__ void reduce_add_256(const double* part, long long n, double* acc) {
  double s[16] = {};
  for (long long i = threadIdx.x; i < n; i += 16 * 256) {
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (i + j * 256 < n) s[j] += part[i + j * 256];
  }
#pragma unroll
  for (int h = 8; h > 0; h >>= 1)
#pragma unroll
    for (int j = 0; j < h; ++j) s[j] += s[j + h];
  double v = s[0];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  __shared__ double ws[8];
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += ws[w];
    *acc += t;
  }
}

// Step 2: the wall rows' share of the transposed bc, after step 1 has written every
// lambda entry: lambda_j(x, 0) += sum over the bottom slots of column x of the slot's value
// times its ghost's weight w_i P_i(T_bottom), for all j (the ghost values' dependence on
// rho_w(x) = sum_j f_j(x, 0)), and likewise for row ly - 1.  One warp per column and wall: a lane
// per slot, a tree of shuffles, and each of the 37 entries receives the same value.  (One thread per
// entry, each forming its column's sum from the 26 slots, took 41 operations of the float64
// pipe a thread.)  The grid's last block adds the step's dL/dtau partials to *dtau (the reduction
// needs step 1 complete too, so it shares this launch).
__global__ void __launch_bounds__(256) k_adj_walls(const double* side, double* lam, StepArgs a,
                                                   const double* part, long long n_part,
                                                   double* dtau) {
  pdl_trigger();
  pdl_wait();
  if (blockIdx.x == gridDim.x - 1) {  // uniform per block
    reduce_add_256(part, n_part, dtau);
    return;
  }
  const int lane = threadIdx.x & 31;
  const unsigned col = blockIdx.x * 8u + (threadIdx.x >> 5);  // top * lx + x: the slot column of `side`
  if (col >= 2u * (unsigned)a.lx) return;  // uniform per warp
  const bool top = col >= (unsigned)a.lx;
  const unsigned x = top ? col - (unsigned)a.lx : col;
  double* const dst = lam + ((long long)x * a.pitch + (top ? a.ly - 1 : 0));
  const double l0 = dst[lane * a.pop], l1 = lane + 32 < Q ? dst[(lane + 32) * a.pop] : 0.0;
  double wall = 0.0;
  if (lane < kGhostSlots) {
    const double v = side[(long long)col * kGhostSlots + lane];
    wall = v * (top ? a.wall_t[c_ghost_slots.top[lane]] : a.wall_b[c_ghost_slots.bottom[lane]]);
  }
#pragma unroll
  for (int m = 16; m > 0; m >>= 1) wall += __shfl_xor_sync(0xffffffffu, wall, m);
  dst[lane * a.pop] = l0 + wall;
  if (lane + 32 < Q) dst[(lane + 32) * a.pop] = l1 + wall;
}

// Adds sum(part[0..n)) to *acc in a fixed order (one block of 256 threads).
__global__ void __launch_bounds__(256) k_reduce_add(const double* part, long long n, double* acc) {
  reduce_add_256(part, n, acc);
}

// dE/df_i for E = sum 1/2 |J|^2 / rho:  -|u|^2/2 + u . xi_i.
__global__ void __launch_bounds__(128) k_ke_grad(const double* __restrict__ f, double* __restrict__ lam, StepArgs a) {
  const int x = blockIdx.y * 4 + threadIdx.y;
  const int y = blockIdx.x * 32 + threadIdx.x;
  if (x >= a.lx || y >= a.ly) return;
  const long long o = (long long)x * a.pitch + y;
  double g[Q];
#pragma unroll
  for (int i = 0; i < Q; ++i) g[i] = __ldg(f + o + i * a.pop);
  double rho, jx, jy, e;
  moments_int(g, rho, jx, jy, e);
  const double ux = C * jx / rho, uy = C * jy / rho;
  const double h = -0.5 * fma(ux, ux, uy * uy);
#pragma unroll
  for (int i = 0; i < Q; ++i) lam[o + i * a.pop] = h + C * (ux * (double)vx(i) + uy * (double)vy(i));
}

__device__ __noinline__ EqVjp init_vjp_float64(double rho, double ux, double uy, double T, const double* __restrict__ lam,
                                               long long pop) {
  return eq_vjp_pairs(rho, ux, uy, T - 1.0, [&](int i) { return __ldg(lam + i * pop); });
}

// A site's lambda as fix_mu_moments reads it, without populations to weigh it with.
struct InitIo {
  const double* lam;
  unsigned pop;
  __device__ __forceinline__ const double* at(int i) const { return lam + (unsigned long long)pop * (unsigned)i; }
  __device__ __forceinline__ double mu(const double* h, int k) const {
    return __ldg(k ? h + (unsigned long long)pop * NPAIR : h);
  }
  __device__ __forceinline__ FxHalves fixed(const double*, int) const { return FxHalves{0, 0}; }
  __device__ __forceinline__ void keep(const double*, int, FxHalves) const {}
};

// Gradient of f^0 = f^eq(rho, u, T) with respect to the four fields, against lambda^0: the moments of
// lambda^0 in fixed point as in step 1 (256 x 512: 24 us; one float64 polynomial and its
// derivatives per opposite pair, the route of sites out of its range, took 171 us).
__global__ void __launch_bounds__(128, 4) k_init_adjoint(const double* __restrict__ rho, const double* __restrict__ ux,
                                                      const double* __restrict__ uy, const double* __restrict__ T,
                                                      const double* __restrict__ lam, double* __restrict__ g_rho,
                                                      double* __restrict__ g_ux, double* __restrict__ g_uy,
                                                      double* __restrict__ g_T, StepArgs a) {
  const int x = blockIdx.y * 4 + threadIdx.y;
  const int y = blockIdx.x * 32 + threadIdx.x;
  if (x >= a.lx || y >= a.ly) return;
  const long long fi = (long long)x * a.ly + y;
  const double* l = lam + (long long)x * a.pitch + y;
  unsigned top = 0;
#pragma unroll
  for (int i = 0; i < Q; ++i) top = max(top, __ldg(reinterpret_cast<const unsigned*>(l + i * a.pop) + 1) & 0x7fffffffu);
  const unsigned E = top == 0u ? 512u : top >> 20;
  const double r = rho[fi], u = ux[fi], v = uy[fi], t = T[fi];
  int kb;
  const FixScalars s = fix_scalars_of(r, u, v, t, kb);
  EqVjp G = {};
  if (s.ok && E - 100u < 978u) {
    const int K = (1080 - (int)E) << 20;
    const FixGradients g = fix_gradients(s, fix_mu_moments(K + (1 << 20), c_fix_groups, InitIo{l, (unsigned)a.pop}));
    if (top != 0u) {  // lambda = 0: no rounding residue
      const int K4 = K + (4 << 20);
      const double rc = r * C;
      G = {fx_lower_exponent(g.Gr, K4), rc * fx_lower_exponent(g.GX, K4), rc * fx_lower_exponent(g.GY, K4),
           r * fx_lower_exponent(g.Gt, K4)};
    }
  } else {
    G = init_vjp_float64(r, u, v, t, l, a.pop);
  }
  g_rho[fi] = G.Grho;
  g_ux[fi] = G.Gux;
  g_uy[fi] = G.Guy;
  g_T[fi] = G.Gt;
}

static inline dim3 site_grid(const StepArgs& a) { return dim3((a.ly + 31) / 32, (a.lx + 3) / 4); }

long long adjoint_partial_count(const StepArgs& a) {
  const dim3 g = site_grid(a);
  return (long long)g.x * g.y;
}

long long adjoint_side_count(const StepArgs& a) { return 2LL * a.lx * kGhostSlots; }

cudaError_t launch_adjoint_step(const double* fin, const double* lam_next, double* lam, double* side, double* part,
                                double* dtau, const StepArgs& a, double tau, double gx, double gy, cudaStream_t s) {
  const dim3 blk(32, 4);
  constexpr size_t smem = 4 * Q * 32 * sizeof(double);
  AdjConsts k;
  k.om = 1.0 / tau;
  k.om2 = k.om * k.om;
  k.om1 = 1.0 - k.om;
  k.om_c = k.om * C;
  k.om_c2 = k.om * C2;
  k.tgx = tau * gx;
  k.tgy = tau * gy;
  const double gg = gx * gx + gy * gy;
  k.tshift = tau * (1.0 - tau) * gg / D - 1.0;
  k.gx = gx;
  k.gy = gy;
  k.dts_dtau = (1.0 - 2.0 * tau) * gg / D;
  k.fx = make_adj_fix_consts(tau, gx, gy);
  const cudaError_t e = launch_dependent(a.periodic ? k_adj_collide<true> : k_adj_collide<false>, site_grid(a), blk, smem,
                                         s, fin, lam_next, lam, side, part, a, k);
  if (e != cudaSuccess) return e;
  if (a.periodic) {
    k_reduce_add<<<1, 256, 0, s>>>(part, adjoint_partial_count(a), dtau);
    return cudaGetLastError();
  }
  const unsigned walls = (2u * (unsigned)a.lx + 7) / 8;  // 8 warps a block, plus one block for the dtau sum
  return launch_dependent(k_adj_walls, dim3(walls + 1), dim3(256), 0, s, side, lam, a, part,
                          adjoint_partial_count(a), dtau);
}

cudaError_t launch_ke_grad(const double* f, double* lam, const StepArgs& a, cudaStream_t s) {
  k_ke_grad<<<site_grid(a), dim3(32, 4), 0, s>>>(f, lam, a);
  return cudaGetLastError();
}

cudaError_t launch_init_adjoint(const double* rho, const double* ux, const double* uy, const double* T,
                                const double* lam, double* g_rho, double* g_ux, double* g_uy, double* g_T,
                                const StepArgs& a, cudaStream_t s) {
  k_init_adjoint<<<site_grid(a), dim3(32, 4), 0, s>>>(rho, ux, uy, T, lam, g_rho, g_ux, g_uy, g_T, a);
  return cudaGetLastError();
}

}  // namespace d2q37

using namespace d2q37;

namespace {

int32_t status_of(cudaError_t e) { return e == cudaSuccess ? LBM_OK : LBM_ECUDA; }

bool a16(const void* p) { return p && ((uintptr_t)p % 16) == 0; }
bool a8(const void* p) { return p && ((uintptr_t)p % 8) == 0; }

}  // namespace

extern "C" {

int64_t lbm_adjoint_work_bytes(const lbm_params* p) {
  if (!params_valid(p) || p->precision != LBM_FP64) return -1;
  const StepArgs a = make_step_args(p);
  return (adjoint_side_count(a) + adjoint_partial_count(a)) * (int64_t)sizeof(double);
}

int32_t lbm_adjoint_step(const lbm_params* p, const void* f_n, const void* lam_next, void* lam_n, double* dtau_accum,
                         void* work, size_t work_bytes, void* stream) {
  if (!params_valid(p) || p->precision != LBM_FP64 || !a16(f_n) || !a16(lam_next) || !a16(lam_n) ||
      !a8(dtau_accum) || !a16(work))
    return LBM_EINVAL;
  const StepArgs a = make_step_args(p);
  const int64_t need = (adjoint_side_count(a) + adjoint_partial_count(a)) * (int64_t)sizeof(double);
  if ((int64_t)work_bytes < need || lam_next == lam_n || f_n == lam_n) return LBM_EINVAL;
  double* side = (double*)work;
  double* part = side + adjoint_side_count(a);
  return status_of(launch_adjoint_step((const double*)f_n, (const double*)lam_next, (double*)lam_n, side, part,
                                       dtau_accum, a, p->tau, p->gx, p->gy, (cudaStream_t)stream));
}

int32_t lbm_kinetic_energy_grad(const lbm_params* p, const void* f, void* lam, void* stream) {
  if (!params_valid(p) || p->precision != LBM_FP64 || !a16(f) || !a16(lam) || f == lam) return LBM_EINVAL;
  const StepArgs a = make_step_args(p);
  return status_of(launch_ke_grad((const double*)f, (double*)lam, a, (cudaStream_t)stream));
}

int32_t lbm_init_adjoint(const lbm_params* p, const double* rho, const double* ux, const double* uy, const double* T,
                         const void* lam0, double* g_rho, double* g_ux, double* g_uy, double* g_T, void* stream) {
  if (!params_valid(p) || p->precision != LBM_FP64 || !a8(rho) || !a8(ux) || !a8(uy) || !a8(T) || !a16(lam0) ||
      !a8(g_rho) || !a8(g_ux) || !a8(g_uy) || !a8(g_T))
    return LBM_EINVAL;
  const StepArgs a = make_step_args(p);
  return status_of(launch_init_adjoint(rho, ux, uy, T, (const double*)lam0, g_rho, g_ux, g_uy, g_T, a,
                                       (cudaStream_t)stream));
}

}  // extern "C"
