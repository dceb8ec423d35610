// The adjoint (vector-Jacobian product) of one site's collision in 64-bit fixed point, the
// counterpart of site_fix64.cuh.
//
// With f^eq_i = w_i rho sum_pq b_pq(X, Y, t) vx^p vy^q (X = c u_s,x, Y = c u_s,y, t = T_s - 1;
// b_pq are c_pq / (omega rho) of site_fix64.cuh) the adjoint vector mu enters the product only
// through its 15 weighted moments m_pq = sum_i w_i mu_i vx^p vy^q:
//   G_rho = sum b_pq m_pq,  G_X = sum (db_pq/dX) m_pq,  G_Y,  G_t likewise (per unit density),
// and the derivatives are again low polynomials in X, Y, t, most of them coefficients b_pq of
// lower order (db40/dX = b30, db22/dX = b12, db31/dX = b21, ...).  So a site costs 37
// weightings, 53 terms of four scalar products and ~45 products for the coefficients; a
// population then costs one product, (1 - w) mu_i, and adds (evaluating four polynomials and
// their products with mu per opposite pair took 12.9 k instructions per site).
//
// Formats ([] = fraction bits).  mu is block floating point: all 37 values share the power of
// two 2^K with max |mu_i| 2^K in [2^57, 2^58) (held with one bit more).  m_pq are in units of
// 2^(-1-K), the four products of 2^(-4-K) and outputs of 2^-K.  Over the range |G| < 1.1 max|mu|
// and |out_i| < 20.4 max|mu| (the largest absolute row sums of the derivatives, omega = 2),
// below 2^62.4 units.  The error of an output is about a unit, 2^-57 of max |mu|.
// The scalar products share their cross terms (FxDot), so a term costs three multiply-adds.
//
// Range: that of the forward path (fix_scalars), and 100 <= biased exponent of max |mu| < 1078
// (or every mu zero); other sites use float64.
#pragma once
#include "site_fix64.cuh"

namespace d2q37 {

constexpr long long kFxSixth_64 = 3074457345618258603LL;  // round(2^64 / 6)

// The lattice's constants of the adjoint that FixConsts does not hold.
struct AdjFixConsts {
  int usable;
  FxHalves om1;         // 1 - omega [63]
  FxHalves omc2;        // omega c^2 [61]
  FxHalves sx, sy, st;  // c tau gx, c tau gy, tau d T_s / d tau = tau (1 - 2 tau) |g|^2 / 2 [63]
  long long tg;         // tau (1 - tau) |g|^2 / 2 [60]
};

inline AdjFixConsts make_adj_fix_consts(double tau, double gx, double gy) {
  AdjFixConsts r = {};
  const double om1 = 1.0 - 1.0 / tau, gg = gx * gx + gy * gy;
  const double sx = C * tau * gx, sy = C * tau * gy, st = tau * (1.0 - 2.0 * tau) * gg / 2.0,
               tg = tau * (1.0 - tau) * gg / 2.0;
  const auto small = [](double v) { return v > -0.125 && v < 0.125; };
  // 1 - omega [63] to 2^-30 of the format's ends, as omega in make_fix_consts
  constexpr double end = 1.0 - 0x1p-30;
  r.usable = om1 >= -end && om1 <= end && small(sx) && small(sy) && small(st) && small(tg);
  if (!r.usable) return r;
  const auto fix = [](double v, int k) {
    bool unused = false;
    return fx_from_double(v, k, 64, unused);
  };
  r.om1 = fx_halves(fix(om1, 63));
  r.omc2 = fx_halves(fix(C2 / tau, 61));
  r.sx = fx_halves(fix(sx, 63));
  r.sy = fx_halves(fix(sy, 63));
  r.st = fx_halves(fix(st, 63));
  r.tg = fix(tg, 60);
  return r;
}

// A sum of products a b, high and cross parts apart (the low words' products left out).
struct FxDot {
  long long h = 0, t = 0;
  __host__ __device__ __forceinline__ void add(FxHalves a, FxHalves b) {
    h = fx_wide(a.h, b.h, h);
    t = fx_wide(a.l, b.h, fx_wide(a.h, b.l, t));
  }
  // the sum times 2^(s - 64)
  __host__ __device__ __forceinline__ long long high(int s) const { return (h << s) + (t >> (32 - s)); }
};

// mu 2^(K + 1) rounded to an integer, by an addition to the exponent field and the float64 pipe's
// conversion (that pipe is otherwise idle but for the outputs' conversions).  K1 = (K + 1) << 20
// with 3 <= K + 1 <= 981: a field of the block's largest exponent or less stays below 1082, and a
// zero or subnormal becomes a number below 2^-41, which rounds to 0.
__host__ __device__ __forceinline__ long long fx_block(double v, int K1) {
#ifdef __CUDA_ARCH__
  return __double2ll_rn(__hiloint2double(__double2hiint(v) + K1, __double2loint(v)));
#else
  unsigned long long b;
  __builtin_memcpy(&b, &v, 8);
  b += (unsigned long long)K1 << 32;
  __builtin_memcpy(&v, &b, 8);
  return (long long)__builtin_rint(v);
#endif
}

// ---- 1. the moments of mu -----------------------------------------------------------------------
struct FixMu {
  long long m00, m10, m01, m20, m11, m02, m30, m21, m12, m03, m40, m31, m22, m13, m04;  // units 2^(-1 - K)
  long long mf;  // sum mu_i f_i, in units of 2^(k - K - 1)
};

// `io.at(i)` returns a handle of population i's pair (i, i + NPAIR), and for population i + k NPAIR
// `io.mu(h, k)` its mu, `io.fixed(h, k)` the halves of f' (fix_moments); `io.keep(h, k, q)` takes the
// halves of its mu 2^(K + 1), after the other two calls.  
template <class Io>
__host__ __device__ __forceinline__ FixMu fix_mu_moments(int K1, const FixGroup* groups,
                                                                Io&& io) {
  FixMu r;
  r.mf = 5;
  FxDot mf;
  const auto get = [&](auto at, int k, double m) {
    const long long q = fx_block(m, K1);
    const FxHalves h = fx_halves(q);
    mf.add(h, io.fixed(at, k));
    io.keep(at, k, h);
    return q;
  };
  const auto flush = [&](int e) {  // the populations' scale 2^e taken off
    r.mf += mf.high(4) >> e;
    mf = FxDot();
  };
  // w_s v: the weights are scaled by 2^e_s [63], so the product has e_s - 1 more bits than v; taking
  // e_s - 1 off leaves the sums' unit
  const auto weigh = [](long long v, FxHalves w, int e) { return fx_smul(v, w) >> (e - 1); };
  // every weighting rounds down, half a unit on average: the sums start with what they lack (the
  // sum of half their multiples); without it the bias, times |v|^2 c^2 / 2 in the outputs, is
  // 2^-53 of max |mu|
  unsigned long long m00 = 6, m20 = 17, m02 = 17, m40 = 107, m04 = 107, m22 = 21, m11 = 7, m31 = 28, m13 = 28;
  unsigned long long m10 = 8, m01 = 8, m30 = 41, m03 = 41, m12 = 13, m21 = 13;
  m00 += (unsigned long long)weigh(get(io.at(0), 0, io.mu(io.at(0), 0)), fx_halves_ct(kCw(0)), shell_exp(0));
  flush(shell_exp(0));
  // each group's mu are loaded while the group before it is worked on
  double m[4];
  const auto fetch = [&](int n) {
    const auto ai = io.at(groups[n].i), aj = io.at(groups[n].j);
    m[0] = io.mu(ai, 0), m[1] = io.mu(ai, 1), m[2] = io.mu(aj, 0), m[3] = io.mu(aj, 1);
  };
  fetch(0);
#pragma unroll 1
  for (int n = 0; n < kFixAxes; ++n) {
    const FixGroup& g = groups[n];
    const auto ai = io.at(g.i), aj = io.at(g.j);
    const double m0 = m[0], m1 = m[1], m2 = m[2], m3 = m[3];
    fetch(n + 1 < kFixGroups ? n + 1 : n);
    const long long p = get(ai, 0, m0), q = get(ai, 1, m1), u = get(aj, 0, m2), v = get(aj, 1, m3);
    flush(g.sh);
    const unsigned long long ex = (unsigned long long)weigh(p + q, g.w, g.sh), ox = (unsigned long long)weigh(p - q, g.w, g.sh);
    const unsigned long long ey = (unsigned long long)weigh(u + v, g.w, g.sh), oy = (unsigned long long)weigh(u - v, g.w, g.sh);
    m00 += ex + ey;
    m20 += g.a2 * ex;
    m02 += g.a2 * ey;
    m40 += g.a4 * ex;
    m04 += g.a4 * ey;
    m10 += g.a * ox;
    m01 += g.a * oy;
    m30 += g.a3 * ox;
    m03 += g.a3 * oy;
  }
#pragma unroll 1
  for (int n = kFixAxes; n < kFixGroups; ++n) {
    const FixGroup& g = groups[n];
    const auto ai = io.at(g.i), aj = io.at(g.j);
    const double m0 = m[0], m1 = m[1], m2 = m[2], m3 = m[3];
    fetch(n + 1 < kFixGroups ? n + 1 : n);
    const long long p = get(ai, 0, m0), q = get(ai, 1, m1), u = get(aj, 0, m2), v = get(aj, 1, m3);
    flush(g.sh);
    const long long pp = p + q, pm = p - q, up = u + v, um = u - v;
    const unsigned long long S = (unsigned long long)weigh(pp + up, g.w, g.sh), D = (unsigned long long)weigh(pp - up, g.w, g.sh);
    const unsigned long long x = (unsigned long long)weigh(pm + um, g.w, g.sh), y = (unsigned long long)weigh(pm - um, g.w, g.sh);
    m00 += S;
    m20 += g.a2 * S;
    m02 += g.b2 * S;
    m40 += g.a4 * S;
    m04 += g.b4 * S;
    m22 += (g.a2 * g.b2) * S;
    m11 += (g.a * g.b) * D;
    m31 += (g.a3 * g.b) * D;
    m13 += (g.a * g.b3) * D;
    m10 += g.a * x;
    m30 += g.a3 * x;
    m12 += (g.a * g.b2) * x;
    m01 += g.b * y;
    m03 += g.b3 * y;
    m21 += (g.a2 * g.b) * y;
  }
  r.m00 = (long long)m00, r.m10 = (long long)m10, r.m01 = (long long)m01, r.m20 = (long long)m20;
  r.m11 = (long long)m11, r.m02 = (long long)m02, r.m30 = (long long)m30, r.m21 = (long long)m21;
  r.m12 = (long long)m12, r.m03 = (long long)m03, r.m40 = (long long)m40, r.m31 = (long long)m31;
  r.m22 = (long long)m22, r.m13 = (long long)m13, r.m04 = (long long)m04;
  return r;
}

// ---- 2. the products with the equilibrium's derivatives, and the outputs' terms ---------------------
struct FixVjp {
  // out_i = (1 - w) mu_i + R + E |v_i|^2 + Bx vx + By vy
  long long R, E;    // w nu_rho and w c^2 nu_E, in units of 2^(-1-K)
  long long Bx, By;  // w c nu_J, in units of 2^-K
  long long D;       // tau^2 d/dtau of the site, in units of 2^(k - K - 1)
};

// The derivatives of sum_i mu_i f^eq_i / rho, in units of 2^(-4 - K): G_rho and, per unit density, those
// with respect to X, Y and t.
struct FixGradients {
  long long Gr, GX, GY, Gt;
};

__host__ __device__ __forceinline__ FixGradients fix_gradients(const FixScalars& v, const FixMu& m) {
  const long long X = v.X, Y = v.Y, XX = v.XX, YY = v.YY, U = v.U, t = v.t;
  const FxHalves xh = fx_halves(X), yh = fx_halves(Y), xxh = fx_halves(XX), yyh = fx_halves(YY), th = fx_halves(t),
                 uh = fx_halves(U);
  const FxHalves ic2 = fx_halves(kFxInvC2_63);
  constexpr long long one = 1LL << 60;
  const long long XY = fx_smul(xh, yh);
  const FxHalves xyh = fx_halves(XY);
  const long long t2 = fx_smul(th, th), tU = fx_smul(th, uh), U2 = fx_smul(uh, uh);       // [64]
  const long long h = fx_smul(th, fx_halves(kFxC2q_64)), h2 = h * 2;                       // c^2 t / 4, twice [64]
  const long long a01 = fx_smul((t >> 1) - (tU >> 2) - t2, fx_halves(kFxC2_62)) >> 2;      // [62] -> [60]
  const long long a02 = fx_smul(t2, fx_halves(kFxC4_64));                                  // [64]
  const long long a10 = one - (U >> 5) - (t >> 3), a20 = (one >> 1) - (U >> 6) - (t >> 4) - (t >> 5);  // [60]
  const FxHalves a10h = fx_halves(a10), a20h = fx_halves(a20);
  const long long ax = fx_smul(xxh, fx_halves(kFxSixth_64)), ay = fx_smul(yyh, fx_halves(kFxSixth_64));  // X^2/6 [64]
  const FxHalves alpha = fx_halves(h2 + ax), beta = fx_halves(h2 + ay);                    // [64]
  const long long gx = h2 + (XX >> 1), gy = h2 + (YY >> 1);                                // [64]
  const long long b10 = fx_smul(xh, a10h), b01 = fx_smul(yh, a10h);                        // [60]
  // coefficients at 60 bits, as halves
  const auto h60 = [](long long c64) { return fx_halves(c64 >> 4); };
  const FxHalves B30 = h60(fx_smul(xh, alpha)), B03 = h60(fx_smul(yh, beta));
  const FxHalves B21 = h60(fx_smul(yh, fx_halves(gx))), B12 = h60(fx_smul(xh, fx_halves(gy)));
  const FxHalves XYh = h60(XY), GX2 = h60(gx), GY2 = h60(gy);
  const FxHalves m00 = fx_halves(m.m00), m10 = fx_halves(m.m10), m01 = fx_halves(m.m01), m20 = fx_halves(m.m20),
                 m11 = fx_halves(m.m11), m02 = fx_halves(m.m02), m30 = fx_halves(m.m30), m21 = fx_halves(m.m21),
                 m12 = fx_halves(m.m12), m03 = fx_halves(m.m03), m40 = fx_halves(m.m40), m31 = fx_halves(m.m31),
                 m22 = fx_halves(m.m22), m13 = fx_halves(m.m13), m04 = fx_halves(m.m04);
  // every sum below in units of 2^(-4 - K)
  FxDot g;  // G_rho
  g.add(m00, fx_halves(one - (U >> 5) - (t >> 4) + (U2 >> 7) + (tU >> 4) + (t2 >> 4)));
  g.add(m10, fx_halves(b10));
  g.add(m01, fx_halves(b01));
  g.add(m20, fx_halves(a01 + fx_smul(a20h, xxh)));
  g.add(m02, fx_halves(a01 + fx_smul(a20h, yyh)));
  g.add(m11, fx_halves(fx_smul(a20h, xyh) * 2));
  g.add(m30, B30);
  g.add(m21, B21);
  g.add(m12, B12);
  g.add(m03, B03);
  g.add(m40, h60(a02 + fx_smul(xxh, fx_halves(h + (ax >> 2)))));
  g.add(m04, h60(a02 + fx_smul(yyh, fx_halves(h + (ay >> 2)))));
  g.add(m22, h60(a02 * 2 + fx_smul(xxh, fx_halves(h)) + fx_smul(yyh, fx_halves(h + (XX >> 2)))));
  g.add(m31, h60(fx_smul(xyh, alpha)));
  g.add(m13, h60(fx_smul(xyh, beta)));
  const long long Gr = g.high(7);
  const long long cxx = fx_smul(xxh, ic2) >> 3, cyy = fx_smul(yyh, ic2) >> 3, cxy = fx_smul(xyh, ic2) >> 3;  // / c^2 [60]
  const FxHalves ncxy = fx_halves(-cxy);
  g = FxDot();  // G_X
  g.add(m00, fx_halves(fx_smul(fx_halves(b10), ic2) * -2));
  g.add(m10, fx_halves(a10 - cxx));
  g.add(m01, ncxy);
  g.add(m20, fx_halves(fx_smul(xh, fx_halves(2 * a20 - (t >> 5) - (cxx >> 1)))));
  g.add(m02, fx_halves(-(fx_smul(xh, fx_halves((t >> 4) + cyy)) >> 1)));
  g.add(m11, fx_halves(fx_smul(yh, fx_halves(2 * a20 - cxx))));
  g.add(m30, GX2);
  g.add(m21, XYh);
  g.add(m12, GY2);
  g.add(m40, B30);
  g.add(m22, B12);
  g.add(m31, B21);
  g.add(m13, B03);
  const long long GX = g.high(7);
  g = FxDot();  // G_Y
  g.add(m00, fx_halves(fx_smul(fx_halves(b01), ic2) * -2));
  g.add(m01, fx_halves(a10 - cyy));
  g.add(m10, ncxy);
  g.add(m02, fx_halves(fx_smul(yh, fx_halves(2 * a20 - (t >> 5) - (cyy >> 1)))));
  g.add(m20, fx_halves(-(fx_smul(yh, fx_halves((t >> 4) + cxx)) >> 1)));
  g.add(m11, fx_halves(fx_smul(xh, fx_halves(2 * a20 - cyy))));
  g.add(m03, GY2);
  g.add(m12, XYh);
  g.add(m21, GX2);
  g.add(m04, B03);
  g.add(m22, B21);
  g.add(m13, B12);
  g.add(m31, B30);
  const long long GY = g.high(7);
  // G_t: the orders above two share the factor c^2 / 2
  g = FxDot();
  g.add(fx_halves(m.m30 + m.m12), h60(X));
  g.add(fx_halves(m.m03 + m.m21), h60(Y));
  g.add(fx_halves(m.m31 + m.m13), XYh);
  g.add(fx_halves(m.m40 + m.m22), fx_halves(XX >> 5));
  g.add(fx_halves(m.m04 + m.m22), fx_halves(YY >> 5));
  g.add(fx_halves(m.m40 + m.m04 + 2 * m.m22), h60(h2));
  const long long high2 = fx_smul(g.high(7), fx_halves(kFxC2_62)) * 2;  // c^2 / 2
  g = FxDot();
  const long long e0 = fx_smul((one >> 1) - (U >> 6) - (t >> 3), fx_halves(kFxC2_62)) * 4;  // c^2 (1/2 - U/4 - 2t) [58]
  g.add(m00, fx_halves((U >> 4) + (t >> 3) - one));
  g.add(m10, fx_halves(-(X >> 3)));
  g.add(m01, fx_halves(-(Y >> 3)));
  g.add(m20, fx_halves(e0 - (XX >> 4) - (XX >> 5)));
  g.add(m02, fx_halves(e0 - (YY >> 4) - (YY >> 5)));
  g.add(m11, fx_halves(-((XY * 3) >> 4)));
  const long long Gt = g.high(7) + high2;
  return {Gr, GX, GY, Gt};
}

__host__ __device__ __forceinline__ FixVjp fix_vjp(const FixMoments& f, const FixScalars& v, const FixMu& m,
                                                   const FixConsts& k, const AdjFixConsts& ka) {
  const FixGradients G = fix_gradients(v, m);
  const long long Gr = G.Gr, GX = G.GX, GY = G.GY, Gt = G.Gt;
  constexpr long long one = 1LL << 60;
  // nu = (d f^eq / d(rho, J, E))^T mu through u = J / rho, T = (E / rho - |u|^2) / D (per unit
  // density): nu_rho = G_rho - G_X X0 - G_Y Y0 + G_t (|u|^2 - D T) / 2 ..., with
  // |u|^2 - (E / rho) / 2 = kap; c nu_J = c^2 G_X - X0 G_t; nu_E = G_t / 2
  const FxHalves gxh = fx_halves(GX), gyh = fx_halves(GY), gth = fx_halves(Gt);
  const FxHalves x0 = fx_halves(v.X0), y0 = fx_halves(v.Y0);
  const long long kap = (v.e + 2 * ka.tg - (v.t >> 3) - one) << 2;                 // [62], below 1.6
  const long long nR = Gr - fx_smul(gxh, x0) - fx_smul(gyh, y0) + fx_smul(gth, fx_halves(kap)) * 4;
  const FxHalves c2 = fx_halves(kFxC2_62);
  const FxHalves nx = fx_halves(fx_smul(gxh, c2) * 4 - fx_smul(gth, x0));
  const FxHalves ny = fx_halves(fx_smul(gyh, c2) * 4 - fx_smul(gth, y0));
  FixVjp r;
  r.R = (fx_smul(fx_halves(nR), k.om) + 1) >> 1;
  r.Bx = (fx_smul(nx, k.om) + 2) >> 2;
  r.By = (fx_smul(ny, k.om) + 2) >> 2;
  r.E = (fx_smul(gth, ka.omc2) + 1) >> 1;  // omega c^2 G_t / 2
  // sum mu f - rho (G_rho - (tau g) . G - tau (dT_s/dtau) G_t)
  const long long V = Gr - (fx_smul(gxh, ka.sx) + fx_smul(gyh, ka.sy) + fx_smul(gth, ka.st)) * 2;
  r.D = m.mf - (fx_smul(V, f.R << 3) >> 2);
  return r;
}

// The site's part of dL/dtau, D omega^2 2^(k - K - 1): K and kb = k in units of the exponent field.  Two
// exact scalings: either exponent alone is within what the first or a float64 factor holds, their sum
// is not (lambda and the density both large, or both small).
__host__ __device__ __forceinline__ double fix_dtau(long long D, double om2, int K, int kb) {
  const double v = om2 * fx_lower_exponent(D, K + (1 << 20));
#ifdef __CUDA_ARCH__
  return v * __hiloint2double(0x3FF00000 + kb, 0);
#else
  const unsigned long long b = (unsigned long long)(0x3FF00000 + kb) << 32;
  double s;
  __builtin_memcpy(&s, &b, 8);
  return v * s;
#endif
}

// ---- 3. the outputs ----------------------------------------------------------------------------------
// `io.held(i)` returns the halves of mu_i 2^(K + 1); `io.out(i, v)` takes the site's out_i in units
// of 2^-K.  One rolled loop over the opposite pairs (v, -v), out = (1 - w) mu + A +- B; `pairs` is
// the table c_pair_fix.
template <class Io>
__host__ __device__ __forceinline__ void fix_adj_outputs(const FixVjp& v, FxHalves om1, const PairFix* pairs, Io&& io) {
  const auto emit = [&](int i, long long add) {
    const FxHalves m = io.held(i);
    const long long t = fx_wide(m.l, om1.h, fx_wide(m.h, om1.l));
    io.out(i, fx_wide(m.h, om1.h, add) + (t >> 32));
  };
  emit(0, v.R >> 1);
#pragma unroll 2
  for (int j = 1; j <= NPAIR; ++j) {
    const PairFix p = pairs[j];
    const long long A = (v.R + v.E * p.v2) >> 1, B = v.Bx * p.vx + v.By * p.vy;
    emit(j, A + B);
    emit(j + NPAIR, A - B);
  }
}

}  // namespace d2q37
