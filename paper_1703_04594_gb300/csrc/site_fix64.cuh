// Collision of one site in 64-bit fixed point on the integer pipes.
//
// The update is collide_site's (Sec. 3, eq. "lbequation"; equilibrium and moments as in
// collide_fp64.cuh).  GB300 runs float64 at 1/64 of its float32 rate, and a float64
// collision needs ~260 operations of that pipe per site; here only the 37 conversions of the
// results back to float64 run on it.
//
// The equilibrium is expanded in the monomials vx^p vy^q, p + q <= 4, of the integer
// velocities: omega f^eq_i = w_i sum_pq c_pq vx^p vy^q, with 15 coefficients c_pq that
// depend on the site alone (X = c u_s,x, Y = c u_s,y, t = T_s - 1, U = |u_s|^2,
// R = omega rho, h = R c^2 t / 4):
//   c00 = R (1 - U/2 - t + U^2/8 + t U + t^2)
//   c10 = R (1 - U/2 - 2t) X                      c01: Y
//   c20 = R c^2 (t/2 - t U/4 - t^2) + R20 X^2     c02: Y^2     R20 = R (1/2 - U/4 - 3t/2)
//   c11 = 2 R20 X Y
//   c30 = X (2h + R X^2/6)   c21 = Y (2h + R X^2/2)   c12 = X (2h + R Y^2/2)   c03: Y, Y^2/6
//   c40 = R c^4 t^2/8 + X^2 (h + R X^2/24)            c04: Y
//   c22 = R c^4 t^2/4 + h (X^2 + Y^2) + R X^2 Y^2/4
//   c31 = X Y (2h + R X^2/6)                          c13 = X Y (2h + R Y^2/6)
// The velocity set is closed under sign changes, so the populations come in quads
// (a, b), (-a, -b), (a, -b), (-a, b) that share four sums S (even, even), D (odd, odd),
// Ox and Oy: p = S + D + Ox + Oy, S + D - Ox - Oy, S - D + Ox - Oy, S - D - Ox + Oy.  With
// |a|, |b| <= 3 every multiple is a shift or two and an add: 30 full 64-bit products make
// the coefficients of a site, and a population costs about eight 64-bit adds and two
// products, w_s p and (1 - omega) f.  (Evaluating the polynomial in s = v.u_s per opposite
// pair took 6 products per pair and 5 per shell, 4387 instructions per site in all.)
//
// Scales.  Populations of shell s are scaled by 2^e_s (w_s 2^e_s in [0.5, 1)), and the whole
// site by 2^-k, with k read off the rest population's exponent, f_0 2^(e_0 - k) in [1/4, 1/2):
// the path is the same at every density.  Numbers in [] below are fraction bits.
//   f_i 2^(e_s - k) [60], in [2^-8, 2): exact (a shift of the significand); moments [60]
//   omega f^eq / w_s [58], below 32; (1 - omega) [61]; w_s 2^e_s [63]; outputs [57]
// With every rounding counted an output carries less than one unit of 2^-57 at a scaled size of
// 1/4 to 1/2 or more, below a float64 rounding (2^-54 of it); the coefficients that large
// integers multiply carry 61 to 64 bits.
//
// Range: 2^-8 <= f_i 2^(e_s - k) < 2, 9/64 <= rho 2^-k < 1, omega rho 2^-k < 1.8, |X|, |Y| < 3/8
// (|u_s| < 0.31), |t| < 2/5, and |c tau g| < 1/8, omega <= 2 - 2^-30; other sites take the float64 collision.
#pragma once
#include "collide_fix64.cuh"

namespace d2q37 {

// ---- products of signed fixed-point numbers ------------------------------------------------
// a = hi 2^32 + lo with a signed low word: three signed 32 x 32 -> 64 products then give the
// high half of a 64-bit product (the low words' product, at most 1/4 unit and as often
// negative as positive, is left out), half a unit below the exact value on average.
struct __align__(8) FxHalves {
  int l, h;
};
__host__ __device__ __forceinline__ FxHalves fx_halves(long long a) {
  const unsigned lo = (unsigned)a;
  return FxHalves{(int)lo, (int)((unsigned)((unsigned long long)a >> 32) + (lo >> 31))};
}
// 32 x 32 -> 64 multiply(-add) of signed numbers, as the one instruction each is (from C++ sums of
// widened products the compiler makes about twice the instructions).
__host__ __device__ __forceinline__ long long fx_wide(int a, int b) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
#else
  return (long long)a * b;
#endif
}
__host__ __device__ __forceinline__ long long fx_wide(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (long long)a * b + c;
#endif
}
__host__ __device__ __forceinline__ long long fx_smul(FxHalves a, FxHalves b) {
  const long long t = fx_wide(a.l, b.h, fx_wide(a.h, b.l));
  return fx_wide(a.h, b.h, t >> 32);
}
__host__ __device__ __forceinline__ long long fx_smul(long long a, FxHalves b) { return fx_smul(fx_halves(a), b); }
__host__ __device__ __forceinline__ long long fx_smul(long long a, long long b) {
  return fx_smul(fx_halves(a), fx_halves(b));
}
constexpr long long kFxC2_62 = (long long)fx_const(C2, 1.0, 62);
constexpr long long kFxC2q_64 = (long long)fx_const(C2, 0.25, 64);          // c^2 / 4 [64]
constexpr long long kFxC4_64 = (long long)fx_const(C2, C2 * 0.125, 64);    // c^4 / 8 [64]
constexpr long long kFxInvC2_63 = (long long)(kInvC2 >> 1);                // 1 / c^2 [63]
constexpr long long kFxTwoThirds_63 = 6148914691236517205LL;               // round(2^64 / 3)
// w_s 2^e_s [63]: the constants kCw (correctly rounded from the float64 weights)

// ---- per-lattice constants -------------------------------------------------------------------
struct FixConsts {
  int usable;          // 0: the lattice's constants are outside the formats
  FxHalves om1;        // 1 - omega [61]
  FxHalves om;         // omega [62]
  FxHalves hgx, hgy;   // 2 c tau g / c^2 [63]
  long long cgx, cgy;  // c tau g [60]
  long long tc;        // tau (1 - tau) |g|^2 / 2 - |c tau g|^2 / (2 c^2) [60]
};

inline FixConsts make_fix_consts(double tau, double gx, double gy) {
  FixConsts r = {};
  const double om = 1.0 / tau, sx = C * tau * gx, sy = C * tau * gy;
  const double tc = tau * (1.0 - tau) * (gx * gx + gy * gy) / 2.0 - (sx * sx + sy * sy) / (2.0 * C2);
  const double om1 = 1.0 - om;  // as CollideConst::om1
  const auto small = [](double v) { return v > -0.125 && v < 0.125; };
  // omega [62] up to 2 - 2^-30 (tau from 0.5 + 2.4e-10): from 2 - 2^-31 on its high half would round up
  // to 2^31
  r.usable = om > 0.0 && om <= 2.0 - 0x1p-30 && om1 > -1.0 && om1 < 1.0 && small(sx) && small(sy) && small(tc);
  if (!r.usable) return r;
  // (doubles of this size are multiples of 2^-60 or round there; conversions are exact or
  // round to nearest)
  const auto fix = [](double v, int k) {
    bool unused = false;
    return fx_from_double(v, k, 64, unused);
  };
  r.om1 = fx_halves(fix(om1, 61));
  r.om = fx_halves(fix(om, 62));
  r.cgx = fix(sx, 60);
  r.cgy = fix(sy, 60);
  r.hgx = fx_halves(fix(2.0 * sx / C2, 63));
  r.hgy = fx_halves(fix(2.0 * sy / C2, 63));
  r.tc = fix(tc, 60);
  return r;
}

template <int V>
struct IntC {
  static constexpr int value = V;
};

// ---- index of a velocity -----------------------------------------------------------------------
__host__ __device__ constexpr int pop_index(int a, int b) {
  for (int i = 0; i < Q; ++i)
    if (vx(i) == a && vy(i) == b) return i;
  return -1;
}

// The groups of four populations (a, b), (-a, -b), (a, -b), (-a, b), and for the axes (a, 0),
// (-a, 0), (0, a), (0, -a), as tables for rolled loops.
struct FixGroup {
  int i, j;                               // first population of each opposite pair (the other is + 18)
  int sh;                                 // e_s
  FxHalves w;                             // w_s 2^e_s [63]
  unsigned a, b, a2, b2, a3, b3, a4, b4;  // powers of a and b
};
#define LBM_FIX_GROUP(A, B, J)                                                                                      \
  {                                                                                                               \
    pop_index(A, B), J, shell_exp(shell_of_v2(A * A + B * B)), fx_halves_ct(kCw(shell_of_v2(A * A + B * B))), A, B, \
        A *A, B *B, A *A *A, B *B *B, A *A *A *A, B *B *B *B                                                       \
  }
__host__ __device__ constexpr FxHalves fx_halves_ct(long long a) {
  return FxHalves{(int)(unsigned)a, (int)((a >> 32) + ((unsigned)a >> 31))};
}
#define LBM_FIX_GROUPS                                                                             \
  {LBM_FIX_GROUP(1, 0, pop_index(0, 1)), LBM_FIX_GROUP(2, 0, pop_index(0, 2)), LBM_FIX_GROUP(3, 0, pop_index(0, 3)), \
   LBM_FIX_GROUP(1, 1, pop_index(1, -1)), LBM_FIX_GROUP(2, 1, pop_index(2, -1)), LBM_FIX_GROUP(1, 2, pop_index(1, -2)), \
   LBM_FIX_GROUP(2, 2, pop_index(2, -2)), LBM_FIX_GROUP(3, 1, pop_index(3, -1)), LBM_FIX_GROUP(1, 3, pop_index(1, -3))}
constexpr int kFixAxes = 3, kFixGroups = 9;  // the axes first
static __constant__ FixGroup c_fix_groups[kFixGroups] = LBM_FIX_GROUPS;

// ---- 1. populations to fixed point, and the moments ---------------------------------------------
struct FixMoments {
  long long R, E, X, Y;  // sum f, sum |v|^2 f, sum vx f, sum vy f, times 2^-k [60]
  int kb;                // k << 20 (the exponent field's unit), for the results
  bool ok;               // every population in range
  bool sums_ok;          // the four sums hold, populations up to twice the range among them
};

// `load(i)` returns f_i as a float64, `keep(i, h)` stores its fixed-point form as halves; each is
// called once per population, load(i) before keep(i).
template <class Load, class Keep>
__host__ __device__ __forceinline__ FixMoments fix_moments(Load&& load, Keep&& keep) {
  // shift of the significand: exponent field + e_s - k + (60 - 52 - 1023); k from f_0, whose
  // field E0 gives f_0 2^(2 - k) in [1/4, 1/2):  k = E0 - 1023 + 2 + 2
  const double f0 = load(0);
  const unsigned E0 = fx_hi_word(f0) >> 20;
  const unsigned base = 4u - E0;  // + E + e_s: with k = E0 - 1019 the shift is E - E0 + e_s + 4
  unsigned worst = 0;
  const auto conv = [&](int i, double f) {
    const int e = shell_exp(shell(i));
    const unsigned sh = (fx_hi_word(f) >> 20) + (base + (unsigned)e);
    worst = worst > sh ? worst : sh;
    const long long q = fx_from_double_shifted(f, sh);
    keep(i, fx_halves(q));
    return q;
  };
  FixMoments m;
  m.kb = (int)((E0 - 1019u) << 20);
  long long R = (conv(0, f0) + 2) >> 2, E = 0, X = 0, Y = 0;  // e_0 = 2
  const auto axis = [&](auto ac) {
    constexpr int a = decltype(ac)::value, e = shell_exp(shell_of_v2(a * a));
    constexpr long long half = 1LL << (e - 1);
    constexpr int ix = pop_index(a, 0), jx = pop_index(-a, 0), iy = pop_index(0, a), jy = pop_index(0, -a);
    const long long p = conv(ix, load(ix)), q = conv(jx, load(jx));
    const long long r = conv(iy, load(iy)), s = conv(jy, load(jy));
    const long long T = (long long)(((unsigned long long)(p + q) + (unsigned long long)(r + s) + half) >> e);
    R += T;
    E += (long long)(a * a) * T;
    X += (long long)a * ((p - q + half) >> e);
    Y += (long long)a * ((r - s + half) >> e);
  };
  const auto quad = [&](auto ac, auto bc) {
    constexpr int a = decltype(ac)::value, b = decltype(bc)::value, e = shell_exp(shell_of_v2(a * a + b * b));
    constexpr long long half = 1LL << (e - 1);
    constexpr int i1 = pop_index(a, b), i2 = pop_index(-a, -b), i3 = pop_index(a, -b), i4 = pop_index(-a, b);
    const long long f1 = conv(i1, load(i1)), f2 = conv(i2, load(i2));
    const long long f3 = conv(i3, load(i3)), f4 = conv(i4, load(i4));
    const long long T =
        (long long)(((unsigned long long)(f1 + f2) + (unsigned long long)(f3 + f4) + half) >> e);
    const long long d = f1 - f2, g = f3 - f4;
    R += T;
    E += (long long)(a * a + b * b) * T;
    X += (long long)a * ((d + g + half) >> e);
    Y += (long long)b * ((d - g + half) >> e);
  };
  axis(IntC<1>());
  quad(IntC<1>(), IntC<1>());
  axis(IntC<2>());
  quad(IntC<2>(), IntC<1>());
  quad(IntC<1>(), IntC<2>());
  quad(IntC<2>(), IntC<2>());
  axis(IntC<3>());
  quad(IntC<3>(), IntC<1>());
  quad(IntC<1>(), IntC<3>());
  m.R = R;
  m.E = E;
  m.X = X;
  m.Y = Y;
  // shifts 0 .. 8; E0 in [128, 1078], f_0 below 2^56, keeps every result a normal float64 and
  // k below 60 (fx_lower_exponent), and rules out a sign bit, zeros, infinities and NaNs (with
  // f_0 ordinary, the others' shifts rule theirs out)
  m.ok = worst <= 8u && E0 - 128u <= 950u;
  // below 4: four of them stay below 2^64, and the sums below 8 (E, the largest, below 6.9)
  m.sums_ok = worst <= 9u && E0 - 128u <= 950u;
  return m;
}

// The same in loops over the tables above, for kernels whose code overflows the instruction cache
// (about 150 more instructions executed, 400 fewer stored).
template <class Load, class Keep>
__host__ __device__ __forceinline__ FixMoments fix_moments_rolled(const FixGroup* groups, Load&& load, Keep&& keep) {
  const double f0 = load(0);
  const unsigned E0 = fx_hi_word(f0) >> 20;
  const unsigned base = 4u - E0;
  unsigned worst = 0;
  const auto conv = [&](int i, int e, double f) {
    const unsigned sh = (fx_hi_word(f) >> 20) + (base + (unsigned)e);
    worst = worst > sh ? worst : sh;
    const long long q = fx_from_double_shifted(f, sh);
    keep(i, fx_halves(q));
    return (unsigned long long)q;
  };
  FixMoments m;
  m.kb = (int)((E0 - 1019u) << 20);
  unsigned long long R = (conv(0, 2, f0) + 2) >> 2, E = 0, X = 0, Y = 0;
#pragma unroll 1
  for (int n = 0; n < kFixAxes; ++n) {
    const FixGroup& g = groups[n];
    const int e = g.sh;
    const unsigned long long half = 1ull << (e - 1);
    const double a = load(g.i), b = load(g.i + NPAIR), c = load(g.j), d = load(g.j + NPAIR);
    const unsigned long long p = conv(g.i, e, a), q = conv(g.i + NPAIR, e, b), r = conv(g.j, e, c), s = conv(g.j + NPAIR, e, d);
    const unsigned long long T = (p + q + r + s + half) >> e;
    R += T;
    E += g.a2 * T;
    X += g.a * (unsigned long long)((long long)(p - q + half) >> e);
    Y += g.a * (unsigned long long)((long long)(r - s + half) >> e);
  }
#pragma unroll 1
  for (int n = kFixAxes; n < kFixGroups; ++n) {
    const FixGroup& g = groups[n];
    const int e = g.sh;
    const unsigned long long half = 1ull << (e - 1);
    const double a = load(g.i), b = load(g.i + NPAIR), c = load(g.j), dd = load(g.j + NPAIR);
    const unsigned long long f1 = conv(g.i, e, a), f2 = conv(g.i + NPAIR, e, b), f3 = conv(g.j, e, c), f4 = conv(g.j + NPAIR, e, dd);
    const unsigned long long T = (f1 + f2 + f3 + f4 + half) >> e;
    const unsigned long long d = f1 - f2, h = f3 - f4;
    R += T;
    E += (g.a2 + g.b2) * T;
    X += g.a * (unsigned long long)((long long)(d + h + half) >> e);
    Y += g.b * (unsigned long long)((long long)(d - h + half) >> e);
  }
  m.R = (long long)R;
  m.E = (long long)E;
  m.X = (long long)X;
  m.Y = (long long)Y;
  m.ok = worst <= 8u && E0 - 128u <= 950u;
  // below 4: four of them stay below 2^64, and the sums below 8 (E, the largest, below 6.9)
  m.sums_ok = worst <= 9u && E0 - 128u <= 950u;
  return m;
}

// ---- 2. site scalars ------------------------------------------------------------------------------
struct FixScalars {
  long long R;         // omega rho 2^-k [61]
  long long X, Y;      // c u_s [64]
  long long XX, YY, U; // X^2, Y^2, |u_s|^2 [64]
  long long t;         // T_s - 1 [64]
  long long X0, Y0;    // c u [64], before the gravity shift
  long long e;         // (T - 1) + |u|^2 / 2 [60]
  bool ok;
};

// 1 / a float32 to within a few units in its last place.
__host__ __device__ __forceinline__ float fx_rcp_seed(float v) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
#else
  return 1.0f / v;
#endif
}

// 1 / rho [60] of rho [60] in [1/8, 1): a float32 seed of 24 bits (its integer form has 30,
// so the residual is two exact 32 x 64 products) and one step y (1 + e + e^2), e^3 < 2^-63.
__host__ __device__ __forceinline__ long long fx_reciprocal(long long R) {
  const unsigned rh = (unsigned)((unsigned long long)R >> 32), rl = (unsigned)R;  // rh in [2^25, 2^28)
  const unsigned yh = (unsigned)(fx_rcp_seed((float)rh) * 36028797018963968.0f);  // [27], <= 2^30
  // rho y = (rh 2^32 + rl) yh 2^-87
  const unsigned long long pl = (unsigned long long)rl * yh;
  const unsigned long long ph = (unsigned long long)rh * yh + (pl >> 32);  // [55]
  const long long e = (((1LL << 55) - (long long)ph) << 22) - (long long)((unsigned)pl >> 10);  // 1 - rho y [77]
  const int eh = (int)(e >> 32);                                                                  // [45]
  const long long g = e + (fx_wide(eh, eh) >> 13);                                           // e + e^2 [77]
  const long long d = fx_wide((int)(g >> 32), (int)yh, (long long)(((unsigned long long)(unsigned)g * yh) >> 32));
  return ((long long)yh << 33) + ((d + (1LL << 11)) >> 12);  // y + y g, the latter [72] -> [60]
}

__host__ __device__ __forceinline__ FixScalars fix_scalars(const FixMoments& m, const FixConsts& k) {
  FixScalars s;
  // rho in [9/64, 1), |j| < 1/4, |sum |v|^2 f - 2 rho / c^2| < 1/2 (2 rho |t| / c^2 + ... < 0.4 in
  // range): what the formats below hold; unsigned compares of the offset values.  The upper ends lie
  // 2^-30 lower, where the high half of the shifted value still rounds to less than 2^31.
  const long long W = fx_smul(m.R << 3, fx_halves(kFxInvC2_63));  // rho / c^2 [62] = 2 rho / c^2 [61]
  const long long dev = m.E * 2 - W;                               // [61]
  bool ok = m.ok & ((unsigned long long)(m.R - (9LL << 54)) < (55ull << 54) - (1ull << 30)) &
            ((unsigned long long)(m.X + (1LL << 58)) < (1ull << 59) - (1ull << 28)) &
            ((unsigned long long)(m.Y + (1LL << 58)) < (1ull << 59) - (1ull << 28)) &
            ((unsigned long long)(dev + (1LL << 60)) < (1ull << 61) - (1ull << 30));
  const long long yc = fx_smul(fx_reciprocal(m.R) , fx_halves(kFxC2_62)) * 2;  // c^2 / rho [58] -> [59]
  const FxHalves y = fx_halves(yc);
  const long long X0 = fx_smul(m.X << 5, y), Y0 = fx_smul(m.Y << 5, y);  // [60]
  const long long X = X0 + k.cgx, Y = Y0 + k.cgy;
  const long long e2 = fx_smul(dev << 3, y);  // 2 (T - 1) + |u|^2 [59], so half of it [60]
  ok = ok & ((unsigned long long)(X + (3LL << 57)) < (3ull << 58)) &
       ((unsigned long long)(Y + (3LL << 57)) < (3ull << 58));
  s.X = X << 4;
  s.Y = Y << 4;
  const FxHalves xh = fx_halves(s.X), yh = fx_halves(s.Y);
  s.XX = fx_smul(xh, xh);
  s.YY = fx_smul(yh, yh);
  s.U = fx_smul(s.XX + s.YY, fx_halves(kFxInvC2_63)) * 2;
  // |u|^2 of the unshifted velocity from that of the shifted one
  const long long g = fx_smul(xh, k.hgx) + fx_smul(yh, k.hgy);  // [63]
  const long long t = e2 + k.tc - (s.U >> 5) + (g >> 4);        // [60]
  constexpr long long kT = (1LL << 61) / 5;                     // 2/5
  ok = ok & ((unsigned long long)(t + kT) < 2ull * kT);
  s.t = t << 4;
  s.R = fx_smul(m.R << 3, k.om);
  ok = ok & ((unsigned long long)s.R < (9ull << 58) / 5 * 8);
  s.X0 = X0 << 4;
  s.Y0 = Y0 << 4;
  s.e = e2;
  s.ok = ok;
  return s;
}

// The scalars of an equilibrium with the given fields (omega = 1): rho in [1/4, 1/2) 2^k, with k << 20
// in kb.  v.ok as for a collision.
__host__ __device__ __forceinline__ FixScalars fix_scalars_of(double rho, double ux, double uy, double T, int& kb) {
  FixScalars s;
  const unsigned E = fx_hi_word(rho) >> 20;  // rho 2^-k in [1/4, 1/2): k = E - 1021
  kb = (int)((E - 1021u) << 20);
  s.R = (long long)((((unsigned long long)((fx_hi_word(rho) & 0xFFFFFu) | 0x100000u) << 32) | fx_lo_word(rho)) << 7);
  const double X = C * ux, Y = C * uy, t = T - 1.0;
  // positive doubles order like their bit patterns
  const auto below = [](double v, unsigned hi) { return (fx_hi_word(v) & 0x7fffffffu) < hi; };
  s.ok = E - 128u <= 950u && below(X, 0x3FD80000u) && below(Y, 0x3FD80000u) && below(t, 0x3FD99999u);  // 3/8, 3/8, 2/5
  bool unused = false;
  s.X = fx_from_double(s.ok ? X : 0.0, 64, 64, unused);
  s.Y = fx_from_double(s.ok ? Y : 0.0, 64, 64, unused);
  s.t = fx_from_double(s.ok ? t : 0.0, 64, 64, unused);
  const FxHalves xh = fx_halves(s.X), yh = fx_halves(s.Y);
  s.XX = fx_smul(xh, xh);
  s.YY = fx_smul(yh, yh);
  s.U = fx_smul(s.XX + s.YY, fx_halves(kFxInvC2_63)) * 2;
  s.X0 = s.Y0 = s.e = 0;
  return s;
}

// ---- 3. coefficients, and the populations -------------------------------------------------------
// What the shifts and products below round off on average, put back in the even sum [58].
constexpr long long kFixMean = 3;

// `io.at(i)` returns a handle h of population i's pair (i, i + NPAIR); `io.fixed(h, k)` returns the
// halves of f' [60] and `io.put(h, k, v, s)` takes the new value 2^(e_s - k) [57] (shell s) of
// population i + k NPAIR.  (Handles, so that a rolled loop over pairs carries addresses rather than
// multiplying them out.)
// PLAIN: no population to relax, the results are omega f^eq alone (io.fixed is not called).
template <bool PLAIN = false, class Io>
__host__ __device__ __forceinline__ void fix_relax(const FixScalars& v, FxHalves om1, Io&& io) {
  const FxHalves Rh = fx_halves(v.R), th = fx_halves(v.t), Uh = fx_halves(v.U);
  const FxHalves xh = fx_halves(v.X), yh = fx_halves(v.Y), xxh = fx_halves(v.XX), yyh = fx_halves(v.YY);
  const long long Rt = fx_smul(th, Rh) * 2;                          // [62]
  const FxHalves Rth = fx_halves(Rt);
  const long long RU = fx_smul(Uh, Rh);                              // [61]
  const long long h = fx_smul(Rth, fx_halves(kFxC2q_64));            // [62]
  const long long Rt2 = fx_smul(Rth, th);                            // [62]
  const long long RtU = fx_smul(Rth, Uh);                            // [62]
  const long long RU2 = fx_smul(fx_halves(RU), Uh);                  // [61]
  const long long a01 = fx_smul(Rt - (RtU >> 1) - Rt2 * 2, fx_halves(kFxC2_62));  // [63] c^2 [62] -> [61]
  const long long a02 = fx_smul(Rt2 << 2, fx_halves(kFxC4_64));      // [64]
  const long long R1 = v.R - (RU >> 1);
  const long long R10 = R1 - Rt;                                     // [61]
  const FxHalves R20 = fx_halves(R10 - (Rt >> 1));                   // [62]
  const long long S0 = ((R1 - (Rt >> 1) + (RU2 >> 3) + (RtU >> 1) + (Rt2 >> 1)) >> 3) + kFixMean;  // c00 [58]
  const long long XY = fx_smul(xh, yh);                              // [64]
  const FxHalves xyh = fx_halves(XY);
  const long long c20 = a01 + (fx_smul(R20, xxh) >> 1), c02 = a01 + (fx_smul(R20, yyh) >> 1);  // [61]
  const long long c11 = fx_smul(R20, xyh) * 2;                                                  // [62]
  const FxHalves q = fx_halves(fx_smul(Rh, fx_halves(kFxTwoThirds_63)) << 2);                   // R / 6 [64]
  const long long A = fx_smul(q, xxh), B = fx_smul(q, yyh);                                     // [64]
  const long long h1 = h << 2;                                                                  // h [64], 2h [63]
  const FxHalves alpha = fx_halves(h1 + (A >> 1)), beta = fx_halves(h1 + (B >> 1));             // [63]
  const FxHalves R10h = fx_halves(R10);
  const long long c10 = fx_smul(xh, R10h) + 4, c01 = fx_smul(yh, R10h) + 4;  // [61], half a unit of [58] up
  const long long c30 = fx_smul(xh, alpha), c03 = fx_smul(yh, beta);                            // [63]
  const long long c21 = fx_smul(yh, fx_halves(h1 + ((A * 3) >> 1)));                            // [63]
  const long long c12 = fx_smul(xh, fx_halves(h1 + ((B * 3) >> 1)));
  const long long c31 = fx_smul(xyh, alpha), c13 = fx_smul(xyh, beta);                          // [63]
  const long long c40 = a02 + 1 + fx_smul(xxh, fx_halves(h1 + (A >> 2)));                       // [64]
  const long long c04 = a02 + 1 + fx_smul(yyh, fx_halves(h1 + (B >> 2)));
  const long long c22 = a02 * 2 + 1 + fx_smul(xxh, fx_halves(h1)) + fx_smul(yyh, fx_halves(h1 + A + (A >> 1)));
  // multiples, all [58]: S_a = a^2 c20 + a^4 c40, O_a = a c10 + a^3 c30 (and the same in y)
  const auto even = [](long long c2, long long c4, int a) {
    if (a == 1) return (c2 + (c4 >> 3)) >> 3;
    if (a == 2) return (c2 + (c4 >> 1)) >> 1;
    const long long w = c2 + c4 + (c4 >> 3);
    return w + (w >> 3);
  };
  const auto odd = [](long long c1, long long c3, int a) {
    if (a == 1) return (c1 + (c3 >> 2)) >> 3;
    if (a == 2) return (c1 + c3) >> 2;
    const long long w = c1 + c3 * 2 + (c3 >> 2);
    return (w >> 2) + (w >> 3);
  };
  // one result, w p + (1 - omega) f, from p = omega f^eq / w [58]: the cross terms of both
  // products share one sum (|p| < 25 2^58 with |w| < 0.6 2^63 in the outer shells, below
  // 2^61 in the others; |f|, |1 - omega| < 2^61: the sum stays below 2^63)
  const auto emit = [&](auto at, int k, int s, long long pv) {
    const FxHalves w = fx_halves(kCw(s)), p = fx_halves(pv);
    if constexpr (PLAIN) {
      io.put(at, k, fx_smul(p, w), s);
      return;
    }
    const FxHalves f = io.fixed(at, k);
    const long long t = fx_wide(f.l, om1.h, fx_wide(f.h, om1.l, fx_wide(p.l, w.h, fx_wide(p.h, w.l))));
    io.put(at, k, fx_wide(f.h, om1.h, fx_wide(p.h, w.h, t >> 32)), s);
  };
  // two opposite pairs (v, -v), p = P +- u, then M +- w; rolled, for the instruction cache
  const auto pairs = [&](int i, int j, int s, long long P, long long u, long long M, long long w) {
    auto at = io.at(i);
    const auto at_j = io.at(j);
#pragma unroll 1
    for (int r = 0; r < 2; ++r) {
      emit(at, 0, s, P + u);
      emit(at, 1, s, P - u);
      at = at_j;
      P = M;
      u = w;
    }
  };
  emit(io.at(0), 0, 0, S0 - 2);  // its share of the sums' mean is less
  long long Sx[4], Sy[4], Ox[4], Oy[4];
  const auto tables = [&](int a) {
    Sx[a] = even(c20, c40, a);
    Sy[a] = even(c02, c04, a);
    Ox[a] = odd(c10, c30, a);
    Oy[a] = odd(c01, c03, a);
  };
  const auto axes = [&](int a) {
    pairs(pop_index(a, 0), pop_index(0, a), shell_of_v2(a * a), S0 + Sx[a], Ox[a], S0 + Sy[a], Oy[a]);
  };
  const auto quad = [&](int a, int b, long long ds, long long D, long long dx, long long dy) {
    const long long S = S0 + Sx[a] + Sy[b] + ds, ox = Ox[a] + dx, oy = Oy[b] + dy;
    pairs(pop_index(a, b), pop_index(a, -b), shell_of_v2(a * a + b * b), S + D, ox + oy, S - D, ox - oy);
  };
  tables(1);
  axes(1);
  quad(1, 1, c22 >> 6, (c11 + ((c31 + c13) >> 1)) >> 4, c12 >> 5, c21 >> 5);
  tables(2);
  axes(2);
  quad(2, 1, c22 >> 4, (c11 + c31 * 2 + (c13 >> 1)) >> 3, c12 >> 4, c21 >> 3);
  quad(1, 2, c22 >> 4, (c11 + c13 * 2 + (c31 >> 1)) >> 3, c12 >> 3, c21 >> 4);
  quad(2, 2, c22 >> 2, (c11 + (c31 + c13) * 2) >> 2, c12 >> 2, c21 >> 2);
  tables(3);
  axes(3);
  const long long s9 = (c22 + (c22 >> 3)) >> 3;
  const auto d9 = [&](long long c9, long long c1) {  // 3 (c11 + 9 c9 + c1)
    const long long d = c11 + c9 * 4 + ((c9 + c1) >> 1);
    return (d >> 3) + (d >> 4);
  };
  const auto times3 = [](long long c) { return (c >> 4) + (c >> 5); };
  const auto times9 = [](long long c) { return (c >> 2) + (c >> 5); };
  quad(3, 1, s9, d9(c31, c13), times3(c12), times9(c21));
  quad(1, 3, s9, d9(c13, c31), times9(c12), times3(c21));
}

}  // namespace d2q37
