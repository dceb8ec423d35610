// Compile-time constants of the fixed-point collision (site_fix64.cuh, adjoint_fix64.cuh): the
// shells' scales, their weights as correctly rounded fixed-point numbers, and the table of opposite
// pairs.
#pragma once
#include "collide_fp64.cuh"
#include "fixed64.cuh"

namespace d2q37 {

__host__ __device__ constexpr int shell_exp(int s) {
  constexpr int t[8] = {2, 3, 4, 6, 7, 9, 11, 11};
  return t[s];
}

// Compile-time fixed-point constants from the model's float64 constants, computed exactly
// in integers: a positive double is m 2^x with an integer m < 2^53.
struct DoubleParts {
  unsigned long long m;
  int x;
};
__host__ __device__ constexpr DoubleParts double_parts(double v) {  // v > 0, finite
  int x = 0;
  while (v >= 9007199254740992.0) { v *= 0.5; ++x; }
  while (v < 4503599627370496.0) { v *= 2.0; --x; }
  return DoubleParts{(unsigned long long)v, x};
}
// round(a b 2^k / d) for positive doubles a, b and a positive integer d (half up); the
// exact product of the two 53-bit significands fits 106 bits.
__host__ __device__ constexpr unsigned long long fx_const(double a, double b, int k, unsigned d = 1) {
  const DoubleParts pa = double_parts(a), pb = double_parts(b);
  const unsigned __int128 p = (unsigned __int128)pa.m * pb.m;
  const int sh = pa.x + pb.x + k;
  const unsigned __int128 n = sh >= 0 ? (p << sh) : ((p + ((unsigned __int128)1 << (-sh - 1))) >> (-sh));
  return (unsigned long long)((n + d / 2) / d);
}
// Shell constants with w' = w_s 2^e_s (signed formats need values below 2^63):
//   cw = w' (Q0.63), cq = w' q_s (Q4.59), cq2 = w' q_s^2 (Q8.55, with q_s^2 rounded to
//   64 bits first), cw6 = w' / 6 (unsigned Q0.64).  The kernels read cw; the others are what the
//   host tests hold fx_const's roundings to.
__host__ __device__ constexpr long long shell_cw(int s) {
  return (long long)fx_const(w_shell(s), 1.0, shell_exp(s) + 63);
}
__host__ __device__ constexpr long long shell_cq(int s) {
  return (long long)fx_const(w_shell(s), q_shell(s), shell_exp(s) + 59);
}
__host__ __device__ constexpr long long shell_cq2(int s) {
  // round(w' q q 2^55): the 106-bit product w' q is rounded to 64 significant bits, then
  // multiplied by q exactly (117 bits)
  const DoubleParts pw = double_parts(w_shell(s)), pq = double_parts(q_shell(s));
  unsigned __int128 p = (unsigned __int128)pw.m * pq.m;
  int x = pw.x + pq.x;
  while (p >= ((unsigned __int128)1 << 64)) {
    p = (p + 1) >> 1;
    ++x;
  }
  const unsigned __int128 p3 = p * pq.m;
  const int sh = x + pq.x + shell_exp(s) + 55;  // negative for every shell
  return (long long)((p3 + ((unsigned __int128)1 << (-sh - 1))) >> (-sh));
}
__host__ __device__ constexpr unsigned long long shell_cw_div(int s, unsigned d) {
  return fx_const(w_shell(s), 1.0, shell_exp(s) + 64, d);
}

// The tables, evaluated by the compiler (constexpr locals must be constant expressions), so
// kernels only ever read literals.
__host__ __device__ constexpr long long kCw(int s) {
  constexpr long long t[8] = {shell_cw(0), shell_cw(1), shell_cw(2), shell_cw(3),
                              shell_cw(4), shell_cw(5), shell_cw(6), shell_cw(7)};
  return t[s];
}
__host__ __device__ constexpr long long kCq(int s) {
  constexpr long long t[8] = {0, shell_cq(1), shell_cq(2), shell_cq(3), shell_cq(4), shell_cq(5), shell_cq(6),
                              shell_cq(7)};
  return t[s];
}
__host__ __device__ constexpr long long kCq2(int s) {
  constexpr long long t[8] = {0,            shell_cq2(1), shell_cq2(2), shell_cq2(3),
                              shell_cq2(4), shell_cq2(5), shell_cq2(6), shell_cq2(7)};
  return t[s];
}
__host__ __device__ constexpr unsigned long long kCw6(int s) {
  constexpr unsigned long long t[8] = {shell_cw_div(0, 6), shell_cw_div(1, 6), shell_cw_div(2, 6),
                                       shell_cw_div(3, 6), shell_cw_div(4, 6), shell_cw_div(5, 6),
                                       shell_cw_div(6, 6), shell_cw_div(7, 6)};
  return t[s];
}

// round(2^64 / c^2), exact from the float64 c^2 = m 2^x
__host__ __device__ constexpr unsigned long long inv_c2_64() {
  const DoubleParts p = double_parts(C2);
  const unsigned __int128 num = (unsigned __int128)1 << (64 - p.x);
  return (unsigned long long)((num + p.m / 2) / p.m);
}
constexpr unsigned long long kInvC2 = inv_c2_64();

// Per-pair data of representatives 1..18 as a constant-memory table (one uniform load per
// pair; cheaper in issue slots than unpacking the values from immediates).
struct PairFix {
  int vx, vy, v2, sh;
};
#define LBM_PAIR_FIX(j) \
  { rep_vx(j), rep_vy(j), rep_vx(j) * rep_vx(j) + rep_vy(j) * rep_vy(j), shell(j) }
static __constant__ PairFix c_pair_fix[NPAIR + 1] = {
    LBM_PAIR_FIX(0),  LBM_PAIR_FIX(1),  LBM_PAIR_FIX(2),  LBM_PAIR_FIX(3),  LBM_PAIR_FIX(4),
    LBM_PAIR_FIX(5),  LBM_PAIR_FIX(6),  LBM_PAIR_FIX(7),  LBM_PAIR_FIX(8),  LBM_PAIR_FIX(9),
    LBM_PAIR_FIX(10), LBM_PAIR_FIX(11), LBM_PAIR_FIX(12), LBM_PAIR_FIX(13), LBM_PAIR_FIX(14),
    LBM_PAIR_FIX(15), LBM_PAIR_FIX(16), LBM_PAIR_FIX(17), LBM_PAIR_FIX(18)};
#undef LBM_PAIR_FIX

}  // namespace d2q37
