// Host build of the fixed-point adjoint of a site's collision (adjoint_fix64.cuh) for the CPU tests: reads
//   <tau> <gx> <gy> <37 populations> <37 values of lambda>   (all as hex bits)
// lines from stdin, and prints "0" (outside the path's range) or "1 <k> <K> <dL/dtau> <37 results>", the
// scale exponents of the populations and of lambda in decimal, the rest as hex bits.
#include <cstdio>
#include <cstring>

#include "../../paper_1703_04594_gb300/csrc/adjoint_fix64.cuh"

using namespace d2q37;

static const FixGroup kGroups[kFixGroups] = LBM_FIX_GROUPS;

struct Io {
  FxHalves* slots;
  const double* lam;
  double* r;
  int K;
  int at(int i) const { return i; }
  double mu(int i, int k) const { return lam[i + k * NPAIR]; }
  FxHalves fixed(int i, int k) const { return slots[i + k * NPAIR]; }
  void keep(int i, int k, FxHalves q) const { slots[i + k * NPAIR] = q; }
  FxHalves held(int i) const { return slots[i]; }
  void out(int i, long long v) const { r[i] = fx_lower_exponent(v, K); }
};

static bool read_double(double& v) {
  unsigned long long bits;
  if (std::scanf("%llx", &bits) != 1) return false;
  std::memcpy(&v, &bits, 8);
  return true;
}

static void print_double(double v) {
  unsigned long long bits;
  std::memcpy(&bits, &v, 8);
  std::printf(" %llx", bits);
}

int main() {
  double tau, gx, gy, f[Q], lam[Q], r[Q];
  PairFix pairs[NPAIR + 1];
  for (int j = 0; j <= NPAIR; ++j)
    pairs[j] = {rep_vx(j), rep_vy(j), rep_vx(j) * rep_vx(j) + rep_vy(j) * rep_vy(j), shell(j)};
  while (read_double(tau) && read_double(gx) && read_double(gy)) {
    for (int i = 0; i < 2 * Q; ++i)
      if (!read_double(i < Q ? f[i] : lam[i - Q])) return 2;
    FxHalves slots[Q] = {};
    const FixConsts k = make_fix_consts(tau, gx, gy);
    const AdjFixConsts ka = make_adj_fix_consts(tau, gx, gy);
    const FixMoments m =
        fix_moments_rolled(kGroups, [&](int i) { return f[i]; }, [&](int i, FxHalves h) { slots[i] = h; });
    const FixScalars v = fix_scalars(m, k);
    unsigned top = 0;
    for (int i = 0; i < Q; ++i) {
      const unsigned h = fx_hi_word(lam[i]) & 0x7fffffffu;
      top = h > top ? h : top;
    }
    const unsigned E = top >> 20;
    if (!k.usable || !ka.usable || !v.ok || E - 100u >= 978u) {
      std::printf("0\n");
      continue;
    }
    const int K = (1080 - (int)E) << 20;
    const Io io = {slots, lam, r, K};
    const FixMu mm = fix_mu_moments(K + (1 << 20), kGroups, io);
    const FixVjp g = fix_vjp(m, v, mm, k, ka);
    fix_adj_outputs(g, ka.om1, pairs, io);
    std::printf("1 %d %d", m.kb / (1 << 20), K >> 20);
    const double om = 1.0 / tau;
    print_double(fix_dtau(g.D, om * om, K, m.kb));
    for (int i = 0; i < Q; ++i) print_double(r[i]);
    std::printf("\n");
  }
  return 0;
}
