// Host build of the fixed-point site collision (site_fix64.cuh) for the CPU tests: reads
//   <tau> <gx> <gy> <37 populations>   (all as hex bits)
// lines from stdin, and prints "0" (outside the path's range) or "1 <k> <37 results as hex bits>",
// k being the site's scale exponent.
#include <cmath>
#include <cstdio>
#include <cstring>

#include "../../paper_1703_04594_gb300/csrc/site_fix64.cuh"

using namespace d2q37;

struct Io {
  const FxHalves* f;
  double* r;
  int scale;
  int at(int i) const { return i; }
  FxHalves fixed(int i, int k) const { return f[i + k * NPAIR]; }
  void put(int i, int k, long long v, int s) const { r[i + k * NPAIR] = std::ldexp((double)v, scale - 57 - shell_exp(s)); }
};

static bool read_double(double& v) {
  unsigned long long bits;
  if (std::scanf("%llx", &bits) != 1) return false;
  std::memcpy(&v, &bits, 8);
  return true;
}

int main() {
  double tau, gx, gy, f[Q], r[Q];
  while (read_double(tau) && read_double(gx) && read_double(gy)) {
    for (int i = 0; i < Q; ++i)
      if (!read_double(f[i])) return 2;
    FxHalves fixed[Q] = {};
    const FixConsts k = make_fix_consts(tau, gx, gy);
    const FixMoments m = fix_moments([&](int i) { return f[i]; }, [&](int i, FxHalves h) { fixed[i] = h; });
    const FixScalars v = fix_scalars(m, k);
    if (!k.usable || !v.ok) {
      std::printf("0\n");
      continue;
    }
    const int scale = m.kb / (1 << 20);
    fix_relax(v, k.om1, Io{fixed, r, scale});
    std::printf("1 %d", scale);
    for (int i = 0; i < Q; ++i) {
      unsigned long long bits;
      std::memcpy(&bits, &r[i], 8);
      std::printf(" %llx", bits);
    }
    std::printf("\n");
  }
  return 0;
}
