// The rule that lets tensor generation tabulate a radial function (radial.h),
// over grids on both sides of it.  Each line of input: three n, three L, 'h'
// (mesh steps) or 'c' (box), as C99 hexadecimal floats; each line of output:
// "m r0 r1 r2 size" with m = s_min / base, or "no".
#include <cmath>
#include <cstdio>

#include "../paper_2504_19410_gb300/csrc/radial.h"

int main() {
  int n[3];
  double L[3];
  char kind;
  while (std::scanf("%d %d %d %la %la %la %c", n, n + 1, n + 2, L, L + 1, L + 2, &kind) == 7) {
    double s[3], num[3], den[3];
    for (int j = 0; j < 3; ++j) {
      s[j] = kind == 'h' ? 2.0 * L[j] / n[j] : 3.14159265358979323846 / (2 * L[j]);
      num[j] = kind == 'h' ? L[j] : 1.0;
      den[j] = kind == 'h' ? n[j] : L[j];
    }
    fsa::Radial r{};
    const long long total = (long long)(n[0] + 1) * (n[1] + 1) * (n[2] + 1);
    if (!fsa::radial_of(s, num, den, n, total, &r)) {
      std::puts("no");
      continue;
    }
    double lo = s[0];
    for (int j = 1; j < 3; ++j) lo = std::fmin(lo, s[j]);
    std::printf("%d %d %d %d %lld\n", (int)std::lround(lo / r.base), r.r[0], r.r[1], r.r[2], r.size);
  }
  return 0;
}
