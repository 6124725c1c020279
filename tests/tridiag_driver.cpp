// Eigenvalues of a symmetric tridiagonal matrix by the library's section code
// (csrc/tridiag.h), on the host.  Input per matrix: n P, the n diagonal and the
// n - 1 off-diagonal elements (one block, norm below 1); output: the n
// eigenvalues.
#include <cstdio>
#include <vector>

#include "tridiag.h"

int main() {
  int n, P;
  while (std::scanf("%d %d", &n, &P) == 2) {
    std::vector<double> d(n), e2(n, 1.0);
    for (double &x : d) if (std::scanf("%lf", &x) != 1) return 1;
    for (int j = 0; j + 1 < n; ++j) {
      double e;
      if (std::scanf("%lf", &e) != 1) return 1;
      e2[j] = fmax(e * e, etdm::kTriE2Min);
    }
    for (int i = 0; i < n; ++i) {
      double lo = -1.0 - 1e-15, hi = 1.0 + 1e-15;
      for (int it = 0; it < etdm::tri_rounds(P) && etdm::tri_open(lo, hi); ++it) {
        const double w = (hi - lo) * (1.0 / (P + 1)), l = lo;
        int m = 0;
        while (m < P && etdm::tri_count(d.data(), e2.data(), 0, n, etdm::tri_point(l, w, m + 1)) <= i) ++m;
        if (m > 0) lo = etdm::tri_point(l, w, m);
        if (m < P) hi = etdm::tri_point(l, w, m + 1);
      }
      std::printf("%.17g ", 0.5 * (lo + hi));
    }
    std::printf("\n");
    std::fflush(stdout);
  }
}
