// The scaling of face cotangents in adjoint_ff.cuh compiled for the host: reads five cotangents a line and
// prints whether the two-float form takes them, the scaled components times their scale again (exact in
// long double, printed in units of the largest), and the largest slot of a reverse HLLC flux formed with
// them.
#include <cmath>
#include <cstdio>

#include "../../paper_2406_19494_gb300/csrc/adjoint_ff.cuh"

using namespace fl;

int main() {
  Phys ph{};
  ph.gamma = 1.4; ph.gm1 = 1.4 - 1.0; ph.igm1 = 1.0 / ph.gm1; ph.eps = 1e-40;
  set_ff(ph);
  const double l[5] = {1.1, 0.3, -0.2, 0.1, 0.8}, r[5] = {1.0, 0.32, -0.1, 0.15, 0.83};
  ff wl[5], J[5];
  for (int v = 0; v < 5; ++v) {
    wl[v] = ff_of(l[v]);
    J[v] = ff_of(r[v] - l[v]);
  }
  double x[5];
  while (std::scanf("%la %la %la %la %la", x, x + 1, x + 2, x + 3, x + 4) == 5) {
    const int k = cot_exponent(x);
    std::printf("%d", (int)cot_in_range(k));
    ff g[5], gl[5], gr[5];
    for (int v = 0; v < 5; ++v) {
      g[v] = ff_of_shifted(x[v], k);
      std::printf(" %.17g", (double)g[v].h + (double)g[v].l);
    }
    hllc_vjp_ff<0>(wl, J, 0.0f, ph.k, g, gl, gr);
    double m = 0.0;
    for (int v = 0; v < 5; ++v)
      m = std::fmax(m, std::fmax(std::fabs(shifted(ff_to_double(ff_norm(gl[v])), k)), std::fabs(shifted(ff_to_double(ff_norm(gr[v])), k))));
    std::printf(" %d %.17g\n", k, m);
  }
  return 0;
}
