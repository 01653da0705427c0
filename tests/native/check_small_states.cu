// WENO5 face values in two floats (cell_terms, cell_values of face_ff.cuh), compiled for the host, where the
// cell differences are near the epsilon of the weights: windows of a base value (argument 1) and noise of an
// amplitude (argument 2), epsilon argument 3.  Prints per scheme the root-mean-square and the largest error of the FP64
// formula and of the two floats against the definition in long double.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "../../paper_2406_19494_gb300/csrc/face_ff.cuh"

using namespace fl;
typedef long double L;

template <int SCHEME>
static void run(double base, double amp, double eps) {
  Phys ph{};
  ph.gamma = 1.4; ph.eps = eps;
  set_ff(ph);
  std::mt19937_64 gen(5);
  std::uniform_real_distribution<double> un(-1.0, 1.0);
  L e64 = 0, eff = 0, m64 = 0, mff = 0;
  long n = 0;
  for (int it = 0; it < 20000; ++it) {
    double q[7], d[6], t[6];
    for (double& x : q) x = base + amp * un(gen);
    for (int i = 0; i < 6; ++i) d[i] = q[i + 1] - q[i];
    for (int i = 1; i < 6; ++i) t[i] = d[i] - d[i - 1];
    ff A, B, C, x, y, dL, dR;
    cell_terms(ff_of(d[2]), ff_of(t[2]), ph.k.eps4, A, x, y);
    cell_terms(ff_of(d[3]), ff_of(t[3]), ph.k.eps4, x, B, y);
    cell_terms(ff_of(d[4]), ff_of(t[4]), ph.k.eps4, x, y, C);
    const ff T0 = ff_of(t[3]);
    if (!cell_values<SCHEME>(A, B, C, T0 - ff_of(t[2]), ff_of(t[4]) - T0, dL, dR)) continue;
    const double l = fma(kSixth, fma(3.0, d[3], ff_to_double(dL - T0)), q[3]);
    const double l64 = weno5<SCHEME>(q[1], q[2], q[3], q[4], q[5], eps);
    const L a = q[1], b = q[2], m = q[3], f = q[4], e = q[5], k = 13.0L / 12;
    const L t0 = a - 2 * b + m, t1 = b - 2 * m + f, t2 = m - 2 * f + e;
    const L b0 = k * t0 * t0 + 0.25L * (a - 4 * b + 3 * m) * (a - 4 * b + 3 * m), b1 = k * t1 * t1 + 0.25L * (b - f) * (b - f);
    const L b2 = k * t2 * t2 + 0.25L * (3 * m - 4 * f + e) * (3 * m - 4 * f + e), tau = fabsl(b0 - b2);
    const auto w = [&](L beta) { const L r = (SCHEME == FLUID_WENO_JS ? 1 : tau) / (beta + eps); return SCHEME == FLUID_WENO_JS ? r * r : 1 + r * r; };
    const L w0 = 0.1L * w(b0), w1 = 0.6L * w(b1), w2 = 0.3L * w(b2);
    const L r = (w0 * (2 * a - 7 * b + 11 * m) + w1 * (-b + 5 * m + 2 * f) + w2 * (2 * m + 5 * f - e)) / (6 * (w0 + w1 + w2));
    e64 += (l64 - r) * (l64 - r);
    eff += (l - r) * (l - r);
    m64 = fmaxl(m64, fabsl(l64 - r));
    mff = fmaxl(mff, fabsl(l - r));
    ++n;
  }
  std::printf("%ld %.6Le %.6Le %.6Le %.6Le\n", n, sqrtl(e64 / n), sqrtl(eff / n), m64, mff);
}

int main(int argc, char** argv) {
  run<FLUID_WENO_Z>(atof(argv[1]), atof(argv[2]), atof(argv[3]));
  run<FLUID_WENO_JS>(atof(argv[1]), atof(argv[2]), atof(argv[3]));
  return 0;
}
