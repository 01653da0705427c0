// hllc_seeded (csrc/face_ff.cuh) compiled for the host against 80-bit arithmetic: prints, per case, the
// largest error of hllc_seeded and of hllc over 32 units of 2^-53 of the flux's terms.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "face_ff.cuh"
#include "fluid_internal.cuh"

using namespace fl;
using L = long double;

// F and the size of its terms: (|u_n| + c) (|U_L| + |U_R|) + p per component
template <int D>
void exact(const double* wl, const double* wr, const Phys& ph, L* F, L* size) {
  const L g = ph.gamma, gm1 = ph.gm1;
  L w[2][5], U[2][5], c[2], H[2], s[2];
  for (int v = 0; v < 5; ++v) {
    w[0][v] = wl[v];
    w[1][v] = wr[v];
  }
  for (int k = 0; k < 2; ++k) {
    const L r = w[k][0], q2 = w[k][1] * w[k][1] + w[k][2] * w[k][2] + w[k][3] * w[k][3];
    const L E = w[k][4] / gm1 + r * q2 / 2;
    c[k] = sqrtl(g * w[k][4] / r);
    H[k] = (E + w[k][4]) / r;
    s[k] = sqrtl(r);
    U[k][0] = r;
    for (int d = 1; d < 4; ++d) U[k][d] = r * w[k][d];
    U[k][4] = E;
  }
  const L a = s[0] / (s[0] + s[1]), b = s[1] / (s[0] + s[1]);
  L u[3], q2 = 0;
  for (int d = 0; d < 3; ++d) {
    u[d] = a * w[0][1 + d] + b * w[1][1 + d];
    q2 += u[d] * u[d];
  }
  const L ct = sqrtl(gm1 * (a * H[0] + b * H[1] - q2 / 2));
  const L SL = fminl(w[0][1 + D] - c[0], u[D] - ct), SR = fmaxl(w[1][1 + D] + c[1], u[D] + ct);
  const L mL = w[0][0] * (SL - w[0][1 + D]), mR = w[1][0] * (SR - w[1][1 + D]);
  const L Ss = (w[1][4] - w[0][4] + w[0][1 + D] * mL - w[1][1 + D] * mR) / (mL - mR);
  const int k = SL >= 0 || Ss >= 0 ? 0 : 1;
  const L S = k ? SR : SL, un = w[k][1 + D], r = w[k][0], p = w[k][4];
  const bool star = k ? SR > 0 : SL < 0;
  const L f = r * (S - un) / (S - Ss);
  for (int v = 0; v < 5; ++v) {
    L Us = v == 4 ? f * (U[k][4] / r + (Ss - un) * (Ss + p / (r * (S - un)))) : f * (v ? w[k][v] : 1);
    if (v == 1 + D) Us = f * Ss;
    F[v] = U[k][v] * un + (v == 1 + D ? p : 0) + (v == 4 ? p * un : 0) + (star ? S * (Us - U[k][v]) : 0);
    const L uu = fabsl(w[0][1 + D]) + fabsl(w[1][1 + D]) + c[0] + c[1];
    size[v] = uu * (fabsl(U[0][v]) + fabsl(U[1][v])) + (v ? w[0][4] + w[1][4] : 0) * (v == 4 ? uu : 1);
    if (v > 0 && v < 4) size[v] += uu * uu * (w[0][0] + w[1][0]);
    size[v] *= uu / fminl(c[0], c[1]);       // the condition of S - S*
  }
}

int main(int argc, char** argv) {
  const double mach = atof(argv[1]), jump = atof(argv[2]), scale = atof(argv[3]);
  std::mt19937_64 gen(7);
  std::uniform_real_distribution<double> un(-1, 1);
  Phys ph{};
  ph.gamma = 1.4;
  ph.gm1 = 1.4 - 1.0;
  ph.igm1 = 1.0 / ph.gm1;
  set_ff(ph);
  L worst[2] = {0, 0};
  int taken = 0;
  for (int it = 0; it < 100000; ++it) {
    double wl[5], wr[5], a[5], b[5];
    L F[5], size[5];
    wl[0] = scale * (1.0 + 0.3 * un(gen));
    wl[4] = scale * (0.71 + 0.2 * un(gen));
    for (int d = 1; d < 4; ++d) wl[d] = mach * un(gen);
    for (int v = 0; v < 5; ++v) wr[v] = wl[v] + jump * un(gen) * (v >= 1 && v <= 3 ? 1.0 : 0.7 * wl[v]);
    if (!seedable(wl) || !seedable(wr)) continue;
    ++taken;
    hllc_seeded<1>(wl, wr, ph, a);
    hllc<1>(wl, wr, ph, b);
    exact<1>(wl, wr, ph, F, size);
    for (int v = 0; v < 5; ++v) {
      worst[0] = fmaxl(worst[0], fabsl(a[v] - F[v]) / (size[v] * ldexpl(32, -53)));
      worst[1] = fmaxl(worst[1], fabsl(b[v] - F[v]) / (size[v] * ldexpl(32, -53)));
    }
  }
  printf("%d %.4Lf %.4Lf\n", taken, worst[0], worst[1]);
  return 0;
}
