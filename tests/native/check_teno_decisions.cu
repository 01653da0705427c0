// Host build of TENO6-A's FP32 decisions (keep_mask32_scaled) against the FP64 ones, on seeded windows of cell
// differences chosen to be hard for FP32: sizes down to 1e-20, sizes that differ by many decades within a
// window, a nearly uniform stencil beside a steep cell, smooth windows at the rounding level of FP64.
// Prints per family the shares of decisions left open and of clear decisions that differ.
#include <cmath>
#include <cstdio>
#include <random>

#include "../../paper_2406_19494_gb300/csrc/teno_math.cuh"

using namespace fl;
typedef long double L;

static std::mt19937_64 gen(5);
static double u() { return std::uniform_real_distribution<double>(-1.0, 1.0)(gen); }

static void window(int family, double d[5]) {
  const double s = std::pow(10.0, -20.0 * std::fabs(u())), J = u(), e = std::pow(10.0, -4.0 * std::fabs(u()));
  const double p = 3.0 * u(), k = 3.0 * std::fabs(u()), a = u(), b = u(), c = u();
  for (int i = 0; i < 5; ++i) {
    if (family == 0) d[i] = s * u();
    if (family == 1) d[i] = std::pow(10.0, -10.0 - 12.0 * std::fabs(u())) * u();
    if (family == 2) d[i] = J * std::pow(10.0, -6.0 * std::fabs(u())) * u();
    if (family == 3) d[i] = i < 2 ? e * J * u() : J * (1.0 + 0.5 * u());
    if (family == 4) d[i] = i == 2 ? J : e * J * u();
    if (family == 5) d[i] = i >= 3 ? e * J * u() : J * u();
    if (family == 6) d[i] = s * (std::sin(k * i + p) + 1e-3 * u());
    if (family == 7) d[i] = a + b * i + c * i * i + e * e * u();
    if (family == 8) d[i] = i < (int)(2.5 * (1.0 + b)) ? 0.0 : J * u();   // exactly uniform next to a step
    if (family == 9) d[i] = std::pow(10.0, -30.0 - 30.0 * std::fabs(u())) * u();
  }
}

// the left state's mask of the window (of its mirror image for right) from the differences
static int mask64(const double w[5], bool right, double ct) {
  double d[5];
  for (int i = 0; i < 5; ++i) d[i] = right ? -w[4 - i] : w[i];
  const auto K = [](L t, L s) { return (double)(13.0L / 12 * t * t + s * s / 4); };
  const double b0 = K((L)d[2] - d[1], (L)d[2] + d[1]), b1 = K((L)d[3] - d[2], 3 * (L)d[2] - d[3]);
  const double b2 = K((L)d[1] - d[0], 3 * (L)d[1] - d[0]), b3 = teno::beta4_diff(d[2], d[3], d[4]);
  double b6, none;
  teno::beta6_pair_diff(d, b6, none);
  return teno::keep_mask(b0, b1, b2, teno::rcp6(b0), teno::rcp6(b1), teno::rcp6(b2), teno::rcp6(b3), b6, ct);
}

int main() {
  for (int family = 0; family < 10; ++family) {
    long n = 0, open_ = 0, wrong = 0;
    for (int it = 0; it < 400000; ++it) {
      double d[5], t[4];
      window(family, d);
      const double ct = teno::cutoff_of_level(it & 3);
      ff T[4];
      for (int i = 0; i < 4; ++i) {
        t[i] = d[i + 1] - d[i];
        T[i] = ff_of<teno::kMaskScale>(t[i]);
      }
      const float Vm = s_add(s_sub(T[1].h, T[0].h), s_sub(T[1].l, T[0].l)), V = s_add(s_sub(T[2].h, T[1].h), s_sub(T[2].l, T[1].l));
      const float Vp = s_add(s_sub(T[3].h, T[2].h), s_sub(T[3].l, T[2].l)), D = ff_of<teno::kMaskScale>(d[2]).h;
      bool kl, kr;
      const int l = teno::keep_mask32_scaled(D, T[1].h, T[2].h, T[0].h, Vm, V, Vp, (float)ct, kl);
      const int r = teno::keep_mask32_scaled(-D, T[2].h, T[1].h, T[3].h, -Vp, -V, -Vm, (float)ct, kr);
      n += 2;
      open_ += !kl + !kr;
      wrong += (kl && l != mask64(d, false, ct)) + (kr && r != mask64(d, true, ct));
    }
    std::printf("%d %.6e %.6e\n", family, (double)open_ / n, (double)wrong / n);
  }
  return 0;
}
