// Host build of the two-float terms of the FP64 face kernels (ff_math.cuh, face_ff.cuh) and of the FP32
// decisions of TENO6-A (teno_math.cuh), for a CPU check: seeded cell windows and face states through the two-float formulas and through the FP64
// ones (flux_math.cuh), both against the same formulas in long double.  Prints one line per case:
// name, root-mean-square errors of the FP64 and the two-float results (TENO: decisions that FP32 left
// open and decisions that differ, as shares of all).
#include <algorithm>
#include <cstdio>
#include <cstdlib>

#include "../../paper_2406_19494_gb300/csrc/face_ff.cuh"
#include "../../paper_2406_19494_gb300/csrc/teno_math.cuh"

using namespace fl;
typedef long double L;

static unsigned long long s = 88172645463325252ull;
static double u() {                                      // uniform in [-1, 1)
  s ^= s << 13; s ^= s >> 7; s ^= s << 17;
  return (double)(s >> 11) * (2.0 / 9007199254740992.0) - 1.0;
}

static L weno_ref(const L q[5], bool js, L eps) {
  const L a = q[0], b = q[1], m = q[2], d = q[3], e = q[4], k = 13.0L / 12;
  const L t0 = a - 2 * b + m, t1 = b - 2 * m + d, t2 = m - 2 * d + e;
  const L b0 = k * t0 * t0 + 0.25L * (a - 4 * b + 3 * m) * (a - 4 * b + 3 * m);
  const L b1 = k * t1 * t1 + 0.25L * (b - d) * (b - d);
  const L b2 = k * t2 * t2 + 0.25L * (3 * m - 4 * d + e) * (3 * m - 4 * d + e);
  L w0, w1, w2;
  if (js) {
    w0 = 0.1L / ((eps + b0) * (eps + b0)); w1 = 0.6L / ((eps + b1) * (eps + b1)); w2 = 0.3L / ((eps + b2) * (eps + b2));
  } else {
    const L t = fabsl(b0 - b2);
    w0 = 0.1L * (1 + (t / (b0 + eps)) * (t / (b0 + eps)));
    w1 = 0.6L * (1 + (t / (b1 + eps)) * (t / (b1 + eps)));
    w2 = 0.3L * (1 + (t / (b2 + eps)) * (t / (b2 + eps)));
  }
  return (w0 * (2 * a - 7 * b + 11 * m) + w1 * (-b + 5 * m + 2 * d) + w2 * (2 * m + 5 * d - e)) / (6 * (w0 + w1 + w2));
}

template <int SCHEME>
static void weno(double amp) {
  const bool js = SCHEME == FLUID_WENO_JS;
  const double eps = js ? 1e-6 : 1e-40;
  Phys ph{};
  ph.gamma = 1.4; ph.eps = eps;
  set_ff(ph);
  double e64 = 0, eff = 0;
  int n = 0;
  for (int it = 0; it < 20000; ++it) {
    double q[7];
    for (double& x : q) x = 1.0 + amp * u();
    L a[5], b[5];
    for (int i = 0; i < 5; ++i) { a[i] = q[i + 1]; b[i] = q[5 - i]; }
    const L rl = weno_ref(a, js, eps), rr = weno_ref(b, js, eps);
    const double l64 = weno5<SCHEME>(q[1], q[2], q[3], q[4], q[5], eps);
    const double r64 = weno5<SCHEME>(q[5], q[4], q[3], q[2], q[1], eps);
    double d[6], t[6];
    for (int i = 0; i < 6; ++i) d[i] = q[i + 1] - q[i];
    for (int i = 1; i < 6; ++i) t[i] = d[i] - d[i - 1];
    ff A, B, C, x, y, dL, dR;
    cell_terms(ff_of(d[2]), ff_of(t[2]), ph.k.eps4, A, x, y);
    cell_terms(ff_of(d[3]), ff_of(t[3]), ph.k.eps4, x, B, y);
    cell_terms(ff_of(d[4]), ff_of(t[4]), ph.k.eps4, x, y, C);
    const ff T0 = ff_of(t[3]);
    if (!cell_values<SCHEME>(A, B, C, T0 - ff_of(t[2]), ff_of(t[4]) - T0, dL, dR)) continue;
    const double l = fma(kSixth, fma(3.0, d[3], ff_to_double(dL - T0)), q[3]);
    const double r = fma(kSixth, fma(-3.0, d[2], ff_to_double(dR - T0)), q[3]);
    e64 += (double)((l64 - rl) * (l64 - rl) + (r64 - rr) * (r64 - rr));
    eff += (double)((l - rl) * (l - rl) + (r - rr) * (r - rr));
    n += 2;
  }
  std::printf("weno_%s_%g %.6e %.6e\n", js ? "js" : "z", amp, std::sqrt(e64 / n), std::sqrt(eff / n));
}

template <int D>
static void hllc_ref(const L wl[5], const L wr[5], L g, L F[5]) {
  auto E = [&](const L* w) { return w[4] / (g - 1) + 0.5L * w[0] * (w[1] * w[1] + w[2] * w[2] + w[3] * w[3]); };
  const L EL = E(wl), ER = E(wr), sl = sqrtl(wl[0]), sr = sqrtl(wr[0]);
  L v[3];
  for (int c = 0; c < 3; ++c) v[c] = (sl * wl[1 + c] + sr * wr[1 + c]) / (sl + sr);
  const L H = (sl * (EL + wl[4]) / wl[0] + sr * (ER + wr[4]) / wr[0]) / (sl + sr);
  const L ct = sqrtl((g - 1) * (H - 0.5L * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2])));
  const L ul = wl[1 + D], ur = wr[1 + D];
  const L SL = fminl(ul - sqrtl(g * wl[4] / wl[0]), v[D] - ct), SR = fmaxl(ur + sqrtl(g * wr[4] / wr[0]), v[D] + ct);
  const L mL = wl[0] * (SL - ul), mR = wr[0] * (SR - ur);
  const L Ss = (wr[4] - wl[4] + ul * mL - ur * mR) / (mL - mR);
  const bool left = SL >= 0 || Ss >= 0;
  const L* w = left ? wl : wr;
  const L e = left ? EL : ER, S = left ? SL : SR, m = left ? mL : mR, mn = w[0] * w[1 + D];
  F[0] = mn;
  for (int c = 0; c < 3; ++c) F[1 + c] = mn * w[1 + c];
  F[1 + D] += w[4];
  F[4] = w[1 + D] * (e + w[4]);
  if (left ? SL < 0 : SR > 0) {
    const L fac = m / (S - Ss);
    L U[5] = {fac, fac * w[1], fac * w[2], fac * w[3], fac * (e / w[0] + (Ss - w[1 + D]) * (Ss + w[4] / m))};
    U[1 + D] = fac * Ss;
    const L V[5] = {w[0], w[0] * w[1], w[0] * w[2], w[0] * w[3], e};
    for (int k = 0; k < 5; ++k) F[k] += S * (U[k] - V[k]);
  }
}

template <int D>
static void riemann(double mach, double jump) {
  Phys ph{};
  ph.gamma = 1.4; ph.gm1 = 1.4 - 1.0; ph.igm1 = 1.0 / (1.4 - 1.0); ph.eps = 1e-40;
  set_ff(ph);
  double e64 = 0, eff = 0;
  const int n = 20000;
  for (int it = 0; it < n; ++it) {
    double wl[5] = {1.0 + 0.3 * u(), mach * u(), mach * u(), mach * u(), 1.0 / 1.4 + 0.2 * u()}, wr[5];
    L a[5], b[5], F[5];
    ff w[5], J[5], X[5];
    for (int v = 0; v < 5; ++v) {
      wr[v] = wl[v] + jump * u();
      a[v] = wl[v]; b[v] = wr[v];
      w[v] = ff_of(wl[v]);
      J[v] = ff_of(wr[v] - wl[v]);
    }
    hllc_ref<D>(a, b, 1.4, F);
    double f64[5], f[5];
    hllc<D>(wl, wr, ph, f64);
    bool left;
    hllc_ff<D>(w, J, ph.k, left, X);
    euler_flux<D>(left ? wl : wr, ph, f);
    for (int v = 0; v < 5; ++v) {
      f[v] += ff_to_double(X[v]);
      e64 += (double)((f64[v] - F[v]) * (f64[v] - F[v]));
      eff += (double)((f[v] - F[v]) * (f[v] - F[v]));
    }
  }
  std::printf("hllc%d_%g_%g %.6e %.6e\n", D, mach, jump, std::sqrt(e64 / n), std::sqrt(eff / n));
}

static void decisions(int kind) {
  long n = 0, open_ = 0, wrong = 0;
  for (int it = 0; it < 50000; ++it) {
    double q[6], amp = std::pow(10.0, -4.0 + 3.5 * std::fabs(u())), k = 0.05 + 0.5 * std::fabs(u()), p = 3.0 * u();
    const int cut = 1 + it % 5;
    for (int i = 0; i < 6; ++i) {
      if (kind == 0) q[i] = 1.0 + amp * std::sin(k * i + p);
      else if (kind == 1) q[i] = 1.0 + 0.05 * u();
      else if (kind == 2) q[i] = 1.0 + (i >= cut ? p / 3.0 : 0.0) + 0.1 * std::sin(k * i);
      else q[i] = 0.5 * u() * std::pow(10.0, -3.0 * std::fabs(u()));
    }
    double d[5], t[4];
    for (int i = 0; i < 5; ++i) d[i] = q[i + 1] - q[i];
    for (int i = 0; i < 4; ++i) t[i] = d[i + 1] - d[i];
    int level = 3;
    for (int j = 0; j < 4; ++j) {
      const int l = teno::sensor_level(d[j], d[j + 1]);
      bool clear;
      const int f = teno::sensor_level32(ff_of(d[j]).h, ff_of(d[j + 1]).h, clear);
      n += 1; open_ += !clear; wrong += clear && f != l;
      level = std::min(level, l);
    }
    const double ct = teno::cutoff_of_level(level);
    const double b[3] = {weno_B(q[1], q[2], q[3]), weno_C(q[2], q[3], q[4]), weno_A(q[0], q[1], q[2])};
    const double r[3] = {weno_B(q[4], q[3], q[2]), weno_C(q[3], q[2], q[1]), weno_A(q[5], q[4], q[3])};
    double b6l, b6r;
    teno::beta6_pair_diff(d, b6l, b6r);
    auto mask = [&](const double* e, double b4, double b6) {
      return teno::keep_mask(e[0], e[1], e[2], teno::rcp6(e[0]), teno::rcp6(e[1]), teno::rcp6(e[2]), teno::rcp6(b4), b6, ct);
    };
    ff T[4];
    for (int i = 0; i < 4; ++i) T[i] = ff_of(t[i]);
    const float Vm = (T[1].h - T[0].h) + (T[1].l - T[0].l), V = (T[2].h - T[1].h) + (T[2].l - T[1].l);
    const float Vp = (T[3].h - T[2].h) + (T[3].l - T[2].l), D = ff_of(d[2]).h;
    bool cl, cr;
    const int fl_ = teno::keep_mask32(D, T[1].h, T[2].h, T[0].h, Vm, V, Vp, (float)ct, cl);
    const int fr = teno::keep_mask32(-D, T[2].h, T[1].h, T[3].h, -Vp, -V, -Vm, (float)ct, cr);
    n += 2; open_ += !cl + !cr;
    wrong += (cl && fl_ != mask(b, teno::beta4_diff(d[2], d[3], d[4]), b6l)) +
             (cr && fr != mask(r, teno::beta4_diff(d[2], d[1], d[0]), b6r));
  }
  std::printf("teno%d %.6e %.6e\n", kind, (double)open_ / n, (double)wrong / n);
}

int main() {
  // conversions: |x - (h + l)| <= 2^-48 |x|, and back within 2^-52
  double w1 = 0, w2 = 0;
  for (int i = 0; i < 200000; ++i) {
    const double x = std::ldexp(u(), (int)(40 * u()));
    if (x == 0.0) continue;
    const ff a = ff_norm(ff_of(x));
    w1 = std::fmax(w1, std::fabs((double)((L)a.h + a.l - x)) / std::fabs(x));
    const ff b = i % 3 == 0 ? quick_sum(std::ldexp(i & 1 ? 1.0f : -1.0f, i % 50 - 25), std::ldexp((float)u(), i % 50 - 50)) : a;
    const double y = (double)((L)b.h + b.l);
    w2 = std::fmax(w2, std::fabs(ff_to_double(b) - y) / std::fabs(y));
  }
  std::printf("split %.6e %.6e\n", w1, w2);
  for (double amp : {1e-6, 1e-4, 1e-3}) { weno<FLUID_WENO_Z>(amp); weno<FLUID_WENO_JS>(amp); }
  for (double mach : {0.1, 1.0, 3.0})
    for (double jump : {1e-7, 1e-4, 4e-3}) { riemann<0>(mach, jump); riemann<1>(mach, jump); riemann<2>(mach, jump); }
  for (int kind = 0; kind < 4; ++kind) decisions(kind);
  return 0;
}
