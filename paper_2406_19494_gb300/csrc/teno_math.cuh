// TENO6-A reconstruction (the paper's channel scheme, Sec. 3.1), FP64.  The paper names the
// scheme and cites its solver for it; the definition used here is the published one (Fu, Hu &
// Adams 2016 for TENO6, 2017 for the adaptive cut-off):
//   left-biased value at i+1/2 from q_{i-2} .. q_{i+3}; candidate stencils S0 = (i-1, i, i+1),
//   S1 = (i, i+1, i+2), S2 = (i-2, i-1, i), S3 = (i, .., i+3) with the cell-average candidates
//   p_k and the sixth-order linear weights d = (9/20, 3/10, 1/20, 1/5); Jiang-Shu smoothness
//   measures beta_k and beta6 of the six-cell stencil, tau6 = |beta6 - (beta1 + beta2 + 4 beta0)/6|,
//   gamma_k = (1 + tau6 / (beta_k + 1e-40))^6; a stencil is kept unless gamma_k / sum gamma < C_T,
//   and the value is sum d_k p_k over the kept stencils divided by their sum of d_k.
//   Adaptive C_T = 10^-floor(10.5 - 3.5 (1 - g(m))), g = (1 - m)^4 (1 + 4 m),
//   m = 1 - min(1, eta / 0.25), eta the smallest scale sensor
//   (2 |D+ D-| + e) / (D+^2 + D-^2 + e) (D+- the differences to the two neighbours,
//   e = 0.9 * 0.25 * 1e-6 / 0.75) over the cells i-1 .. i+2.
// The right-biased value at i+1/2 is the left-biased value of the mirrored stencil; both use the
// same four cells for the sensor, so one cut-off serves both states of a face.
#pragma once

#include "ff_math.cuh"
#include "flux_math.cuh"
#include "teno_coeffs.cuh"

namespace fl {
namespace teno {

constexpr double kEps = 1e-40;
constexpr double kSensorE = 0.9 * 0.25 * 1e-6 / 0.75;

// 1/y for gamma_k, which only decides the cut-off: one second-order Newton step from the hardware
// estimate of rcp.approx.ftz.f64, relative error the square of the estimate's (about 2^-34 or
// smaller; the third-order fl_rcp squares it once more).  A keep decision can differ from exact
// division only where gamma_k / sum gamma is within about 1e-10 relative of C_T.
FL_HD double rcp_decide(double y) {
#ifdef __CUDA_ARCH__
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(y));
  return fma(r, fma(-y, r, 1.0), r);
#else
  return 1.0 / y;
#endif
}

// Cut-off level of a cell from the differences dm, dp to its two neighbours: how many of the
// thresholds kCutEta8 < kCutEta9 < kCutEta10 (teno_coeffs.cuh) its scale sensor
// eta = N / D = (2 |dp dm| + e) / (dp^2 + dm^2 + e) reaches, decided as N >= eta_k D (D > 0)
// without forming the quotient.  The adaptive C_T = 10^-floor(alpha1 - alpha2 (1 - g(m))) of a
// stencil (C_r = 0.25, alpha1 = 10.5, alpha2 = 3.5) is a step function of its smallest sensor,
// since g grows with eta, so it follows from the smallest level of the stencil's cells.
FL_HD int sensor_level(double dm, double dp) {
  const double N = fma(2.0, fabs(dp * dm), kSensorE);
  const double Dn = fma(dp, dp, fma(dm, dm, kSensorE));
  return (fma(-kCutEta8, Dn, N) >= 0.0 ? 1 : 0) + (fma(-kCutEta9, Dn, N) >= 0.0 ? 1 : 0) +
         (fma(-kCutEta10, Dn, N) >= 0.0 ? 1 : 0);
}

// C_T of a level: 1e-7, 1e-8, 1e-9, 1e-10
FL_HD double cutoff_of_level(int level) {
  return level >= 3 ? 1e-10 : (level == 2 ? 1e-9 : (level == 1 ? 1e-8 : 1e-7));
}

// linear weights d_k = (9/20, 3/10, 1/20, 1/5) (sixth-order combination of the four candidates)
FL_HD double lin_weight(int k) { return k == 0 ? 0.45 : (k == 1 ? 0.3 : (k == 2 ? 0.05 : 0.2)); }

// Normalised weights of the kept stencils for each keep mask (bit k set: stencil k kept):
// omega[k][mask] = d_k / sum of the kept d_j, 0 for a cut stencil (mask 0 cannot occur: the
// largest gamma_k / sum gamma is at least 1/4), times the common factor of candidate k's
// coefficients (1/6 for the three-cell candidates, 1/12 for the four-cell one), which the
// candidates below leave out.  Entry i of the 64 is written by call i.
FL_HD void weight_entry(int i, double omega[4][16]) {
  const int k = i >> 4, mask = i & 15;
  double den = 0.0;
  for (int j = 0; j < 4; ++j)
    if ((mask >> j) & 1) den += lin_weight(j);
  omega[k][mask] = ((mask >> k) & 1) ? lin_weight(k) / (den * (k < 3 ? 6.0 : 12.0)) : 0.0;
}

// TENO6 value from the candidates p_k (times 6, the four-cell one times 12), the three-cell
// smoothness measures b_k and i_k = rcp6(b_k) of all four (b6 = 6 beta6): stencil k is kept
// unless gamma_k / sum gamma < C_T, and the value is the kept candidates' combination with the
// normalised weights of omega (weight_entry)
// 1 / (6 (beta + eps)), the factor of tau in gamma_k
FL_HD double rcp6(double beta) { return rcp_decide(fma(6.0, beta, 6.0 * kEps)); }

// Which stencils are kept (bit k), from the three-cell smoothness measures b_k, i_k = rcp6(b_k) of all
// four stencils, b6 = 6 beta6 (beta6_pair) and the cut-off: tau = 6 tau6 and
// gamma_k = (1 + tau / (6 (beta_k + eps)))^6
FL_HD int keep_mask(double b0, double b1, double b2, double i0, double i1, double i2, double i3, double b6,
                    double ct) {
  const double tau = fabs(b6 - fma(4.0, b0, b1 + b2));
  double g[4];
  const double ik[4] = {i0, i1, i2, i3};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double x = fma(tau, ik[k], 1.0);
    const double x2 = x * x;
    g[k] = x2 * x2 * x2;
  }
  const double thr = ct * ((g[0] + g[1]) + (g[2] + g[3]));
  return (g[0] < thr ? 0 : 1) | (g[1] < thr ? 0 : 2) | (g[2] < thr ? 0 : 4) | (g[3] < thr ? 0 : 8);
}

FL_HD double combine(double p0, double p1, double p2, double p3, double b0, double b1, double b2,
                     double i0, double i1, double i2, double i3, double b6, double ct,
                     const double (*omega)[16]) {
  const int mask = keep_mask(b0, b1, b2, i0, i1, i2, i3, b6, ct);
  return fma(omega[3][mask], p3, fma(omega[2][mask], p2, fma(omega[1][mask], p1, omega[0][mask] * p0)));
}

// Both states of the face a+1/2 from q[0..5] = q_{a-2} .. q_{a+3} and the window's consecutive
// differences d[0..4] (d_j = q[j+1] - q[j]; the march carries d[0..3] and forms d[4]) while
// marching along +D.
//   * the candidates are written as offsets from 6 q_a (6 q_{a+1} for the mirrored stencil), the
//     smoothness measures in the differences (beta4_diff, beta6_pair_diff);
//   * the left state's central and downwind candidates are the right state's downwind and central
//     ones (the same quadratics through cells a-1..a+1 and a..a+2, at the same point);
//   * the right state's three-cell measures (B of the stencil centred at a+1, A at a, C at a+2) are
//     the next face's left-state measures (B at a+1, C at a+2, A at a): b3c carries them as
//     (beta0, beta1, beta2) of that next left state, and kk the 13/12 t^2 parts of the stencils
//     centred at a and a+1.
// On entry b3c holds this face's left-state (beta0, beta1, beta2) and i3c their rcp6; on exit the
// next face's.
FL_HD void face_states(const double q[6], const double d[5], double ct, double b3c[3], double i3c[3],
                       double kk[2], const double (*omega)[16], double& wl, double& wr) {
  // candidates times 6 (three cells) and 12 (four cells); the factors are in omega
  const double q6 = 6.0 * q[2], r6 = 6.0 * q[3];
  const double pc = fma(2.0, d[2], d[1]) + q6;                  // cells a-1..a+1
  const double pd = fma(4.0, d[2], -d[3]) + q6;                 // cells a..a+2
  const double pu = fma(5.0, d[1], -2.0 * d[0]) + q6;
  const double p4 = fma(9.0, d[2], fma(-4.0, d[3], d[4])) + 2.0 * q6;
  // 6 beta6 of the window and of its mirror image together (the reversal negates the odd part)
  double b6l, b6r;
  beta6_pair_diff(d, b6l, b6r);
  wl = combine(pc, pd, pu, p4, b3c[0], b3c[1], b3c[2], i3c[0], i3c[1], i3c[2],
               rcp6(beta4_diff(d[2], d[3], d[4])), b6l, ct, omega);
  // right state: the mirrored stencil q'_j = q[5 - j]
  const double ru = fma(-5.0, d[3], 2.0 * d[4]) + r6;
  const double r4 = fma(-9.0, d[2], fma(4.0, d[1], -d[0])) + 2.0 * r6;
  // three-cell measures K + s^2 / 4 with K = 13/12 t^2 of the stencil: K of the stencils centred at
  // a and a+1 carry over from the previous face (kk), the one centred at a+2 is new
  const double t2 = d[4] - d[3];
  const double K2 = k1312 * t2 * t2;
  const double sB = d[2] + d[3], sC = fma(3.0, d[2], -d[1]), sA = fma(-3.0, d[3], d[4]);
  const double rb0 = fma(0.25 * sB, sB, kk[1]);             // B of (q2, q3, q4)
  const double rb1 = fma(0.25 * sC, sC, kk[0]);             // C of (q1, q2, q3)
  const double rb2 = fma(0.25 * sA, sA, K2);                // A of (q3, q4, q5)
  kk[0] = kk[1];
  kk[1] = K2;
  const double ib0 = rcp6(rb0), ib1 = rcp6(rb1), ib2 = rcp6(rb2);
  wr = combine(pd, pc, ru, r4, rb0, rb1, rb2, ib0, ib1, ib2, rcp6(beta4_diff(d[2], d[1], d[0])), b6r,
               ct, omega);
  // next face's left state: beta0 = B at a+1 (rb0), beta1 = C at a+2 (rb2's stencil), beta2 = A at
  // a (rb1's), with their reciprocal factors
  b3c[0] = rb0;
  b3c[1] = rb2;
  b3c[2] = rb1;
  i3c[0] = ib0;
  i3c[1] = ib2;
  i3c[2] = ib1;
}

// ------------------------------------------------------------------------------------------------
// The same decisions in FP32, with a bound of their error: the weights of a face are those of its two
// keep masks and its cut-off level, so an FP32 decision that its error bound cannot turn is the FP64
// decision.  The few that it could turn are taken in FP64.
// ------------------------------------------------------------------------------------------------
// sensor_level in FP32; clear: no threshold lies within the error (each of N and D is within 6 2^-24
// of itself, the differences within 2^-23)
FL_HD int sensor_level32(float dm, float dp, bool& clear) {
  const float e = (float)kSensorE;
  const float N = s_fma(2.0f, fabsf(s_mul(dp, dm)), e);
  const float Dn = s_fma(dp, dp, s_fma(dm, dm, e));
  const float t8 = s_fma((float)-kCutEta8, Dn, N), t9 = s_fma((float)-kCutEta9, Dn, N);
  const float t10 = s_fma((float)-kCutEta10, Dn, N);
  clear = fminf(fminf(fabsf(t8), fabsf(t9)), fabsf(t10)) > 4e-6f * (N + Dn);
  return (t8 >= 0.0f ? 1 : 0) + (t9 >= 0.0f ? 1 : 0) + (t10 >= 0.0f ? 1 : 0);
}

// The left state's keep mask in FP32 from the face's difference D = q_{a+1} - q_a, the second
// differences T0, T1 of cells a and a+1 and Tm of cell a-1, and the third differences
// Vm = T0 - Tm, V = T1 - T0, Vp = T_{a+2} - T1; the right state's is that of the mirrored window
// (-D, T1, T0, T_{a+2}, -Vp, -V, -Vm).  In these terms the measures are sums of few terms, without
// the cancellation of their plain forms:
//   beta0 = 13/12 T0^2 + (D - T0/2)^2, beta1 = 13/12 T1^2 + (D - T1/2)^2,
//   beta2 = 13/12 Tm^2 + (d + Tm/2)^2 with d = D - T0,
//   beta3 = D^2 - D T1 + 4/3 T1^2 + 2/3 D Vp - 5/2 T1 Vp + 547/240 Vp^2,
//   6 tau6 = 2/5 D (F1 - F0) + V (481/120 V - 3379/5040 F0 - 16823/5040 F1) - T0 (46/15 F0 + 1/5 F1)
//            + F0 (27211/2240 F0 - 12281/1008 F1) + 139633/20160 F1^2, F0 = V - Vm, F1 = Vp - V.
// clear: no rounding of this function can turn a decision.  The bounds, with u = 2^-24, vm the largest of
// |Vm|, |V|, |Vp|, and inputs within 2 u of themselves (D, T: cut to 24 bits) or of vm (V), summed over the
// operations as written:
//   tau      (21 |D| + 68 |T0| + 1470 vm) vm u, below E (168 u for each and 1680 for vm)
//   measures 17 u of beta0 and beta1 and 73 u of beta3 (positive definite forms, the sum of whose terms is
//            at most 7.8 times their value); beta2, whose d cancels next to a steeper cell,
//            15 u + 4 u (|D| + |T0|) / sqrt(beta2)
//   gamma    6.4 times the relative errors of tau and of its measure, and 50 u: below the margin's half
//            of 14 E / tau, and its 6e-5 (1000 u) and its beta2 term
// Where the third differences are below 1e-5 of |D| + |T0| + |T1|, their own rounding counts, but then
// no tau / beta exceeds 1e-3.  The window comes times 2^16, so that epsilon (times 2^32) and the squares
// beside it stay normal numbers; a quotient tau / beta beyond the FP32 range ends as a NaN, which is not
// clear.
constexpr int kMaskScale = 16;   // log2 of the window's factor
FL_HD int keep_mask32_scaled(float D, float T0, float T1, float Tm, float Vm, float V, float Vp, float ct, bool& clear) {
  const float k = 13.0f / 12.0f, eps6 = (float)(6.0 * kEps * (double)(1ull << 2 * kMaskScale));
  const float s0 = s_fma(-0.5f, T0, D), s1 = s_fma(-0.5f, T1, D), s2 = s_fma(0.5f, Tm, s_sub(D, T0));
  const float b0 = s_fma(k * T0, T0, s_mul(s0, s0)), b1 = s_fma(k * T1, T1, s_mul(s1, s1));
  const float b2 = s_fma(k * Tm, Tm, s_mul(s2, s2));
  const float b3 = s_fma(D, s_fma(2.0f / 3.0f, Vp, s_sub(D, T1)),
                         s_fma(T1, s_fma(4.0f / 3.0f, T1, -2.5f * Vp), (547.0f / 240.0f) * Vp * Vp));
  const float F0 = s_sub(V, Vm), F1 = s_sub(Vp, V);
  float t = s_mul(0.4f * D, s_sub(F1, F0));
  t = s_fma(V, s_fma(481.0f / 120.0f, V, s_fma(-3379.0f / 5040.0f, F0, (-16823.0f / 5040.0f) * F1)), t);
  t = s_fma(-T0, s_fma(46.0f / 15.0f, F0, 0.2f * F1), t);
  t = s_fma(F0, s_fma(27211.0f / 2240.0f, F0, (-12281.0f / 1008.0f) * F1), t);
  t = s_fma((139633.0f / 20160.0f) * F1, F1, t);
  const float tau = fabsf(t);
  const float vm = fmaxf(fmaxf(fabsf(Vm), fabsf(V)), fabsf(Vp));
  const float E = 1e-5f * vm * (fabsf(D) + fabsf(T0) + fabsf(T1) + 10.0f * vm);
  const float i0 = s_rcp(s_fma(6.0f, b0, eps6)), i1 = s_rcp(s_fma(6.0f, b1, eps6));
  const float i2 = s_rcp(s_fma(6.0f, b2, eps6)), i3 = s_rcp(s_fma(6.0f, b3, eps6));
  const float im = fmaxf(fmaxf(i0, i1), fmaxf(i2, i3));
  // no gamma ratio below (1 / 10)^6 / 4, above every cut-off: all kept
  clear = true;
  if ((tau + E) * im < 9.0f) return 15;
  const float margin = 14.0f * E * s_rcp(tau) + 6e-5f + 1.6e-6f * (fabsf(D) + fabsf(T0)) * s_rsqrt(b2 + eps6);
  const float ix = s_rcp(s_fma(tau, im, 1.0f));
  float g[4] = {s_fma(tau, i0, 1.0f) * ix, s_fma(tau, i1, 1.0f) * ix, s_fma(tau, i2, 1.0f) * ix, s_fma(tau, i3, 1.0f) * ix};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    g[j] = g[j] * g[j] * g[j];
    g[j] = g[j] * g[j];
  }
  const float thr = ct * ((g[0] + g[1]) + (g[2] + g[3]));
  int mask = 0;
  clear = margin < 0.25f;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    mask |= g[j] < thr ? 0 : 1 << j;
    clear = clear && fabsf(g[j] - thr) > margin * (g[j] + thr);
  }
  return mask;
}

// the same from the window as it is
FL_HD int keep_mask32(float D, float T0, float T1, float Tm, float Vm, float V, float Vp, float ct, bool& clear) {
  const float f = (float)(1 << kMaskScale);
  return keep_mask32_scaled(s_mul(D, f), s_mul(T0, f), s_mul(T1, f), s_mul(Tm, f), s_mul(Vm, f), s_mul(V, f), s_mul(Vp, f),
                            ct, clear);
}

// Six times the correction of a face value, w = q + (3 D + c) / 6, as factors of (T_{a-1}, T_a, T_{a+1},
// T_{a+2}) per keep mask: the candidates are 3 D - T_a, 3 D - T_{a+1}, 3 D - 3 T_a + 2 T_{a-1} and
// 3 D - 3/2 T_{a+1} + 1/2 T_{a+2}.  Entry i of the 64 is written by call i.
FL_HD void factor_entry(int i, double alpha[4][16]) {
  const int k = i >> 4, mask = i & 15;
  double w[4], den = 0.0;
  for (int j = 0; j < 4; ++j) {
    w[j] = ((mask >> j) & 1) ? lin_weight(j) : 0.0;
    den += w[j];
  }
  const double f = k == 0 ? 2.0 * w[2] : (k == 1 ? -(w[0] + 3.0 * w[2]) : (k == 2 ? -(w[1] + 1.5 * w[3]) : 0.5 * w[3]));
  alpha[k][mask] = mask ? f / den : 0.0;
}

}  // namespace teno
}  // namespace fl
