// Face flux of the FP64 path with its small terms in two-float arithmetic (ff_math.cuh).
#pragma once

#include "ff_math.cuh"
#include "flux_math.cuh"

namespace fl {

// Indicator terms of cell j from D = q_{j+1} - q_j and T = q_{j+1} - 2 q_j + q_{j-1}:
// 4 (beta + eps) of its three-cell stencil as the left (A), centre (B) and right (C) candidate, all times
// kIndScale^2 (set_ff has eps4 so), a common factor that the weights do not see.
FL_HD void cell_terms(ff D, ff T, ff eps4, ff& A, ff& B, ff& C) {
  const ff k133{4.33333349f, (float)(13.0 / 3.0 - (double)4.33333349f)};
  const ff Ts = ff_scale(T, kIndScale);
  const ff K = fma_weak(sqr_weak(Ts), k133, eps4);
  const ff T2 = ff_twice(Ts);
  const ff sB = add_weak(ff_scale(D, 2.0f * kIndScale), -Ts);
  const ff sA = add_weak(T2, sB), sC = add_weak(T2, -sB);
  A = fma_weak(sA, sA, K);
  B = fma_weak(sB, sB, K);
  C = fma_weak(sC, sC, K);
}

// 6 times the nonlinear parts of cell j's two face values from the indicator set e0 = A_{j-1},
// e1 = B_j, e2 = C_{j+1} and the third differences V0 = T_j - T_{j-1}, V1 = T_{j+1} - T_j:
// w^L_{j+1/2} = q_j + (2 D_j + D_{j-1} + dL) / 6, w^R_{j-1/2} = q_j - (2 D_{j-1} + D_j - dR) / 6.
// False when the indicators leave the FP32 range.
template <int SCHEME>
FL_HD bool cell_values(ff e0, ff e1, ff e2, ff V0, ff V1, ff& dL, ff& dR) {
  ff W0, W1, W2;
  const ff r0 = ff_rcp(e0), r1 = ff_rcp(e1), r2 = ff_rcp(e2);
  const float em = fminf(fminf(e0.h, e1.h), e2.h);
  if (SCHEME == FLUID_WENO_JS) {
    W0 = sqr_weak(mul_weak(r0, em));
    W1 = sqr_weak(mul_weak(r1, em));
    W2 = sqr_weak(mul_weak(r2, em));
  } else {
    const ff tau = e0 - e2;
    const ff Z0 = mul_weak(tau, r0), Z1 = mul_weak(tau, r1), Z2 = mul_weak(tau, r2);
    const ff one{1.0f, 0.0f};
    W0 = fma_weak(Z0, Z0, one);
    W1 = fma_weak(Z1, Z1, one);
    W2 = fma_weak(Z2, Z2, one);
    // tau above 2^30 of an indicator (next to exactly uniform cells): Z^2 drowns the 1 and may leave
    // the FP32 range, so the weights are taken relative to the smallest indicator, as for JS
    if (!(fmaxf(fmaxf(W0.h, W1.h), W2.h) < 1e18f)) {
      W0 = sqr_weak(mul_weak(r0, em));
      W1 = sqr_weak(mul_weak(r1, em));
      W2 = sqr_weak(mul_weak(r2, em));
    }
  }
  const ff P0 = mul_weak(W0, V0), P2 = mul_weak(W2, V1);
  const ff base = add_weak(add_weak(W0, W2), mul_weak(W1, 6.0f));
  const ff denL = add_weak(base, ff_twice(W2));
  const ff denR = add_weak(base, ff_twice(W0));
  const ff S2 = ff_twice(add_weak(P0, P2));           // numL = S2 + P2, numR = S2 + P0
  dL = mul_weak(-P2 - S2, ff_rcp(denL));
  dR = mul_weak(P0 + S2, ff_rcp(denR));
  return em < 1e30f;
}

// HLLC star correction of a face in ff, from the left state wl and the jumps J = wr - wl:
// X = S_K (U*_K - U_K) of the upwind side K, written in the jumps so that its error is relative to
// them (Batten et al., SIAM J. Sci. Comput. 18, 1997, for the speeds):
//   Roe averages u~ = u_L + a_R J_u, c~^2 = a_L c_L^2 + a_R c_R^2 + (gamma - 1)/2 a_L a_R |J_u|^2
//   S* - u_L = (J_p - m_R J_n) / (m_L - m_R), S* - u_R = S* - u_L - J_n, m_K = rho_K (S_K - u_K),
//   theta = (S* - u_K) / (S_K - S*).
// left: K = L.
template <int D>
FL_HD void hllc_ff(const ff wl[5], const ff J[5], const PhysFF& pf, bool& left, ff X[5]) {
  const ff rL = wl[0], pL = wl[4], uL = wl[1 + D];
  const ff rR = rL + J[0], pR = pL + J[4];
  const ff irL = ff_rcp(rL), irR = ff_rcp(rR);
  const ff pirL = pL * irL, pirR = pR * irR;
  const ff c2L = pirL * pf.gamma, c2R = pirR * pf.gamma;
  const ff cL = ff_sqrt(c2L), cR = ff_sqrt(c2R);
  // a_R = sqrt(rho_R) / (sqrt(rho_L) + sqrt(rho_R)) = 1 / (1 + sqrt(rho_L / rho_R))
  const ff aR = ff_rcp(ff_sqrt(rL * irR) + 1.0f);
  const ff aL = (-aR) + 1.0f;
  const ff q2J = ff_fma(J[1], J[1], ff_fma(J[2], J[2], ff_sqr(J[3])));
    const ff ct2 = ff_fma(aR, ff_fma(aL * ff_scale(pf.gm1, 0.5f), q2J, c2R - c2L), c2L);
  const ff ct = ff_sqrt(ct2);
  const ff Jn = J[1 + D];
  const ff ut = aR * Jn;                                 // u~ - u_L
  // S_L - u_L and S_R - u_R
  const ff a1 = ut - ct, b1 = (ut - Jn) + ct;
  const ff sl = ff_float(a1 + cL) < 0.0f ? a1 : -cL;
  const ff sr = ff_float(b1 + (-cR)) > 0.0f ? b1 : cR;
  const ff mL = rL * sl, mR = rR * sr;
  const ff sigL = ff_div(J[4] - mR * Jn, mL - mR);
  const ff Ss = uL + sigL;
  const ff SL = uL + sl;
  left = ff_float(SL) >= 0.0f || ff_float(Ss) >= 0.0f;
  const ff uK = left ? uL : uL + Jn;
  const ff SK = left ? SL : uK + sr;
  const bool star = left ? ff_float(SL) < 0.0f : ff_float(SK) > 0.0f;
  if (!star) {
    for (int v = 0; v < 5; ++v) X[v] = ff{0.0f, 0.0f};
    return;
  }
  const ff sK = left ? sl : sr;                          // S_K - u_K
  const ff sig = left ? sigL : sigL - Jn;                // S* - u_K
  const ff rK = left ? rL : rR, pK = left ? pL : pR;
  const ff v1 = left ? wl[1] : wl[1] + J[1], v2 = left ? wl[2] : wl[2] + J[2], v3 = left ? wl[3] : wl[3] + J[3];
  const ff theta = ff_div(sig, sK - sig);
  const ff q2 = ff_fma(v1, v1, ff_fma(v2, v2, ff_sqr(v3)));
  // rho theta, chi sigma (chi = 1 + theta) and the energy increment theta E + chi sigma (rho S* + p / (S_K - u_K))
  const ff rt = rK * theta;
  const ff cs = ff_fma(theta, sig, sig);
  const ff f0 = SK * rt;
  const ff E = ff_fma(pK, pf.igm1, ff_scale(rK, 0.5f) * q2);
  const ff e1 = ff_fma(rK, Ss, ff_div(pK, sK));
  X[0] = f0;
  X[1] = f0 * v1;
  X[2] = f0 * v2;
  X[3] = f0 * v3;
  // normal momentum: rho (theta u + chi sigma)
  X[1 + D] = X[1 + D] + SK * (rK * cs);
  X[4] = SK * ff_fma(theta, E, cs * e1);
}

// Reciprocal and square root in FP64 by one Newton step from the two-float result (47 bits): two FP64
// instructions, within an ulp.  x in the FP32 range, positive.
FL_HD double rcp_seeded(double x) {
  const ff q = ff_rcp(ff_of(x));
  const double r = ff_to_double(quick_sum(q.h, q.l));
  return fma(r, fma(-x, r, 1.0), r);
}
FL_HD double sqrt_seeded(double x) {
  const ff a = ff_of(x);
  const int h = s_bits(s_mul(0.5f, s_rsqrt(a.h)));
  const double s = ff_to_double(ff_sqrt(a));
  return fma(fma(-s, s, x), d_from((h >> 3) + ((1023 - 127) << 20), h << 29), s);
}

// States whose terms the seeds cover: rho and p in [2^-31, 2^33), |u| below 2^33
FL_HD bool seedable(const double w[5]) {
  constexpr int lo = 0x3e000000, hi = 0x42000000;
  return d_hi(w[0]) >= lo && d_hi(w[0]) < hi && d_hi(w[4]) >= lo && d_hi(w[4]) < hi && (d_hi(w[1]) & 0x7fffffff) < hi &&
         (d_hi(w[2]) & 0x7fffffff) < hi && (d_hi(w[3]) & 0x7fffffff) < hi;
}

// hllc of flux_math.cuh in about 80 FP64 instructions instead of 114, for seedable states: reciprocals and
// roots from two-float seeds, and the averaged sound speed from the jumps, c~^2 = a_L c_L^2 + a_R c_R^2 +
// (gamma - 1)/2 a_L a_R |J_u|^2 (hllc_ff), which needs neither the averaged enthalpy nor |u|^2 of both
// sides and does not cancel at high Mach numbers.  Its error against 80-bit arithmetic is that of hllc
// or less over Mach 0.1 to 20 and jumps of 2 to 60 %.  TENO6-A channel 192 x 128 x 128 with 5 % noise,
// where most faces take it: 20.1 -> 18.6 ms a step; shock tube of 200 cells 1.38 -> 1.34 ms.
template <int D>
FL_HD void hllc_seeded(const double wl[5], const double wr[5], const Phys& ph, double F[5]) {
  const double rL = wl[0], pL = wl[4], rR = wr[0], pR = wr[4];
  const double unL = wl[1 + D], unR = wr[1 + D];
  const double irL = rcp_seeded(rL), irR = rcp_seeded(rR);
  const double pirL = pL * irL, pirR = pR * irR;
  const double c2L = ph.gamma * pirL, c2R = ph.gamma * pirR;
  const double cL = sqrt_seeded(c2L), cR = sqrt_seeded(c2R);
  // sqrt(rho_R) / (sqrt(rho_L) + sqrt(rho_R))
  const double aR = rcp_seeded(1.0 + sqrt_seeded(rL * irR));
  const double aL = 1.0 - aR;
  const double J0 = wr[1] - wl[1], J1 = wr[2] - wl[2], J2 = wr[3] - wl[3];
  const double Jn = D == 0 ? J0 : (D == 1 ? J1 : J2);
  const double q2J = fma(J0, J0, fma(J1, J1, J2 * J2));
  const double ct = sqrt_seeded(fma(aR, fma(aL * (0.5 * ph.gm1), q2J, c2R - c2L), c2L));
  const double utn = fma(aR, Jn, unL);
  const double SL = fmin(unL - cL, utn - ct);
  const double SR = fmax(unR + cR, utn + ct);
  const double mL = rL * (SL - unL), mR = rR * (SR - unR);
  const double Ss = (pR - pL + unL * mL - unR * mR) * -rcp_seeded(mR - mL);

  const bool left = fl_nonneg(SL) || fl_nonneg(Ss);
  const bool star = left ? !fl_nonneg(SL) : fl_pos(SR);
  const double r = left ? rL : rR, p = left ? pL : pR, un = left ? unL : unR;
  const double S = left ? SL : SR, m = left ? mL : mR, pir = left ? pirL : pirR;
  const double u0 = left ? wl[1] : wr[1], u1 = left ? wl[2] : wr[2], u2 = left ? wl[3] : wr[3];
  const double H = fma(pir, ph.gamma * ph.igm1, 0.5 * (u0 * u0 + u1 * u1 + u2 * u2));
  const double mn = r * un;
  F[0] = mn;
  F[1] = mn * u0;
  F[2] = mn * u1;
  F[3] = mn * u2;
  F[1 + D] += p;
  F[4] = mn * H;
  if (star) {
    // U*_K = m/(S - S*) [1, S* (normal), tangential u, E/rho + (S* - un)(S* + p/m)]; S - S* has m's sign
    const double ds = S - Ss;
    const double q = left ? -rcp_seeded(-ds) : rcp_seeded(ds);
    const double fac = m * q;
    const double eir = H - pir;                       // E / rho
    const double dU0 = fac - r;
    double dU[3] = {dU0 * u0, dU0 * u1, dU0 * u2};
    dU[D] = fac * Ss - r * un;
    const double Es = fac * eir + (Ss - un) * (fac * Ss + p * q);
    F[0] += S * dU0;
    F[1] += S * dU[0];
    F[2] += S * dU[1];
    F[3] += S * dU[2];
    F[4] += S * (Es - r * eir);
  }
}

// FP64 Euler flux of the state w along D
template <int D>
FL_HD void euler_flux(const double w[5], const Phys& ph, double F[5]) {
  const double mn = w[0] * w[1 + D];
  const double q2 = fma(w[1], w[1], fma(w[2], w[2], w[3] * w[3]));
  F[0] = mn;
  F[1] = D == 0 ? fma(mn, w[1], w[4]) : mn * w[1];
  F[2] = D == 1 ? fma(mn, w[2], w[4]) : mn * w[2];
  F[3] = D == 2 ? fma(mn, w[3], w[4]) : mn * w[3];
  F[4] = fma(w[1 + D], (ph.gamma * ph.igm1) * w[4], (0.5 * mn) * q2);
}

// x^n for 1 <= n <= 16 by binary powering
FL_HD ff ff_ipow(ff x, int n) {
  ff r = x, b = x;
  bool have = false;
  while (true) {
    if (n & 1) {
      r = have ? r * b : b;
      have = true;
    }
    n >>= 1;
    if (!n) break;
    b = ff_sqr(b);
  }
  return r;
}

// mu(T) in ff; false where the law or the range needs FP64 (a power law whose exponent is no ratio
// of small integers, T / T_ref outside [2^-6, 2^6]).  The power law takes fl_pow_rational's Halley
// step from an FP32 estimate.
FL_HD bool viscosity_ff(ff T, const Phys& ph, ff& mu) {
  const PhysFF& pf = ph.k;
  mu = pf.mu_ref;
  if (ph.visc == FLUID_VISC_CONSTANT) return true;
  const ff r = T * pf.iT_ref;
  if (!(r.h >= 0.015625f && r.h <= 64.0f)) return false;
  if (ph.visc == FLUID_VISC_POWER) {
    if (ph.visc_q == 0) return false;
#ifdef __CUDA_ARCH__
    float l, y0;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l) : "f"(r.h));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y0) : "f"(ph.visc_e32 * l));
#else
    const float y0 = powf(r.h, ph.visc_e32);
#endif
    const ff a = ff_ipow(r, ph.visc_p), yq = ff_ipow(ff{y0, 0.0f}, ph.visc_q);
    const ff den = mul_weak(yq, 0.5f * (float)(ph.visc_q + 1)) + mul_weak(a, 0.5f * (float)(ph.visc_q - 1));
    const ff y = ff_div(a - yq, den) * ff{y0, 0.0f} + y0;
    mu = pf.mu_ref * y;
    return true;
  }
  mu = ff_div((r * ff_sqrt(r)) * pf.mu_TS, T + pf.suth_S);
  return true;
}

// Fourth-order dissipative flux of a face in ff (visc_face): value f_a + D/2 - (T_a + T_{a+1})/16 and
// derivative D - (T_{a+1} - T_a)/24 of the 4-cell stencils, with D = f_{a+1} - f_a and T the second
// differences of the two cells.  dn: derivatives of the velocities, vf their values, Tf and dT those of
// the temperature, mf = d(index)/dx; gd, gb: face values of d u_D / d x_b and d u_b / d x_b.
// Fd = (tau, energy).  False where the viscosity needs FP64.
template <int D>
FL_HD bool visc_ff(const ff dn[3], const ff vf[3], ff Tf, ff dT, ff mf, const ff gd[3], const ff gb[3],
                   int ndim, const Phys& ph, ff Fd[4]) {
  ff mu;
  if (!viscosity_ff(Tf, ph, mu)) return false;
  const ff gD = dn[D] * mf;
  ff tr{0.0f, 0.0f};                                     // tangential part of the divergence
#pragma unroll
  for (int b = 0; b < 3; ++b)
    if (b != D && b < ndim) tr = tr + gb[b];
  // tau_DD = mu (4/3 gD - 2/3 tr)
  const ff k23{0.666666687f, (float)(2.0 / 3.0 - (double)0.666666687f)};
  Fd[D] = mu * (k23 * (ff_twice(gD) - tr));
#pragma unroll
  for (int b = 0; b < 3; ++b)
    if (b != D) Fd[b] = mu * (b < ndim ? ff_fma(dn[b], mf, gd[b]) : dn[b] * mf);
  Fd[3] = ff_fma(vf[0], Fd[0], ff_fma(vf[1], Fd[1], ff_fma(vf[2], Fd[2], (mu * ph.k.lam_fac) * (dT * mf))));
  return true;
}

// x as ff, NaN where x is not finite or |x| >= 2^127 (so that the non-finite check sees it)
FL_HD ff ff_checked(double x) {
  ff a = ff_of(x);
  if ((d_hi(x) & 0x7fffffff) - ((1023 - 127) << 20) > 0x0fefffff) a = ff{s_from(0x7fc00000), s_from(0x7fc00000)};
  return a;
}

// The mixed path's conservative -> primitive conversion (prim_from_cons) in ff
FL_HD void prim_ff(const double U[5], const Phys& ph, ff w[6]) {
  const ff r = ff_checked(U[0]), ir = ff_rcp(r);
  const ff m0 = ff_checked(U[1]), m1 = ff_checked(U[2]), m2 = ff_checked(U[3]);
  const ff u = m0 * ir, v = m1 * ir, x = m2 * ir;
  const ff ke2 = ff_fma(m0, u, ff_fma(m1, v, m2 * x));
  const ff p = ph.k.gm1 * (ff_checked(U[4]) - ff_scale(ke2, 0.5f));
  w[0] = quick_sum(r.h, r.l);
  w[1] = u;
  w[2] = v;
  w[3] = x;
  w[4] = p;
  w[5] = (p * ir) * ph.k.iR;
}

}  // namespace fl
