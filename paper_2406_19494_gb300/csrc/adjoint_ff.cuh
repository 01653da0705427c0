// Adjoint of a face in two-float arithmetic (ff_math.cuh): the reconstruction's gradients, the reverse
// HLLC flux and the reverse dissipative flux of adjoint_math.cuh.  The FP64 forms take about 1,400
// FP64-pipe instructions per face.  Their terms are formed from cell differences, which are taken in FP64
// first, and a gradient inherits the rounding of the primitives relative to those differences, which on
// smooth fields is larger than the error of the two floats: over porous layers of 96 x 48 to 700 x 256 cells
// the step adjoint's error against 80-bit arithmetic is 3.5e-13 to 2.9e-12 of its norm with either, and the
// two differ by 0.6e-14 to 1.1e-14; at Mach 0.1 to 1e-5 both lose the same digits.  Where the weights are
// well conditioned (WENO5-JS, noise at the grid scale, jumps) the two floats show: 1e-15 to 7e-15 of the
// summed terms, 1e-17 to 1e-15 in FP64.  Cells and faces whose terms leave the FP32 range, and faces whose
// upwind side rounding may have decided, take the FP64 forms.
#pragma once

#include "adjoint_math.cuh"
#include "face_ff.cuh"

namespace fl {

FL_HD ff ff_const(double x) {
  const float h = (float)x;
  return ff{h, (float)(x - (double)h)};
}
// products and sums in the weak forms; a float factor is exact
FL_HD ff wm(ff a, ff b) { return mul_weak(a, b); }
FL_HD ff wm(float a, ff b) { return mul_weak(b, a); }
FL_HD ff wa(ff a, ff b) { return add_weak(a, b); }
FL_HD ff ws(ff a, ff b) { return add_weak(a, -b); }
// c + a b, c - a b
FL_HD ff wf(ff a, ff b, ff c) { return fma_weak(a, b, c); }
FL_HD ff wfn(ff a, ff b, ff c) { return fma_weak(-a, b, c); }

// weno5_side_vjp; csg = c times the sign of b0 - b2 (WENO5-Z: f and r carry c^2 and c)
template <int SCHEME>
FL_HD void weno5_side_ff(const ff f[3], const ff r[3], const ff iv[3], const ff rho[3], ff csg, ff d0, ff d1, ff d2,
                         const ff C[3], ff& out, ff gC[3], ff gb[3]) {
  const ff a0 = wm(d0, f[0]), a1 = wm(d1, f[1]), a2 = wm(d2, f[2]);
  const ff S = wa(wa(a0, a1), a2);
  const ff N = wf(a2, C[2], wf(a1, C[1], wm(a0, C[0])));
  const ff iS6 = ff_rcp(wm(6.0f, S));
  out = wm(N, iS6);
  const ff gS = wm(-6.0f, wm(out, iS6));
  const ff ga0 = wf(iS6, C[0], gS), ga1 = wf(iS6, C[1], gS), ga2 = wf(iS6, C[2], gS);
  gC[0] = wm(iS6, a0);
  gC[1] = wm(iS6, a1);
  gC[2] = wm(iS6, a2);
  if (SCHEME == FLUID_WENO_JS) {
    gb[0] = wm(-2.0f, wm(wm(ga0, a0), r[0]));
    gb[1] = wm(-2.0f, wm(wm(ga1, a1), r[1]));
    gb[2] = wm(-2.0f, wm(wm(ga2, a2), r[2]));
  } else {
    const ff gr0 = wm(wm(ga0, ff_twice(d0)), r[0]), gr1 = wm(wm(ga1, ff_twice(d1)), r[1]),
             gr2 = wm(wm(ga2, ff_twice(d2)), r[2]);
    const ff gtau = wm(csg, wf(gr2, iv[2], wf(gr1, iv[1], wm(gr0, iv[0]))));
    gb[0] = wfn(gr0, rho[0], gtau);
    gb[1] = -wm(gr1, rho[1]);
    gb[2] = wfn(gr2, rho[2], -gtau);
  }
}

// weno5_vjp_cell from the differences to the cell's value (q0 = q_{i-2} - q_i, ...) and re = 2 sqrt(epsilon): the offsets of the two
// values from it and their gradients.  The gradients do not change when the differences and epsilon's
// root are multiplied by one factor, so both are taken times the power of two that brings the largest
// difference (at least epsilon's root) near one.  False where the indicators leave the FP32 range.
template <int SCHEME>
FL_HD bool weno5_cell_ff(ff q0, ff q1, ff q3, ff q4, ff re, ff& up, ff Ju[5], ff& dn, ff Jd[5]) {
  const ff K4 = ff_const(4.0 * k1312), T = ff_const(8.0 * k1312);
  const float qm = fmaxf(fmaxf(fmaxf(fabsf(q0.h), fabsf(q1.h)), fmaxf(fabsf(q3.h), fabsf(q4.h))), re.h);
  const int ex = s_bits(qm) & 0x7f800000;
  const float sc = s_from(0x7f000000 - ex);
  bool ok = qm < 1e18f;
  q0 = ff_scale(q0, sc);
  q1 = ff_scale(q1, sc);
  q3 = ff_scale(q3, sc);
  q4 = ff_scale(q4, sc);
  const ff eps4 = sqr_weak(ff_scale(re, sc));
  const ff t0 = q0 - ff_twice(q1), s0 = q0 - ff_scale(q1, 4.0f);
  const ff t1 = q1 + q3, s1 = q1 - q3;
  const ff t2 = q4 - ff_twice(q3), s2 = q4 - ff_scale(q3, 4.0f);
  ff e[3] = {wa(wf(wm(K4, t0), t0, sqr_weak(s0)), eps4), wa(wf(wm(K4, t1), t1, sqr_weak(s1)), eps4),
             wa(wf(wm(K4, t2), t2, sqr_weak(s2)), eps4)};
  ff iv[3], r[3], f[3], rho[3];
  ff c{1.0f, 0.0f};
  float sg = 1.0f;
  if (SCHEME == FLUID_WENO_JS) {
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      iv[k] = r[k] = ff_rcp(e[k]);
      f[k] = sqr_weak(iv[k]);
      rho[k] = ff{0.0f, 0.0f};
      ok = ok && iv[k].h < 1e9f;
    }
  } else {
    const ff db = e[0] - e[2];
    sg = ff_float(db) < 0.0f ? -1.0f : 1.0f;
    const ff tau = ff_scale(db, sg), one{1.0f, 0.0f};
    // all (1 + r^2) times c^2, c = min(1, em / tau) with the smallest indicator em, so that none overflows
    const float em = fminf(fminf(e[0].h, e[1].h), e[2].h);
    ok = ok && em > 1e-35f;
    const ff ctau = tau.h < em ? tau : ff{em, 0.0f};
    c = tau.h < em ? one : wm(em, ff_rcp(tau));
    const ff c2 = sqr_weak(c);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      iv[k] = ff_rcp(e[k]);
      r[k] = wm(ctau, iv[k]);
      f[k] = wf(r[k], r[k], c2);
      rho[k] = wm(r[k], iv[k]);
    }
  }
  const ff csg = ff_scale(c, sg);
  const ff A0 = wf(T, t0, ff_twice(s0)), A1 = wf(T, t1, ff_twice(s1)), B1 = wf(T, t1, ff_scale(s1, -2.0f));
  const ff B0 = wf(ff_scale(T, -2.0f), t0, ff_scale(s0, -8.0f)), B2 = wf(ff_scale(T, -2.0f), t2, ff_scale(s2, -8.0f));
  const ff A2 = wf(T, t2, ff_twice(s2));
  const ff d1 = ff_const(0.1), d6 = ff_const(0.6), d3 = ff_const(0.3), one{1.0f, 0.0f};
  ff gC[3], gb[3];
  {
    const ff C[3] = {wa(ff_twice(q0), wm(-7.0f, q1)), ws(ff_twice(q3), q1), ws(wm(5.0f, q3), q4)};
    weno5_side_ff<SCHEME>(f, r, iv, rho, csg, d1, d6, d3, C, up, gC, gb);
    Ju[0] = wf(gb[0], A0, ff_twice(gC[0]));
    Ju[1] = wa(wm(-7.0f, gC[0]), ws(wf(gb[0], B0, wm(gb[1], A1)), gC[1]));
    Ju[3] = wa(ff_twice(gC[1]), wa(wm(5.0f, gC[2]), wf(gb[1], B1, wm(gb[2], B2))));
    Ju[4] = wf(gb[2], A2, -gC[2]);
    Ju[2] = ws(one, wa(wa(Ju[0], Ju[1]), wa(Ju[3], Ju[4])));
  }
  {
    const ff C[3] = {ws(wm(5.0f, q1), q0), ws(ff_twice(q1), q3), wa(ff_twice(q4), wm(-7.0f, q3))};
    weno5_side_ff<SCHEME>(f, r, iv, rho, csg, d3, d6, d1, C, dn, gC, gb);
    Jd[0] = wf(gb[0], A0, -gC[0]);
    Jd[1] = wa(wm(5.0f, gC[0]), wa(ff_twice(gC[1]), wf(gb[0], B0, wm(gb[1], A1))));
    Jd[3] = wa(wm(-7.0f, gC[2]), ws(wf(gb[1], B1, wm(gb[2], B2)), gC[1]));
    Jd[4] = wf(gb[2], A2, ff_twice(gC[2]));
    Jd[2] = ws(one, wa(wa(Jd[0], Jd[1]), wa(Jd[3], Jd[4])));
  }
  const float is = s_from(ex);
  up = ff_scale(up, is);
  dn = ff_scale(dn, is);
  return ok;
}

// hllc_vjp from the left state and the jumps J = wr - wl.  usig: the size below which rounding may have
// decided the sign of S*.  False where the states leave the range of the two floats, and where the upwind
// choice hangs on their rounding.
template <int D>
FL_HD bool hllc_vjp_ff(const ff wl[5], const ff J[5], float usig, const PhysFF& pf, const ff gF[5], ff gwl[5], ff gwr[5]) {
  const ff zero{0.0f, 0.0f};
  const ff wr[5] = {wl[0] + J[0], wl[1] + J[1], wl[2] + J[2], wl[3] + J[3], wl[4] + J[4]};
  const ff rL = wl[0], pL = wl[4], rR = wr[0], pR = wr[4];
  const ff unL = wl[1 + D], unR = wr[1 + D];
  const ff q2L = wf(wl[1], wl[1], wf(wl[2], wl[2], sqr_weak(wl[3])));
  const ff q2R = wf(wr[1], wr[1], wf(wr[2], wr[2], sqr_weak(wr[3])));
  const ff EL = wf(pL, pf.igm1, wm(ff_scale(rL, 0.5f), q2L));
  const ff ER = wf(pR, pf.igm1, wm(ff_scale(rR, 0.5f), q2R));
  const ff irL = ff_rcp(rL), irR = ff_rcp(rR);
  const ff sL = ff_sqrt(rL), sR = ff_sqrt(rR);
  const ff cL = ff_sqrt(wm(wm(pf.gamma, pL), irL)), cR = ff_sqrt(wm(wm(pf.gamma, pR), irR));
  const ff isum = ff_rcp(wa(sL, sR));
  const ff wL = wm(sL, isum), wR = wm(sR, isum);
  ff ut[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) ut[c] = wf(wL, wl[1 + c], wm(wR, wr[1 + c]));
  const ff HL = wm(wa(EL, pL), irL), HR = wm(wa(ER, pR), irR);
  const ff Ht = wf(wL, HL, wm(wR, HR));
  const ff q2t = wf(ut[0], ut[0], wf(ut[1], ut[1], sqr_weak(ut[2])));
  const ff ct = ff_sqrt(wm(pf.gm1, Ht - ff_scale(q2t, 0.5f)));
  const ff aL = unL - cL, bL = ut[D] - ct, aR = unR + cR, bR = ut[D] + ct;
  const bool selL = ff_float(ws(aL, bL)) <= 0.0f, selR = ff_float(ws(aR, bR)) >= 0.0f;
  const ff SL = selL ? aL : bL, SR = selR ? aR : bR;
  const ff dL = SL - unL, dR = SR - unR;
  const ff mL = wm(rL, dL), mR = wm(rR, dR);
  const ff iDd = ff_rcp(ws(mL, mR));
  const ff sig = wm(wfn(mR, J[1 + D], J[4]), iDd);      // S* - u_L
  const ff Ss = unL + sig;
  bool ok = fminf(fminf(rL.h, rR.h), fminf(pL.h, pR.h)) > 1e-9f && fmaxf(fmaxf(rL.h, rR.h), fmaxf(pL.h, pR.h)) < 1e12f &&
            fmaxf(q2L.h, q2R.h) < 1e24f;
  // at S* = 0 the two star fluxes agree, and their derivatives differ by rho*_K, the tangential velocities
  // and the energy that follows from them
  if (fabsf(ff_float(Ss)) < usig) {
    const ff xL = mL * SR, xR = mR * SL;
    const float ut = s_mul(ct.h, 2.3e-13f);
    ok = ok && fabsf(ff_float(xL - xR)) <= s_mul(fabsf(xL.h), 2.3e-13f) && (D == 0 || fabsf(J[1].h) <= ut) &&
         (D == 1 || fabsf(J[2].h) <= ut) && (D == 2 || fabsf(J[3].h) <= ut);
  }
  if (fminf(fabsf(ff_float(SL)), fabsf(ff_float(SR))) < s_mul(ct.h, 2.3e-13f))
    ok = ok && fabsf(J[0].h) <= s_mul(rL.h, 1e-13f) && fmaxf(fmaxf(fabsf(J[1].h), fabsf(J[2].h)), fabsf(J[3].h)) <= s_mul(ct.h, 1e-13f) &&
         fabsf(J[4].h) <= s_mul(pL.h, 1e-13f);
  const bool left = ff_float(SL) >= 0.0f || ff_float(Ss) >= 0.0f;
  const bool star = left ? ff_float(SL) < 0.0f : ff_float(SR) > 0.0f;
  const ff r = left ? rL : rR, p = left ? pL : pR, E = left ? EL : ER;
  const ff un = left ? unL : unR, S = left ? SL : SR, m = left ? mL : mR, ir = left ? irL : irR;
  const ff u[3] = {left ? wl[1] : wr[1], left ? wl[2] : wr[2], left ? wl[3] : wr[3]};
  const ff mn = wm(r, un);

  ff g_r = zero, g_p = gF[1 + D], g_E = wm(gF[4], un), g_u[3], g_S = zero, g_m = zero, g_ir = zero, g_Ss = zero;
  ff g_mn = gF[0];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    g_mn = wf(gF[1 + c], u[c], g_mn);
    g_u[c] = wm(gF[1 + c], mn);
  }
  g_u[D] = wf(gF[4], wa(E, p), g_u[D]);
  g_p = wa(g_p, g_E);
  if (star) {
    const ff q = ff_rcp(S - Ss);
    const ff fac = wm(m, q);
    const ff A = wm(E, ir), B = Ss - un, Cc = wf(fac, Ss, wm(p, q));
    const ff dU0 = fac - r;
    const ff dUn = wf(fac, Ss, -mn), dUe = wf(fac, A, wf(B, Cc, -E));
    ff g_fac = zero;
    g_S = wf(gF[0], dU0, wm(gF[4], dUe));
    const ff g0 = wm(gF[0], S);
    g_fac = g0;
    g_r = -g0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const ff gd = wm(gF[1 + c], S);
      if (c == D) {
        g_S = wf(gF[1 + c], dUn, g_S);
        g_fac = wf(gd, Ss, g_fac);
        g_Ss = wm(gd, fac);
        g_r = wfn(gd, un, g_r);
        g_u[D] = wfn(gd, r, g_u[D]);
      } else {
        g_S = wf(gF[1 + c], wm(dU0, u[c]), g_S);
        g_fac = wf(gd, u[c], g_fac);
        g_r = wfn(gd, u[c], g_r);
        g_u[c] = wf(gd, dU0, g_u[c]);
      }
    }
    const ff gEs = wm(gF[4], S);
    g_E = ws(g_E, gEs);
    g_fac = wf(gEs, A, g_fac);
    const ff gA = wm(gEs, fac), gB = wm(gEs, Cc), gCc = wm(gEs, B);
    g_fac = wf(gCc, Ss, g_fac);
    g_Ss = wa(wf(gCc, fac, g_Ss), gB);
    g_p = wf(gCc, q, g_p);
    g_u[D] = ws(g_u[D], gB);
    g_E = wf(gA, ir, g_E);
    g_ir = wm(gA, E);
    g_m = wm(g_fac, q);
    const ff g_q = wf(g_fac, m, wm(gCc, p));
    const ff g_d = wm(wm(g_q, q), q);                    // minus the cotangent of S - S*
    g_S = ws(g_S, g_d);
    g_Ss = wa(g_Ss, g_d);
  }
  g_r = wf(g_mn, un, g_r);
  g_u[D] = wf(g_mn, r, g_u[D]);

  const ff gNn = wm(g_Ss, iDd);
  ff gSL = left ? g_S : zero, gSR = left ? zero : g_S;
  ff gEL = left ? g_E : zero, gER = left ? zero : g_E;
  ff girL = left ? g_ir : zero, girR = left ? zero : g_ir;
  ff gmL = wfn(gNn, sig, left ? g_m : zero);
  ff gmR = wf(gNn, ws(sig, J[1 + D]), left ? zero : g_m);
  gwl[0] = left ? g_r : zero;
  gwr[0] = left ? zero : g_r;
  gwl[4] = ws(left ? g_p : zero, gNn);
  gwr[4] = wa(left ? zero : g_p, gNn);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    gwl[1 + c] = left ? g_u[c] : zero;
    gwr[1 + c] = left ? zero : g_u[c];
  }
  // m = rho (S - un)
  const ff gmrL = wm(gmL, rL), gmrR = wm(gmR, rR);
  gwl[1 + D] = ws(wf(gNn, mL, gwl[1 + D]), gmrL);
  gwr[1 + D] = ws(wfn(gNn, mR, gwr[1 + D]), gmrR);
  gwl[0] = wf(gmL, dL, gwl[0]);
  gwr[0] = wf(gmR, dR, gwr[0]);
  gSL = wa(gSL, gmrL);
  gSR = wa(gSR, gmrR);
  // Einfeldt bounds
  ff gutn = zero, gct = zero, gcL = zero, gcR = zero;
  if (selL) { gwl[1 + D] = wa(gwl[1 + D], gSL); gcL = -gSL; } else { gutn = gSL; gct = -gSL; }
  if (selR) { gwr[1 + D] = wa(gwr[1 + D], gSR); gcR = gSR; } else { gutn = wa(gutn, gSR); gct = wa(gct, gSR); }
  // ct = sqrt(gm1 (Ht - |ut|^2 / 2))
  const ff gHt = wm(pf.gm1, ff_scale(wm(gct, ff_rcp(ct)), 0.5f));
  const ff gHL = wm(gHt, wL), gHR = wm(gHt, wR);
  ff guL = wm(gHt, HL), guR = wm(gHt, HR), gdot = wm(gHt, Ht);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const ff gut = wfn(gHt, ut[c], c == D ? gutn : zero);
    guL = wf(gut, wl[1 + c], guL);
    guR = wf(gut, wr[1 + c], guR);
    gdot = wf(gut, ut[c], gdot);
    gwl[1 + c] = wf(gut, wL, gwl[1 + c]);
    gwr[1 + c] = wf(gut, wR, gwr[1 + c]);
  }
  // d / d s_K = isum (.. K - the average): the average's part of both is -gdot isum
  const ff gsL = wm(guL - gdot, isum), gsR = wm(guR - gdot, isum);
  // H = (E + p) ir
  const ff hL = wm(gHL, irL), hR = wm(gHR, irR);
  gEL = wa(gEL, hL);
  gER = wa(gER, hR);
  girL = wf(gHL, wa(EL, pL), girL);
  girR = wf(gHR, wa(ER, pR), girR);
  // c = sqrt(gamma p ir)
  const ff gYL = wm(pf.gamma, ff_scale(wm(gcL, ff_rcp(cL)), 0.5f)), gYR = wm(pf.gamma, ff_scale(wm(gcR, ff_rcp(cR)), 0.5f));
  gwl[4] = wa(gwl[4], wa(hL, wm(gYL, irL)));
  gwr[4] = wa(gwr[4], wa(hR, wm(gYR, irR)));
  girL = wf(gYL, pL, girL);
  girR = wf(gYR, pR, girR);
  // s = sqrt(rho): ds/drho = s / (2 rho); ir = 1 / rho; E = p / (gamma - 1) + rho |u|^2 / 2
  gwl[0] = wa(gwl[0], wm(irL, ws(ff_scale(wm(gsL, sL), 0.5f), wm(girL, irL))));
  gwr[0] = wa(gwr[0], wm(irR, ws(ff_scale(wm(gsR, sR), 0.5f), wm(girR, irR))));
  gwl[4] = wf(gEL, pf.igm1, gwl[4]);
  gwr[4] = wf(gER, pf.igm1, gwr[4]);
  gwl[0] = wf(gEL, ff_scale(q2L, 0.5f), gwl[0]);
  gwr[0] = wf(gER, ff_scale(q2R, 0.5f), gwr[0]);
  const ff eL = wm(gEL, rL), eR = wm(gER, rR);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    gwl[1 + c] = wf(eL, wl[1 + c], gwl[1 + c]);
    gwr[1 + c] = wf(eR, wr[1 + c], gwr[1 + c]);
  }
  return ok;
}

// visc_face_vjp: a[c], b[c] (c < 3 the velocities, 3 the temperature) are the cotangents of the face value
// and of the derivative per cell of the 4-cell stencils, which the cells receive times (-1, 9, 9, -1) / 16 and
// (1, -27, 27, -1) / 24.  vf, dn (without the metric mf), Tf, dT, gd and gb as in visc_ff.  False where the
// viscosity needs FP64.
template <int D>
FL_HD bool visc_vjp_ff(const ff dn[3], const ff vf[3], ff Tf, ff dTc, ff mf, const ff gd[3], const ff gb[3], int ndim,
                       const Phys& ph, const ff gFd[4], ff a[4], ff b[4], ff gGD[3], ff gGB[3]) {
  ff mu;
  if (!viscosity_ff(Tf, ph, mu)) return false;
  ff muT{0.0f, 0.0f};
  if (ph.visc == FLUID_VISC_POWER) muT = wm(wm(ph.k.visc_exp, mu), ff_rcp(Tf));
  else if (ph.visc == FLUID_VISC_SUTHERLAND)
    muT = wm(mu, wm(1.5f, ff_rcp(Tf)) - ff_rcp(Tf + ph.k.suth_S));
  const ff gD = wm(dn[D], mf), zero{0.0f, 0.0f};
  ff tr = zero;
#pragma unroll
  for (int c = 0; c < 3; ++c)
    if (c != D && c < ndim) tr = wa(tr, gb[c]);
  const ff k23 = ff_const(2.0 / 3.0);
  ff e[3];                                              // tau / mu
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (c == D) e[c] = wm(k23, ff_twice(gD) - tr);
    else e[c] = c < ndim ? wf(dn[c], mf, gd[c]) : wm(dn[c], mf);
  }
  const ff dT = wm(dTc, mf);
  ff gmu = wm(wm(gFd[3], dT), ph.k.lam_fac), gtD = zero;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const ff gt = wf(gFd[3], vf[c], gFd[c]);
    gmu = wf(gt, e[c], gmu);
    a[c] = wm(gFd[3], wm(mu, e[c]));
    const ff gm = wm(gt, mu);
    if (c == D) {
      gtD = wm(k23, gm);
      b[c] = wm(ff_twice(gtD), mf);
    } else {
      b[c] = wm(gm, mf);
      gGD[c] = c < ndim ? gm : zero;
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c)
    if (c != D) gGB[c] = c < ndim ? -gtD : zero;
  gGD[D] = gGB[D] = zero;
  a[3] = wm(gmu, muT);
  b[3] = wm(wm(wm(gFd[3], mu), ph.k.lam_fac), mf);
  return true;
}

// x 2^-k and x 2^k for face cotangents: the exponent moved by integer operations, k = cot_exponent of the
// face's five, 0 where all of them are zero.  A zero or subnormal x gives a zero pair: its exponent field is
// not the exponent of a leading one, and moved it would read as 2^(-k-1023) (for k = -1023 as 1).
FL_HD int cot_exponent(const double x[5]) {
  int e = 0, any = 0;
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const int t = d_hi(x[v]) & 0x7fffffff;
    e = t > e ? t : e;
    any |= t | d_lo(x[v]);
  }
  return any ? (e >> 20) - 1023 : 0;
}
// Cotangents that the scaling serves: above 2^-912 a subnormal component is below 2^-110 of the largest,
// and below 2^880 no two-float slot (under 2^128) passes the largest FP64 exponent on its way back
FL_HD bool cot_in_range(int k) { return k > -912 && k < 880; }
FL_HD ff ff_of_shifted(double x, int k) {
  const int hi = d_hi(x), e = (hi & 0x7ff00000) - (k << 20);
  return (hi & 0x7ff00000) && e > 0x39000000 ? ff_of(d_from(hi - (k << 20), d_lo(x))) : ff{0.0f, 0.0f};
}
FL_HD double shifted(double x, int k) {
  const int hi = d_hi(x), e = (hi & 0x7ff00000) + (k << 20);
  return (hi & 0x7ff00000) && e > 0 ? d_from(hi + (k << 20), d_lo(x)) : 0.0;
}

}  // namespace fl
