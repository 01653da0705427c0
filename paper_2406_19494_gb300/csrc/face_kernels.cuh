// FP64 face kernels with WENO5 reconstruction: F^c - F^d at every face of axis D and the flux
// difference into R.  Included by the translation units that instantiate them.
//
// What bounds them and how the work is split between the pipes.  The FP64 pipe takes a warp
// instruction every 16 cycles per SM, in which the four schedulers issue 64 others; with the whole
// face in FP64 (510 FP64-pipe instructions) that pipe is about 85 % busy and everything else
// idle.  Here only what carries the full size of the state is FP64: the cell differences and
// second differences, the face state m + c / 6 with m the mean of the two cells, its Euler flux,
// and the flux difference (about 50 instructions).  The small terms -- the nonlinear weights and
// their corrections c, the HLLC star correction, the dissipative flux -- are two-float numbers
// (ff_math.cuh, face_ff.cuh), whose error is relative to the term.  A face whose terms are not
// small against the state (kFF... below; or a value outside the FP32 range, or not finite) takes the FP64 formulas of
// flux_math.cuh instead (the whole convective flux, or only HLLC where just the jump is large),
// so its rounding is theirs.  The choice depends on the face's cells only,
// hence not on the launch shape.
#pragma once

#include <cuda_runtime.h>

#include "face_ff.cuh"
#include "fluid_internal.cuh"

namespace fl {

// limits of the ff path relative to the state: a cell's third differences (next to a discontinuity
// they are large even where the weights hide it), six times its corrections, a face's jump, and the
// dissipative flux
constexpr float kFFThird = 1.0f / 64, kFFCorr = 1.0f / 16, kFFJump = 1.0f / 64, kFFVisc = 1.0f / 32;
constexpr float kFFMin = 1.9e-6f, kFFMax = 1e12f;     // range of rho, p and c

struct Flux5 {
  double f[5];
};

// The two values of one primitive at a face in FP64 from its six cells (f: the primitive's cell a)
template <int SCHEME>
__device__ __forceinline__ void values_fp64(const double* __restrict__ f, int s, double eps4, double& wl, double& wr) {
  double q[6];
#pragma unroll
  for (int o = 0; o < 6; ++o) q[o] = ld(f + (o - 2) * s);
  const double d0 = q[1] - q[0], d1 = q[2] - q[1], d2 = q[3] - q[2], d3 = q[4] - q[3], d4 = q[5] - q[4];
  const double c = 4.0 * k1312;
  const double tm = d1 - d0, t0 = d2 - d1, t1 = d3 - d2, t2 = d4 - d3;
  const double km = fma(c * tm, tm, eps4), k0 = fma(c * t0, t0, eps4);
  const double k1 = fma(c * t1, t1, eps4), k2 = fma(c * t2, t2, eps4);
  const double aA = fma(3.0, d1, -d0), aB = d1 + d2, aC = fma(-3.0, d2, d3);
  const double bA = fma(3.0, d2, -d1), bB = d2 + d3, bC = fma(-3.0, d3, d4);
  double X[3];
  weno_x<SCHEME>(fma(aA, aA, km), fma(aB, aB, k0), fma(aC, aC, k1), X);
  wl = weno_x_value(q[2], d0, d1, d2, d3, X);
  weno_x<SCHEME>(fma(bC, bC, k2), fma(bB, bB, k1), fma(bA, bA, k0), X);
  wr = weno_x_value(q[3], -d4, -d3, -d2, -d1, X);
}

template <int D>
__device__ __noinline__ Flux5 hllc_unseeded(Flux5 wl, Flux5 wr, const Phys* __restrict__ php) {
  Flux5 F;
  hllc<D>(wl.f, wr.f, *php, F.f);
  return F;
}

// The convective flux in FP64 from the two face states.  Not inlined: every kernel has the same bits.
template <int D>
__device__ __noinline__ Flux5 hllc_fp64(Flux5 wl, Flux5 wr, const Phys* __restrict__ php) {
  if (!seedable(wl.f) || !seedable(wr.f)) return hllc_unseeded<D>(wl, wr, php);
  Flux5 F;
  hllc_seeded<D>(wl.f, wr.f, *php, F.f);
  return F;
}

// The convective flux of a face in FP64 from its six cells
template <int D, int SCHEME>
__device__ __noinline__ Flux5 face_flux_fp64(const double* __restrict__ W, int nc, int cell, int s,
                                             const Phys* __restrict__ php) {
  Flux5 wl, wr;
#pragma unroll
  for (int v = 0; v < 5; ++v) values_fp64<SCHEME>(W + v * nc + cell, s, 4.0 * php->eps, wl.f[v], wr.f[v]);
  return hllc_fp64<D>(wl, wr, php);
}

// The dissipative flux of a face in FP64 (negated: to be added)
template <int D, int NP>
__device__ __noinline__ Flux5 visc_flux_fp64(const double* __restrict__ W, const double* __restrict__ G,
                                             int cell, int s, int a, const Geo* __restrict__ gp,
                                             const Phys* __restrict__ php) {
  double q[5][6];
#pragma unroll
  for (int v = 1; v < 4; ++v)
#pragma unroll
    for (int o = 0; o < 6; ++o) q[v][o] = ld(W + v * gp->ncell + cell + (o - 2) * s);
  Flux5 F;
#pragma unroll
  for (int v = 0; v < 5; ++v) F.f[v] = 0.0;
  add_visc_face<D, NP>(W, G, cell, s, a, *gp, *php, q, F.f);
  return F;
}

// FP32 scales of a cell: rho, p and the sound speed, and whether they lie in the ff range
struct Scale {
  float r, p, c;
  bool ok;
};
__device__ __forceinline__ bool in_range(const Scale& s) {
  return s.r >= kFFMin && s.r <= kFFMax && s.p >= kFFMin && s.p <= kFFMax && s.c >= kFFMin && s.c <= kFFMax;
}
__device__ __forceinline__ Scale scale_of(double rho, double p, const Phys& ph) {
  Scale s;
  s.r = ff_of(rho).h;
  s.p = ff_of(p).h;
  const float c2 = s_mul(ph.k.gamma.h, s_mul(s.p, s_rcp(s.r)));
  s.c = s_mul(c2, s_rsqrt(c2));
  s.ok = in_range(s);
  return s;
}
__device__ __forceinline__ float scale_at(const Scale& s, int v) { return v == 0 ? s.r : (v == 4 ? s.p : s.c); }

constexpr float k24H = 0.0416666679f, k24L = (float)(1.0 / 24.0 - (double)0.0416666679f);
constexpr float kSixthH = 0.166666672f;
__device__ __forceinline__ ff sixth() { return ff{kSixthH, (float)(1.0 / 6.0 - (double)kSixthH)}; }

// face value of an FP64 array: (9 (f1 + f2) - (f0 + f3)) / 16, or with six cells
// (150 (f2 + f3) - 25 (f1 + f4) + 3 (f0 + f5)) / 256
template <int NP>
__device__ __forceinline__ ff interp_ff(const double* __restrict__ f, int s) {
  const ff f0 = ff_of(ld(f - s)), f1 = ff_of(ld(f)), f2 = ff_of(ld(f + s)), f3 = ff_of(ld(f + 2 * s));
  if (NP == 4) return ff_scale(mul_weak(add_weak(f1, f2), 9.0f) - add_weak(f0, f3), 0.0625f);
  const ff e = add_weak(ff_of(ld(f - 2 * s)), ff_of(ld(f + 3 * s)));
  return ff_scale(mul_weak(add_weak(f1, f2), 150.0f) + (mul_weak(e, 3.0f) - mul_weak(add_weak(f0, f3), 25.0f)), 1.0f / 256);
}

template <int D, int NP>
__device__ __forceinline__ void add_visc_fp64(const double* __restrict__ W, const double* __restrict__ G, int cell,
                                              int s, int a, const Geo& g, const Phys& ph, double F[5]) {
  const Flux5 e = visc_flux_fp64<D, NP>(W, G, cell, s, a, &g, &ph);
#pragma unroll
  for (int v = 1; v < 5; ++v) F[v] += e.f[v];
}

// Subtract the dissipative flux of the face: in ff from X where it is small against the state, else in
// FP64 from F.  dv, dt: the differences of the velocities and the temperature per cell, vf and Tf their
// face values.  sc: scales of cell a+1.
template <int D, int NP>
__device__ __forceinline__ void add_visc(const double* __restrict__ W, const double* __restrict__ G, int cell,
                                         int s, int a, const Geo& g, const Phys& ph, const Scale& sc,
                                         const ff dv[3], const ff vf[3], ff Tf, ff dt, ff X[5], double F[5]) {
  ff Fd[4], gd[3], gb[3];
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    if (b == D || b >= g.ndim) continue;
    gd[b] = interp_ff<NP>(G + (D * 3 + b) * g.ncell + cell, s);
    gb[b] = interp_ff<NP>(G + (b * 3 + b) * g.ncell + cell, s);
  }
  bool ok = sc.ok && visc_ff<D>(dv, vf, Tf, dt, ff_of(g.mf[D][a]), gd, gb, g.ndim, ph, Fd);
  const float lm = kFFVisc * sc.p;
  ok = ok && fabsf(Fd[0].h) <= lm && fabsf(Fd[1].h) <= lm && fabsf(Fd[2].h) <= lm && fabsf(Fd[3].h) <= lm * sc.c;
  if (ok) {
#pragma unroll
    for (int v = 0; v < 4; ++v) X[1 + v] = X[1 + v] - Fd[v];
  } else {
    add_visc_fp64<D, NP>(W, G, cell, s, a, g, ph, F);
  }
}

// The face flux F^c - F^d at a+1/2 from the terms of its two cells: d[v] = q_{a+1} - q_a, cL and cR
// six times the corrections of the left and right values (w_L = q_a + (3 d + cL) / 6,
// w_R = q_{a+1} + (cR - 3 d) / 6: one rounding of the state's size), and for the dissipative flux
// vv = V_a = T_{a+1} - T_a and tv = T_a + T_{a+1} of the velocities and dt, tt, tm of the temperature
// (D_a - V_a / 24, T_a + T_{a+1} + 8 D_a, and the value of cell a+1).  ok: the cells' own limits.  sc:
// scales of cell a+1.  DEFER: where the cells' limits fail, the convective flux is left to the caller
// (true is returned and F holds the dissipative part).
template <int D, int SCHEME, bool VISC, bool DEFER>
__device__ __forceinline__ bool face_of_terms(const double* __restrict__ W, const double* __restrict__ G,
                                              int cell, int s, int a, const Geo& g, const Phys& ph,
                                              bool ok, const Scale& sc, const double d[5], const ff cL[5],
                                              const ff cR[5], const ff vv[3], const ff tv[3], ff dt, ff tt,
                                              double tm, double F[5]) {
  ff X[5], wl[5], J[5], m3[3], dv[3];
  bool small = true;                                       // the jump's limit
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const float lim = scale_at(sc, v);
    J[v] = (cR[v] - cL[v]) * sixth();
    ok = ok && fabsf(cL[v].h) <= kFFCorr * lim && fabsf(cR[v].h) <= kFFCorr * lim;
    small = small && fabsf(J[v].h) <= kFFJump * lim;
    // the mean of the two cells
    const ff Dv = ff_of(d[v]);
    const ff m = ff_of(ld(W + v * g.ncell + cell)) + ff_scale(Dv, 0.5f);
    if (VISC && v >= 1 && v <= 3) {
      m3[v - 1] = m;
      dv[v - 1] = Dv - vv[v - 1] * ff{k24H, k24L};
    }
    wl[v] = ff_fma(cL[v], sixth(), m);
  }
  if (ok && small) {
    bool left;
    hllc_ff<D>(wl, J, ph.k, left, X);
    double w[5];
    const int o = left ? 0 : s;
    const double three = left ? 3.0 : -3.0;
#pragma unroll
    for (int v = 0; v < 5; ++v)
      w[v] = fma(kSixth, fma(three, d[v], ff_to_double(left ? cL[v] : cR[v])), ld(W + v * g.ncell + cell + o));
    euler_flux<D>(w, ph, F);
  } else {
    Flux5 e;
    if (DEFER && !ok) {
#pragma unroll
      for (int v = 0; v < 5; ++v) e.f[v] = 0.0;
    } else if (ok) {
      Flux5 l, r;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const double* f = W + v * g.ncell + cell;
        l.f[v] = fma(kSixth, fma(3.0, d[v], ff_to_double(cL[v])), ld(f));
        r.f[v] = fma(kSixth, fma(-3.0, d[v], ff_to_double(cR[v])), ld(f + s));
      }
      e = hllc_fp64<D>(l, r, &ph);
    } else {
      e = face_flux_fp64<D, SCHEME>(W, g.ncell, cell, s, &ph);
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      F[v] = e.f[v];
      X[v] = ff{0.0f, 0.0f};
    }
  }
  if (VISC) {
    ff vf[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) vf[c] = m3[c] - ff_scale(tv[c], 0.0625f);
    if (ph.visc_order == 4)
      add_visc<D, 4>(W, G, cell, s, a, g, ph, sc, dv, vf, ff_of(tm) - ff_scale(tt, 0.0625f), dt, X, F);
    else
      add_visc_fp64<D, 6>(W, G, cell, s, a, g, ph, F);
  }
#pragma unroll
  for (int v = 0; v < 5; ++v) F[v] = __dadd_rn(F[v], ff_to_double(X[v]));
  return DEFER && !ok;
}

// R_a (+)= -(F_{a+1/2} - F_{a-1/2}) / dx_a along D, the same operations in every kernel: the first axis
// writes R, the others add to it (a constant, as a run-time choice executes both)
template <int D>
__device__ __forceinline__ void update_r(double* dst, double F, double Fp, double id) {
  const double dF = __dsub_rn(F, Fp);
  *dst = D > 0 ? fma(-id, dF, *dst) : __dmul_rn(-id, dF);
}

// ------------------------------------------------------------------------------------------------
// y and z: one thread marches along a segment of a grid line, lanes along x (along x itself, with
// lanes along y, only where a caller sets a segment length)
// ------------------------------------------------------------------------------------------------
// Terms carried along the march when face a+1/2 (j = a + 1) is next, per primitive: dm = q_j - q_a and
// d0 = q_{j+1} - q_j, the second differences Tm, T0 of a and j, the indicator terms Am (A of a), A0 and
// B0 (of j) and the left value's correction cL of a; ok: cell a's limits.
struct March {
  double dm[5], d0[5];
  ff Tm[5], T0[5], Am[5], A0[5], B0[5], cL[5];
  ff Dm, D0;        // temperature: differences q_a - q_{a-1} and q_j - q_a
  bool ok;
};

// corrections of cell j's two values (cell_values) and its limits; sc: its scales
template <int SCHEME>
__device__ __forceinline__ bool cell_corr(ff e0, ff e1, ff e2, ff T0, ff V0, ff V1, float lim, ff& cL, ff& cR) {
  ff dL, dR;
  const bool ok = cell_values<SCHEME>(e0, e1, e2, V0, V1, dL, dR);
  cL = dL - T0;
  cR = dR - T0;
  return ok && fabsf(V0.h) <= kFFThird * lim && fabsf(V1.h) <= kFFThird * lim;
}

template <int D, int SCHEME, bool VISC>
__device__ __forceinline__ void march_start(const double* __restrict__ W, int nc, int cell, int s,
                                            const Phys& ph, March& M) {
  const Scale sc = scale_of(ld(W + cell), ld(W + 4 * nc + cell), ph);
  M.ok = sc.ok;
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const double* f = W + v * nc + cell;                   // cell a
    const double q0 = ld(f - 2 * s), q1 = ld(f - s), q2 = ld(f), q3 = ld(f + s), q4 = ld(f + 2 * s);
    const double d0 = q1 - q0, d1 = q2 - q1, d2 = q3 - q2, d3 = q4 - q3;
    const ff T1 = ff_of(d1 - d0), T2 = ff_of(d2 - d1), T3 = ff_of(d3 - d2);
    ff A1, A2, A3, B2, B3, C3, x, y, cR;
    cell_terms(ff_of(d1), T1, ph.k.eps4, A1, x, y);
    cell_terms(ff_of(d2), T2, ph.k.eps4, A2, B2, y);
    cell_terms(ff_of(d3), T3, ph.k.eps4, A3, B3, C3);
    const bool ok = cell_corr<SCHEME>(A1, B2, C3, T2, add_weak(T2, -T1), add_weak(T3, -T2), scale_at(sc, v), M.cL[v], cR);
    M.ok = M.ok && ok;
    M.dm[v] = d2;
    M.d0[v] = d3;
    M.Tm[v] = T2;
    M.T0[v] = T3;
    M.Am[v] = A2;
    M.A0[v] = A3;
    M.B0[v] = B3;
  }
  if (VISC) {
    const double* f = W + 5 * nc + cell;
    const double t0 = ld(f - s), t1 = ld(f), t2 = ld(f + s);
    M.Dm = ff_of(t1 - t0);
    M.D0 = ff_of(t2 - t1);
  }
}

// the flux at a+1/2 (`cell` is cell a), advancing the march by one cell
template <int D, int SCHEME, bool VISC>
__device__ __forceinline__ void march_face(const double* __restrict__ W, const double* __restrict__ G,
                                           int cell, int s, int a, const Geo& g, const Phys& ph, March& M,
                                           double F[5]) {
  const int nc = g.ncell;
  const Scale sc = scale_of(ld(W + cell + s), ld(W + 4 * nc + cell + s), ph);
  bool okj = sc.ok;
  double d[5];
  ff cLn[5], cR[5], vv[3], tv[3], dt{0.0f, 0.0f}, tt{0.0f, 0.0f};
  double tm = 0.0;
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const double* f = W + v * nc + cell;
    const double dp = ld(f + 3 * s) - ld(f + 2 * s);
    const ff Tp = ff_of(dp - M.d0[v]);
    ff Ap, Bp, Cp;
    cell_terms(ff_of(dp), Tp, ph.k.eps4, Ap, Bp, Cp);
    const ff V0 = add_weak(M.T0[v], -M.Tm[v]), V1 = add_weak(Tp, -M.T0[v]);
    const bool ok = cell_corr<SCHEME>(M.Am[v], M.B0[v], Cp, M.T0[v], V0, V1, scale_at(sc, v), cLn[v], cR[v]);
    okj = okj && ok;
    d[v] = M.dm[v];
    if (VISC && v >= 1 && v <= 3) {
      vv[v - 1] = V0;
      tv[v - 1] = M.Tm[v] + M.T0[v];
    }
    M.dm[v] = M.d0[v];
    M.d0[v] = dp;
    M.Tm[v] = M.T0[v];
    M.T0[v] = Tp;
    M.Am[v] = M.A0[v];
    M.A0[v] = Ap;
    M.B0[v] = Bp;
  }
  if (VISC) {
    const double* f = W + 5 * nc + cell;
    const double t1 = ld(f + s), t2 = ld(f + 2 * s);
    const ff Dp = ff_of(t2 - t1);
    const ff Ta = M.D0 - M.Dm, Tj = Dp - M.D0;
    dt = M.D0 - (Tj - Ta) * ff{k24H, k24L};
    // value: t_{a+1} - D/2 - (T_a + T_{a+1}) / 16, with 8 D folded into the sum
    tt = (Ta + Tj) + ff_scale(M.D0, 8.0f);
    tm = t1;
    M.Dm = M.D0;
    M.D0 = Dp;
  }
  face_of_terms<D, SCHEME, VISC, false>(W, G, cell, s, a, g, ph, M.ok && okj, sc, d, M.cL, cR, vv, tv, dt, tt, tm, F);
#pragma unroll
  for (int v = 0; v < 5; ++v) M.cL[v] = cLn[v];
  M.ok = okj;
}

// With a seam buffer FB (2 x 5 doubles per segment, [side][v][item]), a segment after the first
// starts its march at face a0+1/2 instead of a0-1/2: it leaves its first cell a0 to k_face_seam,
// with the flux at a0+1/2 in FB side 0, and its own last flux goes to FB side 1 of the next
// segment, which is the flux at that segment's a0-1/2.  Every face is then formed once; without FB
// each segment forms the face before its first cell as well.  Both give the same bits.
template <int D, int SCHEME, bool VISC>
__device__ __forceinline__ void k_face_body(const double* __restrict__ W, const double* __restrict__ G,
                                            double* __restrict__ R, double* __restrict__ FB, const Geo& g,
                                            const Phys& ph, int seg, uint3 bid, uint3 gdim) {
  constexpr int A1 = (D == 0) ? 1 : 0;
  constexpr int A2 = (D == 2) ? 1 : 2;
  const int n1 = g.n[A1], n2 = g.n[A2], nd = g.n[D];
  const int nseg = (nd + seg - 1) / seg;
  const long long lines = (long long)n1 * n2;
  const long long total = lines * nseg;
  const int s = D == 0 ? 1 : (D == 1 ? g.sy : g.sz);
  const int nc = g.ncell;
  for (long long t = bid.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gdim.x * blockDim.x) {
    const int i1 = (int)(t % n1);
    const long long r = t / n1;
    const int i2 = (int)(r % n2);
    const int sg = (int)(r / n2);
    int c[3];
    c[A1] = i1 + g.h[A1];
    c[A2] = i2 + g.h[A2];
    const int a0 = g.h[D] + sg * seg;
    const int a1 = min(a0 + seg, g.h[D] + nd);
    const bool seam = FB != nullptr && sg > 0;
    c[D] = seam ? a0 : a0 - 1;
    int cell = c[0] + c[1] * g.sy + c[2] * g.sz;
    March M;
    march_start<D, SCHEME, VISC>(W, nc, cell, s, ph, M);
    double Fp[5];
    cell -= s;
    const int first = seam ? a0 : a0 - 1;
    for (int a = first; a < a1; ++a) {
      cell += s;
      double F[5];
      march_face<D, SCHEME, VISC>(W, G, cell, s, a, g, ph, M, F);
      if (a > first) {
        const double id = g.idx[D][a];
#pragma unroll
        for (int v = 0; v < 5; ++v) update_r<D>(R + v * nc + cell, F[v], Fp[v], id);
      } else if (seam) {
#pragma unroll
        for (int v = 0; v < 5; ++v) FB[v * total + t] = F[v];
      }
#pragma unroll
      for (int v = 0; v < 5; ++v) Fp[v] = F[v];
    }
    if (FB != nullptr && sg + 1 < nseg) {
#pragma unroll
      for (int v = 0; v < 5; ++v) FB[(5 + v) * total + t + lines] = Fp[v];
    }
  }
}

// ------------------------------------------------------------------------------------------------
// Tiles: one thread per cell of TD consecutive padded cells along D (the lines laid end to end) by
// TX columns along x, the terms of neighbouring cells passing through shared memory.  The first
// three and the last two rows of a tile only serve their neighbours (8 x 32 was the fastest of
// 8 x 16, 8 x 32, 4 x 32 and 4 x 64 along y and z by up to 20 %).  The loops over the primitives stay
// rolled: the unrolled body is larger than the instruction cache holds.
// Issue of instructions binds (two thirds of the issue slots at 24 warps per SM; 16 warps took 5 % longer).
// TGV 128^3, one launch: x 0.40 ms, y and z 0.50 ms; the marching kernel with the whole face in FP64
// took 1.9 ms, the march below with the same arithmetic as the tiles 1.2 ms (255 registers, 6.6
// warps per SM: loads and instruction fetch are exposed).
// ------------------------------------------------------------------------------------------------
template <int D>
struct TileShape {
  static constexpr int TX = D == 0 ? 1 : 8, TD = D == 0 ? 128 : 32;
  static constexpr int threads = TX * TD, step = TD - 5;
  // 24 warps per SM (85 registers): on TGV 128^3 the y and z launches took 0.49 ms, 0.56 ms at 16
  // warps (116 registers); x 0.38 ms against 0.41 ms
  static constexpr int blocks = 24 * 32 / threads;
};

// Tiles of a quarter of the threads along y and z, for grids that leave SMs without a tile of the shape above
// (a tile's instructions pass through one SM).  Against that shape on the same grids: vortex of 32^2 to 80^2,
// ten steps, 4 to 5 % shorter (64^2: 1.03 -> 0.98 ms), 90^2 to 128^2 0 to 2 %; right-hand sides of boxes in
// FP64 throughout, 12^3 to 18^3 16 to 21 %, 20^3 to 26^3 7 to 12 %; TGV 12^3 to 20^3 4 to 8 %.  TGV 22^3 to
// 26^3 took 6 to 11 % longer, boundary layers of 64 x 64 to 140 x 100 1 to 4 %.  Along x, 32 threads took
// longer than 128 (shock tube 1.35 -> 1.59 ms: fewer threads share the FP64 faces).
struct SmallTile {
  static constexpr int TX = 2, TD = 32, threads = TX * TD, step = TD - 5, blocks = 24 * 32 / threads;
};

template <int N>
struct TileShared {
  double d[5][N];          // q_{j+1} - q_j
  ff T[5][N], A[5][N], B[5][N], C[5][N];
  ff Dt[N];
  Scale sc[N];
  double F[5][N];          // cR (as two floats), then the face flux
  int deferred[N], ndef;   // threads whose face takes the FP64 convective flux
};

// tiles along (x, D) that cover the interior cells
template <int D, class S = TileShape<D>>
__host__ __device__ __forceinline__ long long tile_rows(const Geo& g) {
  const long long lines = (long long)g.n[0] * g.n[1] * g.n[2] / g.n[D] / (D == 0 ? 1 : g.n[0]);
  return (lines * g.p[D] + S::step - 1) / S::step;
}
template <int D, class S = TileShape<D>>
__host__ __device__ __forceinline__ int tile_cols(const Geo& g) {
  return D == 0 ? 1 : (g.n[0] + S::TX - 1) / S::TX;
}

// this thread's cell: its padded index i along D and its cell; live: on a line of the grid, pair: the
// line has a cell after it
struct TileCell {
  int i, cell;
  bool live, pair;
};
template <int D, class S = TileShape<D>>
__device__ __forceinline__ TileCell tile_cell(const Geo& g, int col, long long tile) {
  constexpr int TX = S::TX;
  constexpr int A1 = D == 0 ? 1 : 0, A2 = D == 2 ? 1 : 2;
  const int t = threadIdx.x, P = g.p[D];
  const long long idx = tile * S::step + t / TX;
  const long long line = idx / P;
  TileCell r;
  r.i = (int)(idx - line * P);
  int c[3];
  if (D == 0) {
    r.live = line < (long long)g.n[1] * g.n[2];
    c[1] = g.h[1] + (r.live ? (int)(line % g.n[1]) : 0);
    c[2] = g.h[2] + (r.live ? (int)(line / g.n[1]) : 0);
  } else {
    const int x = col * TX + t % TX;
    r.live = line < g.n[A2] && x < g.n[0];
    c[A1] = g.h[0] + (r.live ? x : 0);
    c[A2] = g.h[A2] + (r.live ? (int)line : 0);
  }
  c[D] = r.live ? r.i : 0;
  r.cell = c[0] + c[1] * g.sy + c[2] * g.sz;
  r.pair = r.live && r.i + 1 < P;
  return r;
}

template <int D, int SCHEME, bool VISC, class S = TileShape<D>>
__device__ __forceinline__ void k_face_tile_body(const double* __restrict__ W, const double* __restrict__ G,
                                                 double* __restrict__ R, const Geo& g, const Phys& ph,
                                                 TileShared<S::threads>& sh,
                                                 int col, long long tile) {
  constexpr int TX = S::TX, TD = S::TD;
  const int t = threadIdx.x, row = t / TX, nc = g.ncell;
  const int s = D == 0 ? 1 : (D == 1 ? g.sy : g.sz);
  const TileCell tc = tile_cell<D, S>(g, col, tile);
  const bool live = tc.live, pair = tc.pair;
  const int i = tc.i, cell = tc.cell;
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    const double* f = W + v * nc + cell;
    sh.d[v][t] = pair ? ld(f + s) - ld(f) : 0.0;
  }
  ff Dt{0.0f, 0.0f};
  double tq = 0.0;
  if (VISC) {
    if (pair) {
      tq = ld(W + 5 * nc + cell + s);
      Dt = ff_of(tq - ld(W + 5 * nc + cell));
    }
    sh.Dt[t] = Dt;
  }
  Scale sc{1.0f, 1.0f, 1.0f, false};
  if (live) sc = scale_of(ld(W + cell), ld(W + 4 * nc + cell), ph);
  if (t == 0) sh.ndef = 0;
  __syncthreads();
#pragma unroll 1
  for (int v = 0; v < 5; ++v) {
    const double d0 = sh.d[v][t];
    const ff T0 = ff_of(d0 - (row > 0 ? sh.d[v][t - TX] : 0.0));
    ff A, B, Cc;
    cell_terms(ff_of(d0), T0, ph.k.eps4, A, B, Cc);
    sh.T[v][t] = T0;
    sh.A[v][t] = A;
    sh.B[v][t] = B;
    sh.C[v][t] = Cc;
  }
  __syncthreads();
  // cell j: its corrections; B then holds cL, F holds cR
  const bool inner = row >= 2 && row < TD - 1;
  bool ok = sc.ok;
  if (inner) {
#pragma unroll 1
    for (int v = 0; v < 5; ++v) {
      const ff T0 = sh.T[v][t];
      ff cL, cR;
      const bool k = cell_corr<SCHEME>(sh.A[v][t - TX], sh.B[v][t], sh.C[v][t + TX], T0, add_weak(T0, -sh.T[v][t - TX]),
                                       add_weak(sh.T[v][t + TX], -T0), scale_at(sc, v), cL, cR);
      ok = ok && k;
      sh.B[v][t] = cL;
      sh.F[v][t] = __hiloint2double(s_bits(cR.l), s_bits(cR.h));
    }
  }
  sc.ok = ok;
  sh.sc[t] = sc;
  __syncthreads();
  // face j + 1/2
  const bool face = row >= 2 && row < TD - 2 && live && i >= g.h[D] - 1 && i < g.h[D] + g.n[D];
  double F[5];
  bool mine = false;
  if (face) {
    Scale sn = sh.sc[t + TX];
    double d[5];
    ff cL[5], cR[5], vv[3], tv[3], dt{0.0f, 0.0f}, tt{0.0f, 0.0f};
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const double r = sh.F[v][t + TX];
      d[v] = sh.d[v][t];
      cL[v] = sh.B[v][t];
      cR[v] = ff{s_from(d_lo(r)), s_from(d_hi(r))};
      if (VISC && v >= 1 && v <= 3) {
        const ff T0 = sh.T[v][t], T1 = sh.T[v][t + TX];
        vv[v - 1] = add_weak(T1, -T0);
        tv[v - 1] = T0 + T1;
      }
    }
    if (VISC) {
      const ff Ta = Dt - sh.Dt[t - TX], Tj = sh.Dt[t + TX] - Dt;
      dt = Dt - (Tj - Ta) * ff{k24H, k24L};
      tt = (Ta + Tj) + ff_scale(Dt, 8.0f);
    }
    const bool both = ok && sn.ok;
    // the dissipative flux only needs the scales in range
    sn.ok = in_range(sn);
    mine = face_of_terms<D, SCHEME, VISC, true>(W, G, cell, s, i, g, ph, both, sn, d, cL, cR, vv, tv, dt, tt, tq, F);
    if (mine) sh.deferred[atomicAdd(&sh.ndef, 1)] = t;
  }
  __syncthreads();
  // Faces beyond the limits: their FP64 formulas cost ten times a face's FP64 work, so the block's few
  // are gathered and spread over its threads, one primitive of one face each, then HLLC, one face
  // each.  (Left to their own lanes they held up every warp that had one: shock tube 26 us a launch.)
  const int ndef = sh.ndef;
  if (ndef > 0) {
    constexpr int N = S::threads;
    sh.sc[t].r = __int_as_float(cell);                     // the scales are done with
    __syncthreads();
    double* wl = &sh.d[0][0];                              // values of (primitive, face), left then right
    double* wr = reinterpret_cast<double*>(&sh.T[0][0]);
    static_assert(sizeof(sh.T) == sizeof(sh.d), "one double per pair");
    for (int k = t; k < 5 * ndef; k += N) {
      const int v = k / ndef, o = sh.deferred[k - v * ndef];
      values_fp64<SCHEME>(W + v * nc + __float_as_int(sh.sc[o].r), s, 4.0 * ph.eps, wl[v * N + o], wr[v * N + o]);
    }
    __syncthreads();
    for (int k = t; k < ndef; k += N) {
      const int o = sh.deferred[k];
      Flux5 l, r;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        l.f[v] = wl[v * N + o];
        r.f[v] = wr[v * N + o];
      }
      const Flux5 f = hllc_fp64<D>(l, r, &ph);
#pragma unroll
      for (int v = 0; v < 5; ++v) sh.F[v][o] = f.f[v];
    }
    __syncthreads();
    if (mine) {
#pragma unroll
      for (int v = 0; v < 5; ++v) F[v] = __dadd_rn(sh.F[v][t], F[v]);
    }
  }
  if (face) {
#pragma unroll
    for (int v = 0; v < 5; ++v) sh.F[v][t] = F[v];
  }
  __syncthreads();
  if (face && row >= 3 && i >= g.h[D]) {
    const double id = g.idx[D][i];
#pragma unroll
    for (int v = 0; v < 5; ++v) update_r<D>(R + v * nc + cell, F[v], sh.F[v][t - TX], id);
  }
}

}  // namespace fl
