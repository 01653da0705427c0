// Mixed-precision face kernels: WENO5 weights and reconstruction, HLLC wave speeds and star
// correction, and the dissipative stencils in FP32; the state and the flux-difference accumulation
// in FP64; the primitives and the cell-centre convective flux as two-float numbers (ff_math.cuh,
// about 47 bits).
//
// Why a delta form.  At low Mach number the pressure (and total enthalpy) is large and nearly
// uniform, so fluxes are large and their differences across a cell small: a flux rounded to FP32
// carries an absolute error ~6e-8 |F| that the divergence divides by dx.  Here every FP32 quantity
// is either a coefficient (used only as a factor) or a small increment that FP32 represents to
// ~6e-8 of its own size:
//   * cell differences D_j = q_{j+1} - q_j of the primitives come from their pairs q = hi + lo:
//     (hi_{j+1} - hi_j) + (lo_{j+1} - lo_j), each FP32 subtraction rounding relative to its own
//     result, so D_j is within ~1 ulp (FP32) of the difference, up to 2^-47 |q| from the pairs;
//   * WENO5 works on D and the second differences T_j = D_j - D_{j-1}: the indicators of a cell serve
//     the values at both of its faces, w^L_{j+1/2} = q_j + (3 D_j + cL_j) / 6 and w^R_{j-1/2} =
//     q_j + (cR_j - 3 D_{j-1}) / 6 (cell_terms, cell_values in face_ff.cuh have the same in ff);
//   * the face flux is F_{a+1/2} = F(q_a) [ff] + X [FP32], where X is the change of the Euler flux from
//     the cell state q_a to the upwind face state, written as a polynomial in the offsets, plus the
//     HLLC star correction S_K (U*_K - U_K), written through the jumps of the reconstructed states
//     (S* - u_K from the pressure and velocity jumps), minus the dissipative flux; the sum is
//     rounded to FP64;
//   * R += -(F_{a+1/2} - F_{a-1/2}) / dx in FP64, so the face fluxes telescope exactly as in the
//     FP64 path (each face value is computed once and shared by its two cells).
#include <cuda_runtime.h>

#include "face_kernels.cuh"
#include "fluid_internal.cuh"

namespace fl {

namespace {

constexpr float kZepsF = 1e-20f;      // WENO5-Z epsilon in FP32 (a normal float)
constexpr float kZclampF = 1e18f;     // bound of tau5 / (beta + eps): keeps its square finite

// FP32 reciprocal, square root and reciprocal square root from the hardware approximations
// (PTX rcp.approx / sqrt.approx / rsqrt.approx, each within a few ulp; denormal inputs flush
// to zero). The FP32 increments need ~1e-7 relative accuracy, so the IEEE-rounded division and
// square root, with their refinement steps and slow-path checks, are not needed here.
__device__ __forceinline__ float rcpf(float y) {
  float r; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y)); return r;
}
__device__ __forceinline__ float sqrtf_a(float y) {
  float r; asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y)); return r;
}
__device__ __forceinline__ float rsqrtf_a(float y) {
  float r; asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y)); return r;
}

// ---- bulk copies into shared memory: cp.async.bulk (the TMA unit's untiled copy) completing on an mbarrier,
// with a bounded wait.  The face kernels load plainly (bulk-staged tiles were slower); what is here serves
// fluid_check_bulk_staging (k_bulk_probe) ----
__device__ __forceinline__ unsigned smem_u32(const void* p) {
  return (unsigned)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// one arrival that also raises the phase's expected transaction count by `bytes`
__device__ __forceinline__ void mbar_arrive_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// global -> shared copy of `bytes` (a multiple of 16; both addresses 16-byte aligned), counted on bar
__device__ __forceinline__ void bulk_to_smem(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_test(unsigned bar, unsigned parity) {
  unsigned done;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
               "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(done) : "r"(bar), "r"(parity) : "memory");
  return done != 0;
}
// Bounded wait for the phase of the given parity: non-blocking tests with a short sleep between
// them, 2^17 of them at most (of the order of 10 ms); false if the phase did not complete.
__device__ __forceinline__ bool mbar_wait_bounded(unsigned bar, unsigned parity) {
  for (int it = 0; it < (1 << 17); ++it) {
    if (mbar_test(bar, parity)) return true;
    __nanosleep(64);
  }
  return false;
}

int grid_for(long long work, int block) {
  long long b = (work + block - 1) / block;
  if (b < 1) b = 1;
  if (b > 152LL * 64) b = 152LL * 64;
  return (int)b;
}

// FP32 copies of the physical constants the increments use (no per-face conversions)
struct PhysF {
  float gamma, gm1, igm1, gg;            // gg = gamma / (gamma - 1)
  float mu_ref, iT_ref, visc_exp, TS, S; // TS = T_ref + S (Sutherland)
  float lam_fac, eps4, dt_visc_k;        // eps4 = 4 epsilon (WENO5-Z: of kZepsF)
  int visc;
};

__host__ __device__ inline PhysF phys_f(const Phys& ph) {
  PhysF f;
  f.gamma = (float)ph.gamma; f.gm1 = (float)ph.gm1; f.igm1 = (float)ph.igm1;
  f.gg = (float)(ph.gamma * ph.igm1);
  f.mu_ref = (float)ph.mu_ref; f.iT_ref = (float)ph.iT_ref; f.visc_exp = (float)ph.visc_exp;
  f.TS = (float)(ph.T_ref + ph.suth_S); f.S = (float)ph.suth_S;
  f.lam_fac = (float)ph.lam_fac; f.eps4 = 4.0f * (ph.weno == FLUID_WENO_JS ? (float)ph.eps : kZepsF); f.dt_visc_k = (float)ph.dt_visc_k;
  f.visc = ph.visc;
  return f;
}

// Indicator terms of cell j in FP32: 4 (beta + eps) of its three-cell stencil as the left (A), centre
// (B) and right (C) candidate (cell_terms)
__device__ __forceinline__ void cell_terms32(float D, float T, float eps4, float& A, float& B, float& C) {
  const float K = s_fma(s_mul(13.0f / 3.0f, T), T, eps4);
  const float sB = s_fma(2.0f, D, -T), sA = s_fma(2.0f, T, sB), sC = s_fma(2.0f, T, -sB);
  A = s_fma(sA, sA, K);
  B = s_fma(sB, sB, K);
  C = s_fma(sC, sC, K);
}

// Six times the corrections of cell j's two face values (cell_values): cL, cR from the indicator set
// A_{j-1}, B_j, C_{j+1}, T_j and the third differences V0 = T_j - T_{j-1}, V1 = T_{j+1} - T_j
template <int SCHEME>
__device__ __forceinline__ void cell_corr32(float e0, float e1, float e2, float T, float V0, float V1, float& cL,
                                            float& cR) {
  const float r0 = rcpf(e0), r1 = rcpf(e1), r2 = rcpf(e2);
  float W0, W1, W2;
  if (SCHEME == FLUID_WENO_JS) {
    const float em = fminf(fminf(e0, e1), e2);           // a common factor keeps the squares in range
    W0 = s_mul(em, r0); W1 = s_mul(em, r1); W2 = s_mul(em, r2);
    W0 = s_mul(W0, W0); W1 = s_mul(W1, W1); W2 = s_mul(W2, W2);
  } else {
    const float tau = fabsf(s_sub(e0, e2));
    W0 = fminf(s_mul(tau, r0), kZclampF);
    W1 = fminf(s_mul(tau, r1), kZclampF);
    W2 = fminf(s_mul(tau, r2), kZclampF);
    W0 = s_fma(W0, W0, 1.0f); W1 = s_fma(W1, W1, 1.0f); W2 = s_fma(W2, W2, 1.0f);
  }
  const float P0 = s_mul(W0, V0), P2 = s_mul(W2, V1), S = s_add(P0, P2);
  const float base = s_fma(6.0f, W1, s_add(W0, W2));
  cL = s_fma(-s_fma(2.0f, S, P2), rcpf(s_fma(2.0f, W2, base)), -T);
  cR = s_fma(s_fma(2.0f, S, P0), rcpf(s_fma(2.0f, W0, base)), -T);
}

__device__ __forceinline__ float viscosity_f(float T, const PhysF& pf) {
  if (pf.visc == FLUID_VISC_CONSTANT) return pf.mu_ref;
  const float r = s_mul(T, pf.iT_ref);
  if (pf.visc == FLUID_VISC_POWER) return s_mul(pf.mu_ref, __powf(r, pf.visc_exp));
  return s_mul(s_mul(s_mul(pf.mu_ref, s_mul(r, sqrtf_a(r))), pf.TS), rcpf(s_add(T, pf.S)));
}

// X: change of the face flux relative to F(q_a), in FP32 (see the file comment).  Every operation is
// explicit, so that all kernels inlining it (and the functions below) give the same bits.
//   b        FP32 cell state q_a (rho, u, v, w, p)
//   dL, J    offset of the reconstructed left face state from q_a, and the jump to the right one
template <int D>
__device__ __forceinline__ void hllc_delta(const float b[5], const float dL[5], const float J[5],
                                           const PhysF& pf, float X[5]) {
  const float g = pf.gamma, gm1 = pf.gm1, igm1 = pf.igm1;
  float wl[5], wr[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    wl[v] = s_add(b[v], dL[v]);
    wr[v] = s_add(wl[v], J[v]);
  }
  const float rL = wl[0], pL = wl[4], rR = wr[0], pR = wr[4];
  const float unL = wl[1 + D], unR = wr[1 + D], Jn = J[1 + D];
  const float isL = rsqrtf_a(rL), isR = rsqrtf_a(rR);          // 1/sqrt(rho)
  const float cL2 = s_mul(s_mul(g, pL), s_mul(isL, isL)), cR2 = s_mul(s_mul(g, pR), s_mul(isR, isR));
  const float cL = sqrtf_a(cL2), cR = sqrtf_a(cR2);
  // Roe averages as in hllc_ff: u~ = u_L + a_R J_u,
  // c~^2 = a_L c_L^2 + a_R c_R^2 + (gamma - 1)/2 a_L a_R |J_u|^2
  const float sL = s_mul(rL, isL), sR = s_mul(rR, isR);
  const float aR = s_mul(sR, rcpf(s_add(sL, sR))), aL = s_sub(1.0f, aR);
  const float q2J = s_fma(J[1], J[1], s_fma(J[2], J[2], s_mul(J[3], J[3])));
  const float ct = sqrtf_a(s_fma(aR, s_fma(s_mul(s_mul(0.5f, gm1), aL), q2J, s_sub(cR2, cL2)), cL2));
  const float ut = s_mul(aR, Jn);                              // u~ - u_L
  const float sl = fminf(-cL, s_sub(ut, ct));                  // S_L - u_L
  const float sr = fmaxf(cR, s_add(s_sub(ut, Jn), ct));        // S_R - u_R
  const float SL = s_add(unL, sl), SR = s_add(unR, sr);
  const float mL = s_mul(rL, sl), mR = s_mul(rR, sr);
  // S* - u_L from the jumps: (dp - m_R du_n) / (m_L - m_R)
  const float sigL = s_mul(s_fma(-mR, Jn, J[4]), rcpf(s_sub(mL, mR)));
  const float Ss = s_add(unL, sigL);

  const bool left = (SL >= 0.0f) || (Ss >= 0.0f);
  const bool star = left ? !(SL >= 0.0f) : (SR > 0.0f);
  // the upwind side's offsets and state, selected value by value so that both arrays stay
  // in registers
  float d[5], w[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) { d[v] = left ? dL[v] : s_add(dL[v], J[v]); w[v] = left ? wl[v] : wr[v]; }

  // Euler-flux change from q_a to the face state K = b + d
  const float un = b[1 + D], unK = w[1 + D];
  const float mn = s_mul(b[0], un);
  const float dm = s_fma(b[0], d[1 + D], s_mul(d[0], unK));    // rho' u_n' - rho u_n
  X[0] = dm;
#pragma unroll
  for (int c = 0; c < 3; ++c) X[1 + c] = s_fma(dm, w[1 + c], s_mul(mn, d[1 + c]));
  X[1 + D] = s_add(X[1 + D], d[4]);
  const float q2b = s_fma(b[1], b[1], s_fma(b[2], b[2], s_mul(b[3], b[3])));
  const float dq2 = s_fma(d[1], s_fma(2.0f, b[1], d[1]),
                          s_fma(d[2], s_fma(2.0f, b[2], d[2]), s_mul(d[3], s_fma(2.0f, b[3], d[3]))));
  const float gg = pf.gg, hr = s_mul(0.5f, b[0]);
  const float Hv = s_fma(gg, b[4], s_mul(hr, q2b));            // E + p of q_a
  const float q2K = s_add(q2b, dq2);
  const float dHv = s_fma(gg, d[4], s_fma(s_mul(0.5f, d[0]), q2K, s_mul(hr, dq2)));
  X[4] = s_fma(d[1 + D], s_add(Hv, dHv), s_mul(un, dHv));

  if (star) {
    // S_K (U*_K - U_K) with theta = (S* - u_K)/(S_K - S*), chi = 1 + theta
    const float S = left ? SL : SR, sK = left ? sl : sr;
    const float sig = left ? sigL : s_sub(sigL, Jn);
    const float rK = w[0], pK = w[4];
    const float EK = s_fma(pK, igm1, s_mul(s_mul(0.5f, rK), q2K));
    const float theta = s_mul(sig, rcpf(s_sub(sK, sig)));
    const float cs = s_fma(theta, sig, sig);                   // chi sigma
    const float f0 = s_mul(S, s_mul(rK, theta));
    X[0] = s_add(X[0], f0);
#pragma unroll
    for (int c = 0; c < 3; ++c) X[1 + c] = s_fma(f0, w[1 + c], X[1 + c]);
    X[1 + D] = s_fma(S, s_mul(rK, cs), X[1 + D]);
    X[4] = s_fma(S, s_fma(theta, EK, s_mul(cs, s_fma(rK, Ss, s_mul(pK, rcpf(sK))))), X[4]);
  }
}

__device__ __forceinline__ float interp32(const float* __restrict__ f, int s) {
  return s_mul(s_fma(9.0f, s_add(ld(f), ld(f + s)), -s_add(ld(f - s), ld(f + 2 * s))), 0.0625f);
}

// The Euler flux of a cell's pairs along D plus the increment X, as FP64
template <int D>
__device__ __forceinline__ void assemble_flux(const ff q[5], const Phys& ph, const float X[5], double F[5]) {
  const ff un = q[1 + D], mn = q[0] * un;
  const ff q2 = fma_weak(q[1], q[1], fma_weak(q[2], q[2], sqr_weak(q[3])));
  const ff gg = ph.k.gg;
  ff f[5];
  f[0] = mn;
#pragma unroll
  for (int c = 0; c < 3; ++c) f[1 + c] = c == D ? ff_fma(mn, q[1 + c], q[4]) : mn * q[1 + c];
  f[4] = ff_fma(mul_weak(un, gg), q[4], mul_weak(ff_scale(mn, 0.5f), q2));
#pragma unroll
  for (int v = 0; v < 5; ++v) F[v] = ff_to_double(f[v] + X[v]);
}

// The face flux at i+1/2 (cell i: `cell`) from its cell's pairs q, the corrections cL, cR, D = q_{i+1} -
// q_i, and for the dissipative flux Ts = T_i + T_{i+1}, Td = T_{i+1} - T_i of the velocities and, last, the
// temperature, whose D is Dt and cell value Tc
template <int D, bool VISC>
__device__ __forceinline__ void mixed_face(const float* __restrict__ W32, const float* __restrict__ G32, int cell,
                                           int s, int i, const Geo& g, const Phys& ph, const PhysF& pf, const ff q[5],
                                           const float cL[5], const float cR[5], const float Dv[5], const float Ts[4],
                                           const float Td[4], float Dt, float Tc, double F[5]) {
  const int nc = g.ncell;
  float b[5], dL[5], J[5], X[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    b[v] = q[v].h;
    dL[v] = s_mul(1.0f / 6.0f, s_fma(3.0f, Dv[v], cL[v]));
    J[v] = s_mul(1.0f / 6.0f, s_sub(cR[v], cL[v]));
  }
  hllc_delta<D>(b, dL, J, pf, X);
  if (VISC) {
    // value f_a + D/2 - (T_a + T_{a+1}) / 16 and derivative D - (T_{a+1} - T_a) / 24 of the 4-cell stencils
    const float mfa = __ldg(g.mf32[D] + i);
    float vf[3], dn[3], gd[3], gb[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      vf[c] = s_add(b[1 + c], s_fma(-0.0625f, Ts[c], s_mul(0.5f, Dv[1 + c])));
      dn[c] = s_mul(s_fma(-1.0f / 24.0f, Td[c], Dv[1 + c]), mfa);
    }
    const float Tf = s_add(Tc, s_fma(-0.0625f, Ts[3], s_mul(0.5f, Dt)));
    const float dT = s_mul(s_fma(-1.0f / 24.0f, Td[3], Dt), mfa);
    float tr = 0.0f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (c == D || c >= g.ndim) continue;
      gd[c] = interp32(G32 + (D * 3 + c) * nc + cell, s);
      gb[c] = interp32(G32 + (c * 3 + c) * nc + cell, s);
      tr = s_add(tr, gb[c]);
    }
    const float mu = viscosity_f(Tf, pf);
    float tau[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (c == D) tau[c] = s_mul(mu, s_mul(2.0f / 3.0f, s_fma(2.0f, dn[D], -tr)));
      else tau[c] = s_mul(mu, c < g.ndim ? s_add(dn[c], gd[c]) : dn[c]);
      X[1 + c] = s_sub(X[1 + c], tau[c]);
    }
    X[4] = s_sub(X[4], s_fma(vf[0], tau[0], s_fma(vf[1], tau[1], s_fma(vf[2], tau[2], s_mul(s_mul(mu, pf.lam_fac), dT)))));
  }
  assemble_flux<D>(q, ph, X, F);
}

// The stage of one interior cell once its right-hand side is complete: R_v = its value from the
// other axes' kernels (null: none) minus this axis's flux difference (the FP64 accumulation of
// update_r), then the arithmetic of k_stage_prim -- body force, the RK3 combination into Ud, the
// primitives of Ud -- into the second buffer.  W32: the current primitives (the body-force
// velocities of the stage's input state).
__device__ __forceinline__ void stage_cell(const StageOut& so, const double* __restrict__ R,
                                           const float* __restrict__ W32, int nc, int cell, double id,
                                           const double F[5], const double Fp[5], double dt, bool hold,
                                           const Phys& ph, bool& bad) {
  double u[5];
  if (hold) {
#pragma unroll
    for (int v = 0; v < 5; ++v) u[v] = so.Un[v * nc + cell];
  } else {
    double r[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const double dF = __dsub_rn(F[v], Fp[v]);
      r[v] = R ? fma(-id, dF, R[v * nc + cell]) : __dmul_rn(-id, dF);
    }
    if (ph.has_force) {
      const double vx = ff_to_double(load_pair(W32, nc, 1, cell)), vy = ff_to_double(load_pair(W32, nc, 2, cell)),
                   vz = ff_to_double(load_pair(W32, nc, 3, cell));
      r[1] += ph.f[0];
      r[2] += ph.f[1];
      r[3] += ph.f[2];
      r[4] += fma(ph.f[0], vx, fma(ph.f[1], vy, ph.f[2] * vz));
    }
    double un[5], us[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) un[v] = so.Un[v * nc + cell];
    if (so.stage != 1) {
#pragma unroll
      for (int v = 0; v < 5; ++v) us[v] = so.Us[v * nc + cell];
    }
    stage_combine(so.stage, dt, un, us, r, u);
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      bad |= !finite_bits(u[v]);
      so.Ud[v * nc + cell] = u[v];
    }
  }
  if (!so.prims) return;
  ff w[NW];
  prim_ff(u, ph, w);
#pragma unroll
  for (int v = 0; v < NW; ++v) store_pair(so.W32, nc, v, cell, w[v]);
}

// Tiles as in k_face_tile_body: one thread per cell of a run along D, the terms of neighbouring cells
// through shared memory.  Waiting for memory binds (the y launch on TGV 128^3 issued in 42 % of the
// cycles at 24 warps per SM), so the tiles take 64 registers for 32 warps and ask L2 early for the lines
// that a thread reads last.  TGV 128^3, one launch (x, y, z with the stage): 0.095, 0.14 and 0.195 ms,
// 0.135, 0.17 and 0.285 ms before with WENO5 formed for each side of a face and the FP64 cell flux.
// Along y and z 8 x 32 was faster than 16 x 32, 32 x 32 and 4 x 64 (z by up to a fifth), and than a march
// with the terms in registers (128 registers, 13 warps per SM: y 0.20, z 0.38 ms).
template <int D>
struct MixedShape {
  // the FP64 tiles' shape, so that batches lay out both alike (batch_plan)
  static constexpr int TX = TileShape<D>::TX, TD = TileShape<D>::TD;
  static constexpr int threads = TX * TD, step = TD - 5, blocks = 32 * 32 / threads;
};

__device__ __forceinline__ void prefetch_line(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

template <int N>
struct MixedShared {
  float D[6][N], T[5][N], A[5][N], C[5][N], cR[5][N];
  double F[5][N];
};

template <int D, int SCHEME, bool VISC, bool STAGE>
__device__ __forceinline__ void k_face_mixed_body(const float* __restrict__ W32, const float* __restrict__ G32,
                                                  double* __restrict__ R, const Geo& g, const Phys& ph, const PhysF& pf,
                                                  MixedShared<MixedShape<D>::threads>& sh, int col,
                                                  long long tile, const StageOut* so) {
  constexpr int TX = MixedShape<D>::TX, TD = MixedShape<D>::TD;
  constexpr int NVW = VISC ? 6 : 5;
  const int t = threadIdx.x, row = t / TX, nc = g.ncell;
  const int s = D == 0 ? 1 : (D == 1 ? g.sy : g.sz);
  const TileCell tc = tile_cell<D, MixedShape<D>>(g, col, tile);
  const int i = tc.i, cell = tc.cell;
  // fused stage: dt of the step, the third stage's hold (dt <= 0) and its clock update
  double dt = 0.0;
  bool hold = false, bad = false;
  if (STAGE) {
    dt = so->ctl->dt;
    hold = so->stage == 3 && !(dt > 0.0);
    if (so->stage == 3 && !hold && col == 0 && tile == 0 && t == 0) {
      const double tn = so->ctl->t + dt;
      so->ctl->t = (so->t_end > 0.0 && !(tn < so->t_end)) ? so->t_end : tn;
    }
  }
  // what the thread reads after its terms are formed (with the stage, whose own reads already fill
  // the memory system, this costs time: z 0.195 -> 0.21 ms)
  if (!STAGE && tc.live && i >= g.h[D] && i < g.h[D] + g.n[D]) {
    if (D > 0) {
#pragma unroll
      for (int v = 0; v < 5; ++v) prefetch_line(R + v * nc + cell);
    }
    if (VISC) {
#pragma unroll
      for (int b = 0; b < 3; ++b)
        if (b != D && b < g.ndim) {
          prefetch_line(G32 + (D * 3 + b) * nc + cell);
          prefetch_line(G32 + (b * 3 + b) * nc + cell);
        }
    }
  }
  float D0[NVW], Tc = 0.0f;
  ff q[5];
#pragma unroll
  for (int v = 0; v < NVW; ++v) {
    const float* hp = W32 + v * nc + cell;
    const float* lp = W32 + (NW + v) * nc + cell;
    const ff q0{ld(hp), ld(lp)};
    D0[v] = tc.pair ? s_add(s_sub(ld(hp + s), q0.h), s_sub(ld(lp + s), q0.l)) : 0.0f;
    if (v < 5) q[v] = q0;
    else Tc = q0.h;
    sh.D[v][t] = D0[v];
  }
  __syncthreads();
  const bool up = row > 0;
  float T0[5], B0[5];
#pragma unroll
  for (int v = 0; v < 5; ++v) {
    T0[v] = s_sub(D0[v], up ? sh.D[v][t - TX] : 0.0f);
    float A, C;
    cell_terms32(D0[v], T0[v], pf.eps4, A, B0[v], C);
    sh.T[v][t] = T0[v];
    sh.A[v][t] = A;
    sh.C[v][t] = C;
  }
  __syncthreads();
  const bool inner = row >= 2 && row < TD - 1;
  float cL[5], Tn[3] = {0.0f, 0.0f, 0.0f};
  if (inner) {
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const float T1 = sh.T[v][t + TX];
      if (v >= 1 && v <= 3) Tn[v - 1] = T1;
      float cR;
      cell_corr32<SCHEME>(sh.A[v][t - TX], B0[v], sh.C[v][t + TX], T0[v], s_sub(T0[v], sh.T[v][t - TX]),
                          s_sub(T1, T0[v]), cL[v], cR);
      sh.cR[v][t] = cR;
    }
  }
  __syncthreads();
  const bool face = row >= 2 && row < TD - 2 && tc.live && i >= g.h[D] - 1 && i < g.h[D] + g.n[D];
  double F[5];
  if (face) {
    float cR[5], Ts[4], Td[4];
#pragma unroll
    for (int v = 0; v < 5; ++v) cR[v] = sh.cR[v][t + TX];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      Ts[c] = s_add(T0[1 + c], Tn[c]);
      Td[c] = s_sub(Tn[c], T0[1 + c]);
    }
    if (VISC) {
      const float Ta = s_sub(D0[NVW - 1], sh.D[NVW - 1][t - TX]), Tj = s_sub(sh.D[NVW - 1][t + TX], D0[NVW - 1]);
      Ts[3] = s_add(Ta, Tj);
      Td[3] = s_sub(Tj, Ta);
    }
    mixed_face<D, VISC>(W32, G32, cell, s, i, g, ph, pf, q, cL, cR, D0, Ts, Td, D0[NVW - 1], Tc, F);
#pragma unroll
    for (int v = 0; v < 5; ++v) sh.F[v][t] = F[v];
  }
  __syncthreads();
  if (face && row >= 3 && i >= g.h[D]) {
    const double id = g.idx[D][i];
    double Fp[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) Fp[v] = sh.F[v][t - TX];
    if (STAGE) {
      stage_cell(*so, R, W32, nc, cell, id, F, Fp, dt, hold, ph, bad);
    } else {
#pragma unroll
      for (int v = 0; v < 5; ++v) update_r<D>(R + v * nc + cell, F[v], Fp[v], id);
    }
  }
  if (STAGE && bad) atomicOr(&so->ctl->flags, FLAG_NONFINITE);
}

template <int SCHEME, bool VISC>
__global__ void __launch_bounds__(MixedShape<0>::threads, MixedShape<0>::blocks) k_face_mixed_x(
    const float* W32, const float* G32, double* R,
    const __grid_constant__ Geo g, const __grid_constant__ Phys ph, PhysF pf) {
  step_wait();
  extern __shared__ __align__(16) unsigned char raw[];
  const int cols = tile_cols<0, MixedShape<0>>(g);
  k_face_mixed_body<0, SCHEME, VISC, false>(W32, G32, R, g, ph, pf,
                                            *reinterpret_cast<MixedShared<MixedShape<0>::threads>*>(raw),
                                            blockIdx.x % cols, blockIdx.x / cols, nullptr);
}

// the tangential axes
template <int D, int SCHEME, bool VISC>
__global__ void __launch_bounds__(MixedShape<D>::threads, MixedShape<D>::blocks) k_face_mixed_t(
    const float* W32, const float* G32, double* R,
    const __grid_constant__ Geo g, const __grid_constant__ Phys ph, PhysF pf) {
  step_wait();
  extern __shared__ __align__(16) unsigned char raw[];
  const int cols = tile_cols<D, MixedShape<D>>(g);
  k_face_mixed_body<D, SCHEME, VISC, false>(W32, G32, R, g, ph, pf,
                                            *reinterpret_cast<MixedShared<MixedShape<D>::threads>*>(raw),
                                            blockIdx.x % cols, blockIdx.x / cols, nullptr);
}

// the last axis's kernel with the stage fused (StageOut): R is read, not written
template <int D, int SCHEME, bool VISC>
__global__ void __launch_bounds__(MixedShape<D>::threads, MixedShape<D>::blocks) k_face_mixed_ts(
    const float* W32, const float* G32, const double* R,
    const __grid_constant__ Geo g, const __grid_constant__ Phys ph, PhysF pf, const __grid_constant__ StageOut so) {
  step_wait();
  extern __shared__ __align__(16) unsigned char raw[];
  const int cols = tile_cols<D, MixedShape<D>>(g);
  k_face_mixed_body<D, SCHEME, VISC, true>(W32, G32, const_cast<double*>(R), g, ph, pf,
                                           *reinterpret_cast<MixedShared<MixedShape<D>::threads>*>(raw),
                                           blockIdx.x % cols, blockIdx.x / cols, &so);
}

// centre velocity gradients in FP32 from the FP32 primitives (fourth-order central)
__device__ __forceinline__ void k_grad32_body(const float* __restrict__ W32, float* __restrict__ G32, Geo g,
    uint3 bid, uint3 gdim) {
  int lo[3], ext[3];
  for (int a = 0; a < 3; ++a) {
    const int m = a < g.ndim ? 2 : 0;
    lo[a] = g.h[a] - m;
    ext[a] = g.n[a] + 2 * m;
  }
  const int total = ext[0] * ext[1] * ext[2];
  for (int t = bid.x * blockDim.x + threadIdx.x; t < total; t += gdim.x * blockDim.x) {
    int c[3];
    c[0] = lo[0] + t % ext[0];
    const int r = t / ext[0];
    c[1] = lo[1] + r % ext[1];
    c[2] = lo[2] + r / ext[1];
    const int cell = c[0] + c[1] * g.sy + c[2] * g.sz;
    // all loads before the first store: TGV 128^3 37 us a launch, 45 with the stores between them
    float d[9];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const bool inb = b < g.ndim && c[b] >= g.h[b] && c[b] < g.h[b] + g.n[b];
      const int s = b == 0 ? 1 : (b == 1 ? g.sy : g.sz);
      const float m = inb ? g.mc32[b][c[b]] : 0.0f;
#pragma unroll
      for (int comp = 0; comp < 3; ++comp) {
        d[comp * 3 + b] = 0.0f;
        if (inb) {
          const float* f = W32 + (1 + comp) * g.ncell + cell;
          d[comp * 3 + b] = ((f[-2 * s] - f[2 * s]) + 8.0f * (f[s] - f[-s])) * (1.0f / 12.0f) * m;
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) G32[k * g.ncell + cell] = d[k];
  }
}

__global__ void k_grad32(const float* W32, float* G32, Geo g) {
  step_wait();
  k_grad32_body(W32, G32, g, blockIdx, gridDim);
}


// CFL partial maxima of the rates (|u| + c) / dx and k nu / dx^2 (the inverse time steps, as in
// the FP64 kernel) from the FP32 primitives: the time step needs no more than FP32 accuracy
__device__ __forceinline__ void k_dt32_body(const float* __restrict__ W32, const Geo& g, const Phys& ph,
                                            const PhysF& pf, double* partial, int nparts, Ctl* ctl, double* dt_out,
                                            int clip, double t_end, uint3 bid, uint3 gdim) {
  if (nparts == 0) {                          // a fixed dt
    if (threadIdx.x == 0) dt_store(0.0, ph, ctl, dt_out, clip, t_end);
    return;
  }
  const int total = g.n[0] * g.n[1] * g.n[2];
  const int nc = g.ncell;
  float best = 0.0f;
  const float gam = pf.gamma, k = pf.dt_visc_k;
  for (int t = bid.x * blockDim.x + threadIdx.x; t < total; t += gdim.x * blockDim.x) {
    const int i = t % g.n[0];
    const int r = t / g.n[0];
    const int j = r % g.n[1];
    const int kk = r / g.n[1];
    const int ci[3] = {i + g.h[0], j + g.h[1], kk + g.h[2]};
    const int c = ci[0] + ci[1] * g.sy + ci[2] * g.sz;
    const float rho = W32[c], p = W32[4 * nc + c];
    const float irho = rcpf(rho);
    const float cs = sqrtf_a(gam * p * irho);
    float knu = 0.0f;
    if (pf.visc != FLUID_VISC_NONE) knu = k * viscosity_f(W32[5 * nc + c], pf) * irho;
    for (int d = 0; d < g.ndim; ++d) {
      const float id = g.idx32[d][ci[d]];
      best = fmaxf(best, (fabsf(W32[(1 + d) * nc + c]) + cs) * id);
      if (pf.visc != FLUID_VISC_NONE) best = fmaxf(best, knu * id * id);
    }
  }
  __shared__ double sm[kDtBlock / 32];
  __shared__ unsigned last;
  best = block_max(best, reinterpret_cast<float*>(sm));
  if (threadIdx.x == 0) {
    __stcg(partial + bid.x, (double)best);
    __threadfence();
    last = atomicInc(&ctl->ticket, nparts - 1) == (unsigned)(nparts - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double top = 0.0;
  for (int i = threadIdx.x; i < nparts; i += blockDim.x) top = fmax(top, __ldcg(partial + i));
  top = block_max(top, sm);
  if (threadIdx.x == 0) dt_store(top, ph, ctl, dt_out, clip, t_end);
}

__global__ void __launch_bounds__(kDtBlock) k_dt32(const float* W32, const __grid_constant__ Geo g,
                                                   const __grid_constant__ Phys ph, const __grid_constant__ PhysF pf,
                                                   double* partial, int nparts, Ctl* ctl, double* dt_out, int clip,
                                                   double t_end) {
  step_wait();
  k_dt32_body(W32, g, ph, pf, partial, nparts, ctl, dt_out, clip, t_end, blockIdx, gridDim);
}

// ---- batched kernels of the serving loop (see BatchTable in fluid_internal.cuh) -----------------
template <int D, int SCHEME, bool VISC>
__global__ void __launch_bounds__(MixedShape<D>::threads, MixedShape<D>::blocks) kbm_face(
    const BatchTable* __restrict__ t, int step) {
  extern __shared__ __align__(16) unsigned char raw[];
  FL_BATCH_LOOP(BK_FACE0 + D)
  (void)gdim;
  if (step < S.steps)
    k_face_mixed_body<D, SCHEME, VISC, false>(S.W32, S.G32, S.R, S.g, S.ph, phys_f(S.ph),
                                              *reinterpret_cast<MixedShared<MixedShape<D>::threads>*>(raw), bid.x, bid.y,
                                              nullptr);
  FL_BATCH_END
}

__global__ void __launch_bounds__(256) kbm_grad(const BatchTable* __restrict__ t, int step) {
  FL_BATCH_LOOP(BK_GRAD)
  if (step < S.steps) k_grad32_body(S.W32, S.G32, S.g, bid, gdim);
  FL_BATCH_END
}

__global__ void __launch_bounds__(kDtBlock) kbm_dt(const BatchTable* __restrict__ t, int step) {
  FL_BATCH_LOOP(BK_DT)
  if (step < S.steps)
    k_dt32_body(S.W32, S.g, S.ph, phys_f(S.ph), S.partial, S.nparts, S.ctl, nullptr, 1, S.t_end, bid, gdim);
  FL_BATCH_END
}

template <int D, int SCHEME, bool VISC>
cudaError_t batch_face_d(const BatchTable* dev, int step, cudaStream_t st) {
  constexpr int n = MixedShape<D>::threads;
  constexpr size_t smem = sizeof(MixedShared<n>);
  const cudaError_t e =
      cudaFuncSetAttribute(kbm_face<D, SCHEME, VISC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  static const int grid = batch_grid(kbm_face<D, SCHEME, VISC>, n, smem);
  (kbm_face<D, SCHEME, VISC><<<grid, n, smem, st>>>(dev, step), ++t_launches);
  return cudaGetLastError();
}

template <int SCHEME, bool VISC>
cudaError_t batch_face_m(const BatchTable* dev, int D, int step, cudaStream_t st) {
  if (D == 0) return batch_face_d<0, SCHEME, VISC>(dev, step, st);
  if (D == 1) return batch_face_d<1, SCHEME, VISC>(dev, step, st);
  return batch_face_d<2, SCHEME, VISC>(dev, step, st);
}

template <int D, int SCHEME, bool VISC>
cudaError_t launch_t(const float* W32, const float* G32, double* R, const Geo& g, const Phys& ph, const StageOut* so,
                     cudaStream_t st) {
  const PhysF pf = phys_f(ph);
  constexpr int n = MixedShape<D>::threads;
  constexpr size_t smem = sizeof(MixedShared<n>);
  const unsigned grid = (unsigned)(tile_rows<D, MixedShape<D>>(g) * tile_cols<D, MixedShape<D>>(g));
  // a tile may need more than the default 48 KB of dynamic shared memory (the attribute is per device)
  cudaError_t e;
  if (so) {
    e = cudaFuncSetAttribute(k_face_mixed_ts<D, SCHEME, VISC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    launch_step(k_face_mixed_ts<D, SCHEME, VISC>, grid, n, smem, st, W32, G32, R, g, ph, pf, *so);
  } else {
    constexpr auto kernel = [] {
      if constexpr (D == 0) return &k_face_mixed_x<SCHEME, VISC>;
      else return &k_face_mixed_t<D, SCHEME, VISC>;
    }();
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    launch_step(kernel, grid, n, smem, st, W32, G32, R, g, ph, pf);
  }
  return cudaGetLastError();
}

template <int SCHEME, bool VISC>
cudaError_t launch_sv(int D, const float* W32, const float* G32, double* R, const Geo& g, const Phys& ph,
                      const StageOut* so, cudaStream_t st) {
  if (D == 0) return launch_t<0, SCHEME, VISC>(W32, G32, R, g, ph, so, st);
  if (D == 1) return launch_t<1, SCHEME, VISC>(W32, G32, R, g, ph, so, st);
  return launch_t<2, SCHEME, VISC>(W32, G32, R, g, ph, so, st);
}

cudaError_t launch_any(int D, const float* W32, const float* G32, double* R, const Geo& g, const Phys& ph,
                       const StageOut* so, cudaStream_t st) {
  const bool visc = ph.visc != FLUID_VISC_NONE;
  if (ph.weno == FLUID_WENO_JS)
    return visc ? launch_sv<FLUID_WENO_JS, true>(D, W32, G32, R, g, ph, so, st)
                : launch_sv<FLUID_WENO_JS, false>(D, W32, G32, R, g, ph, so, st);
  return visc ? launch_sv<FLUID_WENO_Z, true>(D, W32, G32, R, g, ph, so, st)
              : launch_sv<FLUID_WENO_Z, false>(D, W32, G32, R, g, ph, so, st);
}

}  // namespace

cudaError_t launch_face_mixed_stage(const float* W32, const float* G32, const double* R, const Geo& g,
                                    const Phys& ph, const StageOut& so, cudaStream_t st) {
  // one-dimensional: no other axis has written R
  return launch_any(g.ndim - 1, W32, G32, g.ndim > 1 ? const_cast<double*>(R) : nullptr, g, ph, &so, st);
}

cudaError_t launch_face_mixed(int D, const float* W32, const float* G32, double* R, const Geo& g, const Phys& ph,
                              cudaStream_t st) {
  return launch_any(D, W32, G32, R, g, ph, nullptr, st);
}

constexpr int kBulkRow = 36;    // floats per row of the probe

namespace {
// Check of the bulk-staging helpers: one warp stages nrows rows of 36 floats (16-byte aligned) from
// src into shared memory on one mbarrier whose expected transaction count is the rows' bytes plus
// extra_tx, waits with the bounded wait and copies the rows to dst.  With extra_tx > 0 the
// phase cannot complete (every copy lands, the count stays short), so the wait runs out: the block
// sets FLAG_STAGING in *flags, waits once more and returns without writing dst.
constexpr int kProbeRows = 8;
__global__ void k_bulk_probe(const float* __restrict__ src, float* __restrict__ dst, int nrows,
                             unsigned extra_tx, unsigned* flags) {
  __shared__ __align__(16) float rows[kProbeRows * kBulkRow];
  __shared__ __align__(8) unsigned long long s_bar;
  const unsigned bar = smem_u32(&s_bar);
  const int lane = threadIdx.x;
  if (lane == 0) mbar_init(bar, 1);
  __syncthreads();
  if (lane == 0) mbar_arrive_expect(bar, (unsigned)(nrows * kBulkRow * sizeof(float)) + extra_tx);
  __syncwarp();
  if (lane < nrows)
    bulk_to_smem(smem_u32(rows + lane * kBulkRow), src + lane * kBulkRow, kBulkRow * sizeof(float), bar);
  const bool late = !mbar_wait_bounded(bar, 0);
  if (__syncthreads_or(late)) {
    if (lane == 0) atomicOr(flags, FLAG_STAGING);
    if (late) mbar_wait_bounded(bar, 0);
    return;
  }
  for (int i = lane; i < nrows * kBulkRow; i += 32) dst[i] = rows[i];
}
}  // namespace

cudaError_t launch_bulk_probe(const float* src, float* dst, int nrows, unsigned extra_tx,
                              unsigned* flags, cudaStream_t st) {
  if (nrows < 1 || nrows > kProbeRows || (reinterpret_cast<uintptr_t>(src) & 15) != 0)
    return cudaErrorInvalidValue;
  (k_bulk_probe<<<1, 32, 0, st>>>(src, dst, nrows, extra_tx, flags), ++t_launches);
  return cudaGetLastError();
}

cudaError_t launch_batch_mixed(const BatchTable* dev, int kind, int step, cudaStream_t st) {
  static const int gg = batch_grid(kbm_grad, 256);
  static const int gd = batch_grid(kbm_dt, kDtBlock);
  if (kind == BMX_GRAD) (kbm_grad<<<gg, 256, 0, st>>>(dev, step), ++t_launches);
  else (kbm_dt<<<gd, kDtBlock, 0, st>>>(dev, step), ++t_launches);
  return cudaGetLastError();
}

cudaError_t launch_batch_mixed_faces(const BatchTable* dev, int D, int step, int weno, bool visc,
                                     cudaStream_t st) {
  if (weno == FLUID_WENO_JS)
    return visc ? batch_face_m<FLUID_WENO_JS, true>(dev, D, step, st) : batch_face_m<FLUID_WENO_JS, false>(dev, D, step, st);
  return visc ? batch_face_m<FLUID_WENO_Z, true>(dev, D, step, st) : batch_face_m<FLUID_WENO_Z, false>(dev, D, step, st);
}

cudaError_t launch_grad32(const float* W32, float* G32, const Geo& g, cudaStream_t st) {
  long long total = 1;
  for (int a = 0; a < 3; ++a) total *= g.n[a] + (a < g.ndim ? 4 : 0);
  launch_step(k_grad32, grid_for(total, 256), 256, 0, st, W32, G32, g);
  return cudaGetLastError();
}

cudaError_t launch_dt32(const float* W32, const Geo& g, const Phys& ph, double* partial, int nparts, Ctl* ctl,
                        double* dt_out, int clip_to_ctl, double t_end, cudaStream_t st) {
  const int n = ph.dt_fixed > 0.0 ? 0 : nparts;
  launch_step(k_dt32, n > 0 ? n : 1, kDtBlock, 0, st, W32, g, ph, phys_f(ph), partial, n, ctl, dt_out, clip_to_ctl,
              t_end);
  return cudaGetLastError();
}

}  // namespace fl
