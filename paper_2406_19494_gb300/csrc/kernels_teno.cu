// FP64 face kernels with the paper's channel-flow reconstruction (Sec. 3.1): TENO6-A on the
// primitive variables with the interpolation limiter, the HLLC flux, and the dissipative flux by
// central differences of order 4 or 6 (template NP; 0 = inviscid).
//
// Interpolation limiter (reading of the paper's "interpolation limiter", its solver's
// positivity-preserving limiting of reconstructed states): a face state with rho <= 0 or p <= 0
// falls back, in all five primitives, to the cell on its side of the face.
//
// Split between the pipes as in face_kernels.cuh (an FP64 warp instruction costs the issue slots of 64
// others).  The scheme's weights are decisions: they depend on the two keep masks of the face and its
// cut-off level only, and those are taken in FP32 with an error bound, in FP64 where the bound does
// not decide (about 2 windows in 1e5).  The face values are FP64 combinations of the second differences
// with tabulated factors; HLLC's star correction and the dissipative flux are two-float terms where
// they are small against the state, else FP64.  On the channel 192 x 128 x 128 with 5 % noise (where
// HLLC stays FP64 on most faces) a launch takes 1.7 to 2.1 ms; with everything in FP64 (1,149 FP64-pipe
// instructions per face) it took 7.8 ms.
#include <cuda_runtime.h>

#include "face_kernels.cuh"
#include "teno_math.cuh"

namespace fl {

namespace {

struct TwoValues {
  double l, r;
};

// the face values in FP64 (a decision that FP32 leaves open)
__device__ __noinline__ TwoValues face_values_fp64(const double* __restrict__ f, int s, double ct,
                                                   const double (*omega)[16]) {
  double q[6], d[5];
#pragma unroll
  for (int o = 0; o < 6; ++o) q[o] = ld(f + (o - 2) * s);
#pragma unroll
  for (int o = 0; o < 5; ++o) d[o] = q[o + 1] - q[o];
  double b3[3] = {weno_B(q[1], q[2], q[3]), weno_C(q[2], q[3], q[4]), weno_A(q[0], q[1], q[2])};
  double i3[3] = {teno::rcp6(b3[0]), teno::rcp6(b3[1]), teno::rcp6(b3[2])};
  const double t0 = d[2] - d[1], t1 = d[3] - d[2];
  double kk[2] = {k1312 * t0 * t0, k1312 * t1 * t1};
  TwoValues w;
  teno::face_states(q, d, ct, b3, i3, kk, omega, w.l, w.r);
  return w;
}

__device__ __noinline__ int level_fp64(double dm, double dp) { return teno::sensor_level(dm, dp); }

// one tile: cells (col, row) as in k_face_tile_body; NVW: primitives with differences in shared memory
template <int N, int NVW>
struct TenoShared {
  double T[NVW][N];           // second differences
  double d[NVW][N];           // q_{j+1} - q_j
  double F[5][N];
  // primitives, for the reads after the calls (from global memory the x, y, z launches took 3, 2, 2.5 % longer)
  double q[5][N];
  unsigned char lev[5][N];    // cut-off levels of the cells
  double alpha[4][16], omega[4][16];
};

template <int D, int NP>
__global__ void __launch_bounds__(TileShape<D>::threads, 16 * 32 / TileShape<D>::threads) k_face_teno(
    const double* W, const double* G, double* R,
    const __grid_constant__ Geo g, const __grid_constant__ Phys ph) {
  step_wait();
  constexpr int TX = TileShape<D>::TX, TD = TileShape<D>::TD, N = TileShape<D>::threads;
  constexpr int NVW = NP ? 6 : 5;
  extern __shared__ __align__(16) unsigned char raw[];
  TenoShared<N, NVW>& sh = *reinterpret_cast<TenoShared<N, NVW>*>(raw);
  const int t = threadIdx.x, row = t / TX, nc = g.ncell;
  const int s = D == 0 ? 1 : (D == 1 ? g.sy : g.sz);
  const int cols = tile_cols<D>(g);
  const TileCell c = tile_cell<D>(g, blockIdx.x % cols, blockIdx.x / cols);
  const int i = c.i, cell = c.cell;
  if (t < 64) {
    teno::factor_entry(t, sh.alpha);
    teno::weight_entry(t, sh.omega);
  }
#pragma unroll
  for (int v = 0; v < NVW; ++v) {
    const double* f = W + v * nc + cell;
    const double q = ld(f);
    if (v < 5) sh.q[v][t] = q;
    sh.d[v][t] = c.pair ? ld(f + s) - q : 0.0;
  }
  __syncthreads();
#pragma unroll 1
  for (int v = 0; v < NVW; ++v) {
    const double d0 = sh.d[v][t], dm = row > 0 ? sh.d[v][t - TX] : 0.0;
    sh.T[v][t] = d0 - dm;
    if (v < 5) {
      bool clear;
      int l = teno::sensor_level32(ff_of(dm).h, ff_of(d0).h, clear);
      if (!clear) l = level_fp64(dm, d0);
      sh.lev[v][t] = (unsigned char)l;
    }
  }
  __syncthreads();
  // face j + 1/2
  const bool face = row >= 2 && row < TD - 2 && c.live && i >= g.h[D] - 1 && i < g.h[D] + g.n[D];
  double F[5];
  if (face) {
    const Scale sc = scale_of(sh.q[0][t + TX], sh.q[4][t + TX], ph);
    double cL[5], cR[5], d[5];
    bool small = sc.ok;
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      d[v] = sh.d[v][t];
      const double Tm = sh.T[v][t - TX], T0 = sh.T[v][t], T1 = sh.T[v][t + TX], Tp = sh.T[v][t + 2 * TX];
      const int lev = min(min(sh.lev[v][t - TX], sh.lev[v][t]), min(sh.lev[v][t + TX], sh.lev[v][t + 2 * TX]));
      const float ct = lev >= 3 ? 1e-10f : (lev == 2 ? 1e-9f : (lev == 1 ? 1e-8f : 1e-7f));
      constexpr int P = teno::kMaskScale;
      const ff fm = ff_of<P>(Tm), f0 = ff_of<P>(T0), f1 = ff_of<P>(T1), fp = ff_of<P>(Tp);
      const float Vm = s_add(s_sub(f0.h, fm.h), s_sub(f0.l, fm.l)), V = s_add(s_sub(f1.h, f0.h), s_sub(f1.l, f0.l));
      const float Vp = s_add(s_sub(fp.h, f1.h), s_sub(fp.l, f1.l)), Df = ff_of<P>(d[v]).h;
      bool kl, kr;
      const int mL = teno::keep_mask32_scaled(Df, f0.h, f1.h, fm.h, Vm, V, Vp, ct, kl);
      const int mR = teno::keep_mask32_scaled(-Df, f1.h, f0.h, fp.h, -Vp, -V, -Vm, ct, kr);
      if (kl && kr) {
        cL[v] = fma(sh.alpha[0][mL], Tm, fma(sh.alpha[1][mL], T0, fma(sh.alpha[2][mL], T1, sh.alpha[3][mL] * Tp)));
        cR[v] = fma(sh.alpha[0][mR], Tp, fma(sh.alpha[1][mR], T1, fma(sh.alpha[2][mR], T0, sh.alpha[3][mR] * Tm)));
      } else {
        const TwoValues w = face_values_fp64(W + v * nc + cell, s, teno::cutoff_of_level(lev), sh.omega);
        const double q0 = sh.q[v][t], q1 = sh.q[v][t + TX];
        cL[v] = fma(6.0, w.l - q0, -3.0 * d[v]);
        cR[v] = fma(6.0, w.r - q1, 3.0 * d[v]);
      }
      small = small && fabsf(ff_of(cR[v] - cL[v]).h) <= 6.0f * kFFJump * scale_at(sc, v);
    }
    ff X[5], m3[3];
    if (small) {
      ff wl[5], J[5];
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        const ff m = ff_of(sh.q[v][t]) + ff_scale(ff_of(d[v]), 0.5f);
        if (NP && v >= 1 && v <= 3) m3[v - 1] = m;
        J[v] = ff_of(cR[v] - cL[v]) * sixth();
        wl[v] = ff_fma(ff_of(cL[v]), sixth(), m);
      }
      // the limiter's states go to FP64
      small = wl[0].h > 0.0f && wl[4].h > 0.0f && (wl[0] + J[0]).h > 0.0f && (wl[4] + J[4]).h > 0.0f;
      if (small) {
        bool left;
        hllc_ff<D>(wl, J, ph.k, left, X);
        double w[5];
        const int o = left ? 0 : TX;
        const double three = left ? 3.0 : -3.0;
#pragma unroll
        for (int v = 0; v < 5; ++v)
          w[v] = fma(kSixth, fma(three, d[v], left ? cL[v] : cR[v]), sh.q[v][t + o]);
        euler_flux<D>(w, ph, F);
      }
    } else if (NP) {
#pragma unroll
      for (int v = 1; v <= 3; ++v)
        m3[v - 1] = ff_of(sh.q[v][t]) + ff_scale(ff_of(d[v]), 0.5f);
    }
    if (!small) {
      Flux5 l, r;
#pragma unroll
      for (int v = 0; v < 5; ++v) {
        l.f[v] = fma(kSixth, fma(3.0, d[v], cL[v]), sh.q[v][t]);
        r.f[v] = fma(kSixth, fma(-3.0, d[v], cR[v]), sh.q[v][t + TX]);
        X[v] = ff{0.0f, 0.0f};
      }
      // interpolation limiter
      if (l.f[0] <= 0.0 || l.f[4] <= 0.0) {
#pragma unroll
        for (int v = 0; v < 5; ++v) l.f[v] = sh.q[v][t];
      }
      if (r.f[0] <= 0.0 || r.f[4] <= 0.0) {
#pragma unroll
        for (int v = 0; v < 5; ++v) r.f[v] = sh.q[v][t + TX];
      }
      const Flux5 e = hllc_fp64<D>(l, r, &ph);
#pragma unroll
      for (int v = 0; v < 5; ++v) F[v] = e.f[v];
    }
    if (NP) {
      // face values and derivatives of the velocities and the temperature in their second differences:
      // order 4 as in face_of_terms; order 6 value m + (3 (T_{a-1} + T_{a+2}) - 19 (T_a + T_{a+1})) / 256,
      // derivative D + (9 (T_{a+2} - T_{a-1}) - 107 (T_{a+1} - T_a)) / 1920
      ff dv[4], vf[4];
#pragma unroll
      for (int c4 = 0; c4 < 4; ++c4) {
        const int v = c4 < 3 ? 1 + c4 : NVW - 1;
        const ff Dv = ff_of(sh.d[v][t]);
        const ff m = c4 < 3 ? m3[c4] : ff_of(ld(W + 5 * nc + cell)) + ff_scale(Dv, 0.5f);
        const ff f0 = ff_of(sh.T[v][t]), f1 = ff_of(sh.T[v][t + TX]);
        if (NP == 4) {
          dv[c4] = Dv - add_weak(f1, -f0) * ff{k24H, k24L};
          vf[c4] = m - ff_scale(add_weak(f0, f1), 0.0625f);
        } else {
          const ff fm = ff_of(sh.T[v][t - TX]), fp = ff_of(sh.T[v][t + 2 * TX]);
          const ff k1920{5.20833360e-04f, (float)(1.0 / 1920.0 - (double)5.20833360e-04f)};
          dv[c4] = Dv + (mul_weak(add_weak(fp, -fm), 9.0f) - mul_weak(add_weak(f1, -f0), 107.0f)) * k1920;
          vf[c4] = m + ff_scale(mul_weak(add_weak(fm, fp), 3.0f) - mul_weak(add_weak(f0, f1), 19.0f), 1.0f / 256);
        }
      }
      add_visc<D, NP ? NP : 4>(W, G, cell, s, i, g, ph, sc, dv, vf, vf[3], dv[3], X, F);
    }
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      F[v] = __dadd_rn(F[v], ff_to_double(X[v]));
      sh.F[v][t] = F[v];
    }
  }
  __syncthreads();
  if (face && row >= 3 && i >= g.h[D]) {
    const double id = g.idx[D][i];
#pragma unroll
    for (int v = 0; v < 5; ++v) update_r<D>(R + v * nc + cell, F[v], sh.F[v][t - TX], id);
  }
}

template <int D, int NP>
cudaError_t launch_d(const double* W, const double* G, double* R, const Geo& g, const Phys& ph,
                     cudaStream_t st) {
  constexpr int n = TileShape<D>::threads;
  constexpr size_t smem = sizeof(TenoShared<n, NP ? 6 : 5>);
  const cudaError_t e =
      cudaFuncSetAttribute(k_face_teno<D, NP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const unsigned grid = (unsigned)(tile_rows<D>(g) * tile_cols<D>(g));
  launch_step(k_face_teno<D, NP>, grid, n, smem, st, W, G, R, g, ph);
  return cudaGetLastError();
}

template <int NP>
cudaError_t launch_v(int D, const double* W, const double* G, double* R, const Geo& g, const Phys& ph,
                     cudaStream_t st) {
  if (D == 0) return launch_d<0, NP>(W, G, R, g, ph, st);
  if (D == 1) return launch_d<1, NP>(W, G, R, g, ph, st);
  return launch_d<2, NP>(W, G, R, g, ph, st);
}

}  // namespace

cudaError_t launch_face_teno(int D, const double* W, const double* G, double* R, const Geo& g,
                             const Phys& ph, cudaStream_t st) {
  if (ph.visc == FLUID_VISC_NONE) return launch_v<0>(D, W, G, R, g, ph, st);
  if (ph.visc_order == 6) return launch_v<6>(D, W, G, R, g, ph, st);
  return launch_v<4>(D, W, G, R, g, ph, st);
}

}  // namespace fl
