// FP64 kernels of the finite-volume compressible Navier-Stokes right-hand side (Section 2.1,
// Eq. ODE) and of the TVD-RK3 step.
//
// Pipeline of one right-hand-side evaluation:
//   k_prim_bc   primitives (rho, u, v, w, p, T) of every padded cell; halo cells are built directly
//               from interior cells by composing the boundary maps of the active axes in x, y, z
//               order (Section 3.2: halo cells take values assigned by the boundary conditions)
//   k_grad      fourth- or sixth-order central velocity gradients at cell centres (tangential
//               derivatives of the dissipative fluxes)
//   k_face_tile<D>   per axis (face_kernels.cuh, launched from kernels_face_js.cu and kernels_face_z.cu):
//               WENO5 reconstruction of the primitives, HLLC convective flux, the dissipative flux at the
//               same face, and the flux difference -(F+ - F-)/dx into R; one thread per cell of a tile.
//               TENO6-A has its own (k_face_teno, kernels_teno.cu)
//   k_face<D>, k_face_seam<D>   where a caller sets a segment length (fluid_tune_faces): one thread
//               marches along a segment of a grid line, and the first cell of every segment after a
//               line's first gets its update from the two fluxes that the neighbouring segments hand over
//               in the seam buffer.  Same bits as the tiles
//   k_source / k_stage   body-force source, RK3 stage combination, non-finite check
//   k_stage_prim / k_halo_prim   the stage combination fused with the primitives of its result
//               (interior cells), then the halo cells from those; fluid_step uses this pair in
//               place of k_stage followed by the next right-hand side's k_prim_bc
//   k_dt        CFL time step: per-block maxima of the rate, the last block reduces (deterministic)
//
// The state is FP64 structure-of-arrays U[v][z][y][x]; primitives and gradients live in solver
// scratch with the same padded layout.
#include <cuda_runtime.h>

#include <algorithm>

#include "face_kernels.cuh"
#include "fluid_internal.cuh"

namespace fl {

namespace {

int grid_for(long long work, int block) {
  long long b = (work + block - 1) / block;
  if (b < 1) b = 1;
  if (b > 152LL * 64) b = 152LL * 64;
  return (int)b;
}

// ------------------------------------------------------------------------------------------------
// boundary maps
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ int bc_source(int kind, int side, int a, int n, int h) {
  if (kind == FLUID_BC_PERIODIC) return side == 0 ? a + n : a - n;
  if (kind == FLUID_BC_ZERO_GRADIENT) return side == 0 ? h : h + n - 1;
  return side == 0 ? 2 * h - 1 - a : 2 * (h + n) - 1 - a;   // mirror image across the face
}

__device__ __forceinline__ void prim_of(const double* __restrict__ U, int c, int nc, const Phys& ph,
                                        double w[NW]) {
  const double u[5] = {U[c], U[nc + c], U[2 * nc + c], U[3 * nc + c], U[4 * nc + c]};
  prim_from_cons(u, ph, w);
}

__device__ __forceinline__ void wall_map(double w[NW], int kind, double Tw, double vw, int a,
                                         const Phys& ph, unsigned* flags) {
  if (!wall_map_prim(w, kind, Tw, vw, a, ph)) atomicOr(flags, FLAG_GHOST_T);
}

__device__ __forceinline__ void inflow_at(const double* __restrict__ prof, int a, const int c[3],
                                          const Geo& g, const Phys& ph, double w[NW]) {
  // tangential axes t1 < t2; profile laid out [5][p_t2][p_t1]
  const int t1 = (a == 0) ? 1 : 0;
  const int t2 = (a == 2) ? 1 : 2;
  const int plane = g.p[t1] * g.p[t2];
  const int o = c[t2] * g.p[t1] + c[t1];
  for (int v = 0; v < 5; ++v) w[v] = prof[v * plane + o];
  w[5] = w[4] / (w[0] * ph.R);
}

// Source cell of padded cell own[]: ghost[a] / side[a] / src[a] per axis; returns whether any axis
// is a halo axis (then src[] is the interior cell the halo maps start from).
// The halo layers of an exchange face (a sub-domain boundary of a block decomposition) hold the
// neighbouring block's cells: along that axis the cell is its own source, like an interior cell.
__device__ __forceinline__ bool halo_source(const int own[3], const Geo& g, const BC& bc,
                                            bool ghost[3], int side[3], int src[3]) {
  bool any = false;
  for (int a = 0; a < 3; ++a) {
    side[a] = own[a] < g.h[a] ? 0 : 1;
    ghost[a] = (own[a] < g.h[a] || own[a] >= g.h[a] + g.n[a]) &&
               bc.kind[a][side[a]] != FLUID_BC_EXCHANGE;
    src[a] = ghost[a] ? bc_source(bc.kind[a][side[a]], side[a], own[a], g.n[a], g.h[a]) : own[a];
    any |= ghost[a];
  }
  return any;
}

// the maps of the halo axes of a cell, in axis order, applied to the primitives w of its source;
// returns whether any of them changes values (a wall or inflow map) rather than only indices
__device__ __forceinline__ bool halo_maps(const int own[3], const bool ghost[3], const int side[3],
                                          const int src[3], const Geo& g, const Phys& ph,
                                          const BC& bc, Ctl* ctl, double w[NW]) {
  bool valued = false;
  for (int a = 0; a < 3; ++a) {
    if (!ghost[a]) continue;
    const int kind = bc.kind[a][side[a]];
    if (kind == FLUID_BC_PERIODIC || kind == FLUID_BC_ZERO_GRADIENT) continue;
    valued = true;
    int c[3];
    for (int b = 0; b < 3; ++b) c[b] = b < a ? own[b] : src[b];
    if (kind == FLUID_BC_INFLOW) {
      inflow_at(bc.inflow[a][side[a]], a, c, g, ph, w);
      continue;
    }
    double vw = 0.0;
    if (kind == FLUID_BC_POROUS) vw = bc.vw[c[bc.porous_t1]];
    wall_map(w, kind, bc.Tw[a][side[a]], vw, a, ph, &ctl->flags);
  }
  return valued;
}

// whether a halo axis of the cell changes values (a wall or inflow map) rather than only indices
__device__ __forceinline__ bool halo_valued(const bool ghost[3], const int side[3], const BC& bc) {
  bool valued = false;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int kind = bc.kind[a][side[a]];
    valued |= ghost[a] && kind != FLUID_BC_PERIODIC && kind != FLUID_BC_ZERO_GRADIENT;
  }
  return valued;
}

// halo_maps on the mixed path's pairs: the value maps run in FP64
__device__ __forceinline__ void halo_maps_ff(const int own[3], const bool ghost[3], const int side[3],
                                             const int src[3], const Geo& g, const Phys& ph, const BC& bc,
                                             Ctl* ctl, ff w[NW]) {
  if (!halo_valued(ghost, side, bc)) return;
  double d[NW];
  for (int v = 0; v < NW; ++v) d[v] = ff_to_double(w[v]);
  halo_maps(own, ghost, side, src, g, ph, bc, ctl, d);
  for (int v = 0; v < NW; ++v) w[v] = ff_of(d[v]);
}

// One thread per padded cell: x from the thread index, y and z from the block index; interior cells
// from U, halo cells by the composed boundary maps.
//
// The halo passes x -> y -> z compose: the pass of axis a sees own indices on the axes before it
// and source indices on the axes after it, so a halo cell starts from the cell at the source index
// on every axis and then takes the maps of its halo axes in order (an inflow axis replaces the
// state by its profile).  Every cell therefore converts exactly one cell's U -- its own or its
// source -- and only wall halos run map arithmetic, so warps that straddle the x halo do not run
// the conversion twice.
// MIXED: the primitives are pairs of floats and go to W32 instead of W.
template <bool MIXED>
__device__ __forceinline__ void k_prim_bc_body(const double* __restrict__ U, double* __restrict__ W,
                          float* __restrict__ W32, const Geo& g, const Phys& ph, const BC& bc, Ctl* ctl,
    uint3 bid, uint3 gdim) {
  const int i = bid.x * blockDim.x + threadIdx.x;
  if (i >= g.p[0]) return;
  for (int k = bid.z; k < g.p[2]; k += gdim.z)
    for (int j = bid.y; j < g.p[1]; j += gdim.y) {
      const int own[3] = {i, j, k};
      const int cell = i + j * g.sy + k * g.sz;
      bool ghost[3];
      int side[3], src[3];
      const bool any = halo_source(own, g, bc, ghost, side, src);
      const int scell = any ? src[0] + src[1] * g.sy + src[2] * g.sz : cell;
      if (MIXED) {
        double u[5];
        for (int v = 0; v < 5; ++v) u[v] = U[v * g.ncell + scell];
        ff w[NW];
        prim_ff(u, ph, w);
        if (any) halo_maps_ff(own, ghost, side, src, g, ph, bc, ctl, w);
        for (int v = 0; v < NW; ++v) store_pair(W32, g.ncell, v, cell, w[v]);
      } else {
        double w[NW];
        prim_of(U, scell, g.ncell, ph, w);
        if (any) halo_maps(own, ghost, side, src, g, ph, bc, ctl, w);
        for (int v = 0; v < NW; ++v) W[v * g.ncell + cell] = w[v];
      }
    }
}

template <bool MIXED>
__global__ void k_prim_bc(const double* U, double* W,
                          float* W32, Geo g, Phys ph, BC bc, Ctl* ctl) {
  step_wait();
  k_prim_bc_body<MIXED>(U, W, W32, g, ph, bc, ctl, blockIdx, gridDim);
}

// ------------------------------------------------------------------------------------------------
// centre gradients G[c*3+b] = d u_c / d x_b, only where the cell is interior along b (the only
// places the face fluxes read it), for the cells the face stencils reach along the other axes:
//   order 4: ((f[-2] - f[+2]) + 8 (f[+1] - f[-1])) * (mc / 12)
//   order 6: (45 (f[+1] - f[-1]) - 9 (f[+2] - f[-2]) + (f[+3] - f[-3])) * (mc / 60)
// ------------------------------------------------------------------------------------------------
template <int ORDER>
__device__ __forceinline__ void k_grad_body(const double* __restrict__ W, double* __restrict__ G, Geo g,
    uint3 bid, uint3 gdim) {
  constexpr int M = ORDER / 2;
  int lo[3], ext[3];
  for (int a = 0; a < 3; ++a) {
    const int m = a < g.ndim ? M : 0;
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
    for (int b = 0; b < 3; ++b) {
      const bool inb = b < g.ndim && c[b] >= g.h[b] && c[b] < g.h[b] + g.n[b];
      const int s = b == 0 ? 1 : (b == 1 ? g.sy : g.sz);
      // the stencil's 1/12 (1/60) and the metric as one factor per axis
      const double cm = inb ? (ORDER == 4 ? kTwelfth : 1.0 / 60.0) * g.mc[b][c[b]] : 0.0;
      for (int comp = 0; comp < 3; ++comp) {
        double d = 0.0;
        if (inb) {
          const double* f = W + (1 + comp) * g.ncell + cell;
          // explicit fused multiply-adds: every kernel inlining this rounds alike
          if (ORDER == 4)
            d = fma(8.0, f[s] - f[-s], f[-2 * s] - f[2 * s]) * cm;
          else
            d = fma(45.0, f[s] - f[-s], fma(-9.0, f[2 * s] - f[-2 * s], f[3 * s] - f[-3 * s])) * cm;
        }
        G[(comp * 3 + b) * g.ncell + cell] = d;
      }
    }
  }
}

template <int ORDER>
__global__ void k_grad(const double* W, double* G, Geo g) {
  step_wait();
  k_grad_body<ORDER>(W, G, g, blockIdx, gridDim);
}

// ------------------------------------------------------------------------------------------------
// seams of the face kernels' segments (face_kernels.cuh, kernels_teno.cu)
// ------------------------------------------------------------------------------------------------
// The first cell a0 of every segment after the first: the same update as the face kernel that
// filled FB, from the two fluxes its neighbouring segments left there
template <int D>
__device__ __forceinline__ void k_face_seam_body(const double* __restrict__ FB, double* __restrict__ R, Geo g,
                            int seg,
    uint3 bid, uint3 gdim) {
  constexpr int A1 = (D == 0) ? 1 : 0;
  constexpr int A2 = (D == 2) ? 1 : 2;
  const int n1 = g.n[A1], n2 = g.n[A2], nd = g.n[D];
  const int nseg = (nd + seg - 1) / seg;
  const long long lines = (long long)n1 * n2;
  const long long total = lines * nseg;
  const int nc = g.ncell;
  for (long long t = lines + bid.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gdim.x * blockDim.x) {
    const int i1 = (int)(t % n1);
    const long long r = t / n1;
    const int i2 = (int)(r % n2);
    const int sg = (int)(r / n2);
    int c[3];
    c[A1] = i1 + g.h[A1];
    c[A2] = i2 + g.h[A2];
    c[D] = g.h[D] + sg * seg;
    const int cell = c[0] + c[1] * g.sy + c[2] * g.sz;
    const double id = g.idx[D][c[D]];
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      const double Fv = FB[v * total + t], Fpv = FB[(5 + v) * total + t];
      update_r<D>(R + v * nc + cell, Fv, Fpv, id);
    }
  }
}

template <int D>
__global__ void k_face_seam(const double* FB, double* R, Geo g, int seg) {
  step_wait();
  k_face_seam_body<D>(FB, R, g, seg, blockIdx, gridDim);
}

// ------------------------------------------------------------------------------------------------
// source, stage combination, dt
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ int interior_cell(int t, const Geo& g) {
  const int i = t % g.n[0];
  const int r = t / g.n[0];
  const int j = r % g.n[1];
  const int k = r / g.n[1];
  return (i + g.h[0]) + (j + g.h[1]) * g.sy + (k + g.h[2]) * g.sz;
}

// velocity component b of a cell: from the mixed path's pairs when given, else from W
__device__ __forceinline__ double velocity(const double* __restrict__ W, const float* __restrict__ W32, int nc, int b,
                                           int c) {
  return W32 ? ff_to_double(load_pair(W32, nc, 1 + b, c)) : W[(1 + b) * nc + c];
}

__global__ void k_source(double* R, const double* W, const float* W32, Geo g,
                         Phys ph) {
  step_wait();
  const int total = g.n[0] * g.n[1] * g.n[2];
  const int nc = g.ncell;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < total; t += gridDim.x * blockDim.x) {
    const int c = interior_cell(t, g);
    const double u = velocity(W, W32, nc, 0, c), v = velocity(W, W32, nc, 1, c), w = velocity(W, W32, nc, 2, c);
    R[nc + c] += ph.f[0];
    R[2 * nc + c] += ph.f[1];
    R[3 * nc + c] += ph.f[2];
    R[4 * nc + c] += fma(ph.f[0], u, fma(ph.f[1], v, ph.f[2] * w));
  }
}

// stage 1: Ud = Un + dt r; stage 2: Ud = 3/4 Un + 1/4 (Us + dt r); stage 3: Ud = 1/3 Un + 2/3 (Us + dt r)
__device__ __forceinline__ void k_stage_body(int stage, const double* Un, const double* Us, const double* __restrict__ R,
                        double* Ud, const double* __restrict__ W, const float* __restrict__ W32, const Geo& g,
                        const Phys& ph, Ctl* ctl, double t_end, double dt_arg,
    uint3 bid, uint3 gdim) {
  const double dt = dt_arg > 0.0 ? dt_arg : ctl->dt;
  if (stage == 3 && dt_arg <= 0.0 && bid.x == 0 && threadIdx.x == 0 && dt > 0.0) {
    const double tn = ctl->t + dt;
    ctl->t = (t_end > 0.0 && !(tn < t_end)) ? t_end : tn;
  }
  if (stage == 3 && !(dt > 0.0)) return;
  const int total = g.n[0] * g.n[1] * g.n[2];
  const int nc = g.ncell;
  bool bad = false;
  for (int t = bid.x * blockDim.x + threadIdx.x; t < total; t += gdim.x * blockDim.x) {
    const int c = interior_cell(t, g);
    double r[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) r[v] = R[v * nc + c];
    if (ph.has_force) {
      const double u = velocity(W, W32, nc, 0, c), v = velocity(W, W32, nc, 1, c), w = velocity(W, W32, nc, 2, c);
      r[1] += ph.f[0];
      r[2] += ph.f[1];
      r[3] += ph.f[2];
      r[4] += fma(ph.f[0], u, fma(ph.f[1], v, ph.f[2] * w));
    }
    double un[5], us[5], out[5];
#pragma unroll
    for (int v = 0; v < 5; ++v) un[v] = Un[v * nc + c];
    if (stage != 1) {
#pragma unroll
      for (int v = 0; v < 5; ++v) us[v] = Us[v * nc + c];
    }
    stage_combine(stage, dt, un, us, r, out);
#pragma unroll
    for (int v = 0; v < 5; ++v) {
      bad |= !finite_bits(out[v]);
      Ud[v * nc + c] = out[v];
    }
  }
  if (bad) atomicOr(&ctl->flags, FLAG_NONFINITE);
}

__global__ void k_stage(int stage, const double* Un, const double* Us, const double* R,
                        double* Ud, const double* W, const float* W32, Geo g, Phys ph,
                        Ctl* ctl, double t_end, double dt_arg) {
  step_wait();
  k_stage_body(stage, Un, Us, R, Ud, W, W32, g, ph, ctl, t_end, dt_arg, blockIdx, gridDim);
}

// One RK3 stage fused with the primitives of its result (the next right-hand side's first pass):
// interior cell c gets Ud = the stage combination of k_stage, and W (for MIXED: W32) from Ud by the same
// conversion k_prim_bc applies, so the halo cells (k_halo_prim, next) and
// the following kernels see exactly what k_prim_bc would have produced.  W is read (body-force
// velocities of the stage's input state) and rewritten only at the thread's own cell.  A third
// stage with dt <= 0 leaves Un unwritten and converts it as it is.
template <bool MIXED>
__device__ __forceinline__ void k_stage_prim_body(int stage, const double* Un, const double* Us, const double* __restrict__ R,
                             double* Ud, double* W, float* __restrict__ W32, Geo g, Phys ph, Ctl* ctl,
                             double t_end,
    uint3 bid, uint3 gdim) {
  const double dt = ctl->dt;
  const bool hold = stage == 3 && !(dt > 0.0);
  if (stage == 3 && !hold && bid.x == 0 && bid.y == 0 && bid.z == 0 && threadIdx.x == 0) {
    const double tn = ctl->t + dt;
    ctl->t = (t_end > 0.0 && !(tn < t_end)) ? t_end : tn;
  }
  const int i = bid.x * blockDim.x + threadIdx.x;
  if (i >= g.n[0]) return;
  const int nc = g.ncell;
  // two cells per thread, rows j and j + J2, with every load of both issued before any store, so
  // that the two conversions' FP64 chains overlap
  const int J2 = (g.n[1] + 1) >> 1;
  bool bad = false;
  for (int k = bid.z; k < g.n[2]; k += gdim.z)
    for (int j = bid.y; j < J2; j += gdim.y) {
      const int base = (i + g.h[0]) + (k + g.h[2]) * g.sz;
      const bool two = j + J2 < g.n[1];
      const int c[2] = {base + (j + g.h[1]) * g.sy, base + (j + J2 + g.h[1]) * g.sy};
      double un[2][5], rs[2][5], us[2][5], vel[2][3];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (q == 1 && !two) break;
#pragma unroll
        for (int v = 0; v < 5; ++v) un[q][v] = Un[v * nc + c[q]];
        if (!hold) {
#pragma unroll
          for (int v = 0; v < 5; ++v) rs[q][v] = R[v * nc + c[q]];
          if (stage != 1) {
#pragma unroll
            for (int v = 0; v < 5; ++v) us[q][v] = Us[v * nc + c[q]];
          }
          if (ph.has_force) {
#pragma unroll
            for (int b = 0; b < 3; ++b) vel[q][b] = velocity(W, MIXED ? W32 : nullptr, nc, b, c[q]);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (q == 1 && !two) break;
        double u[5];
        if (hold) {
#pragma unroll
          for (int v = 0; v < 5; ++v) u[v] = un[q][v];
        } else {
          double* r = rs[q];
          if (ph.has_force) {
            r[1] += ph.f[0];
            r[2] += ph.f[1];
            r[3] += ph.f[2];
            r[4] += fma(ph.f[0], vel[q][0], fma(ph.f[1], vel[q][1], ph.f[2] * vel[q][2]));
          }
          stage_combine(stage, dt, un[q], us[q], r, u);
#pragma unroll
          for (int v = 0; v < 5; ++v) {
            bad |= !finite_bits(u[v]);
            Ud[v * nc + c[q]] = u[v];
          }
        }
        if (MIXED) {
          ff w[NW];
          prim_ff(u, ph, w);
#pragma unroll
          for (int v = 0; v < NW; ++v) store_pair(W32, nc, v, c[q], w[v]);
        } else {
          double w[NW];
          prim_from_cons(u, ph, w);
#pragma unroll
          for (int v = 0; v < NW; ++v) W[v * nc + c[q]] = w[v];
        }
      }
    }
  if (bad) atomicOr(&ctl->flags, FLAG_NONFINITE);
}

template <bool MIXED>
__global__ void k_stage_prim(int stage, const double* Un, const double* Us, const double* R,
                             double* Ud, double* W, float* W32, Geo g, Phys ph, Ctl* ctl,
                             double t_end) {
  step_wait();
  k_stage_prim_body<MIXED>(stage, Un, Us, R, Ud, W, W32, g, ph, ctl, t_end, blockIdx, gridDim);
}

// Halo cells only, from the interior primitives already in W: the maps of k_prim_bc applied to the
// source cell's primitives.  Cells are enumerated by their highest halo axis a: axes above a
// interior, axis a one of its 2 h[a] halo layers, axes below a anywhere in the padded range.
template <bool MIXED>
__device__ __forceinline__ void k_halo_prim_body(double* __restrict__ W, float* __restrict__ W32, Geo g, Phys ph, BC bc,
                            Ctl* ctl, long long total,
    uint3 bid, uint3 gdim) {
  const int nc = g.ncell;
  for (long long t0 = bid.x * (long long)blockDim.x + threadIdx.x; t0 < total;
       t0 += (long long)gdim.x * blockDim.x) {
    long long t = t0;
    int own[3] = {0, 0, 0};
    for (int a = 2; a >= 0; --a) {
      long long cnt = 2LL * g.h[a];
      for (int b = 0; b < 3; ++b)
        if (b != a) cnt *= b < a ? g.p[b] : g.n[b];
      if (t >= cnt) {
        t -= cnt;
        continue;
      }
      for (int b = 0; b < a; ++b) {
        own[b] = (int)(t % g.p[b]);
        t /= g.p[b];
      }
      const int l = (int)(t % (2 * g.h[a]));
      t /= 2 * g.h[a];
      own[a] = l < g.h[a] ? l : g.n[a] + l;
      for (int b = a + 1; b < 3; ++b) {
        own[b] = g.h[b] + (int)(t % g.n[b]);
        t /= g.n[b];
      }
      break;
    }
    bool ghost[3];
    int side[3], src[3];
    halo_source(own, g, bc, ghost, side, src);
    const int scell = src[0] + src[1] * g.sy + src[2] * g.sz;
    const int cell = own[0] + own[1] * g.sy + own[2] * g.sz;
    if (MIXED) {
      ff w[NW];
#pragma unroll
      for (int v = 0; v < NW; ++v) w[v] = load_pair(W32, nc, v, scell);
      halo_maps_ff(own, ghost, side, src, g, ph, bc, ctl, w);
#pragma unroll
      for (int v = 0; v < NW; ++v) store_pair(W32, nc, v, cell, w[v]);
    } else {
      double w[NW];
#pragma unroll
      for (int v = 0; v < NW; ++v) w[v] = W[v * nc + scell];
      halo_maps(own, ghost, side, src, g, ph, bc, ctl, w);
#pragma unroll
      for (int v = 0; v < NW; ++v) W[v * nc + cell] = w[v];
    }
  }
}

template <bool MIXED>
__global__ void k_halo_prim(double* W, float* W32, Geo g, Phys ph, BC bc,
                            Ctl* ctl, long long total) {
  step_wait();
  k_halo_prim_body<MIXED>(W, W32, g, ph, bc, ctl, total, blockIdx, gridDim);
}


// CFL: dt = cfl * min over cells and axes of dx / (|u| + c) and dx^2 / (k nu), taken as
// cfl / max of the rates (|u| + c) / dx and k nu / dx^2 so that a cell costs no division.
__device__ __forceinline__ double cell_rate(const double* __restrict__ W, const Geo& g, const Phys& ph, int t) {
  const int i = t % g.n[0];
  const int r = t / g.n[0];
  const int j = r % g.n[1];
  const int k = r / g.n[1];
  const int ci[3] = {i + g.h[0], j + g.h[1], k + g.h[2]};
  const int c = ci[0] + ci[1] * g.sy + ci[2] * g.sz, nc = g.ncell;
  const double rho = W[c], p = W[4 * nc + c];
  const double irho = fl_rcp(rho);
  const double cs = fl_sqrt(ph.gamma * p * irho);
  double knu = 0.0, best = 0.0;
  if (ph.visc != FLUID_VISC_NONE) knu = ph.dt_visc_k * viscosity(W[5 * nc + c], ph) * irho;
  for (int d = 0; d < g.ndim; ++d) {
    const double id = g.idx[d][ci[d]];
    best = fmax(best, (fabs(W[(1 + d) * nc + c]) + cs) * id);
    if (ph.visc != FLUID_VISC_NONE) best = fmax(best, knu * id * id);
  }
  return best;
}

// The same in FP32, within 1e-4 of it (the power law's estimate is its least exact part); infinite
// where a value leaves [1e-30, 1e30] or the square of the sound speed [1e-37, 1e37] (an infinity or a
// zero there would become a NaN, which fmaxf drops)
__device__ __forceinline__ float cell_rate32(const double* __restrict__ W, const Geo& g, const Phys& ph, int t) {
  const int i = t % g.n[0];
  const int r = t / g.n[0];
  const int j = r % g.n[1];
  const int k = r / g.n[1];
  const int ci[3] = {i + g.h[0], j + g.h[1], k + g.h[2]};
  const int c = ci[0] + ci[1] * g.sy + ci[2] * g.sz, nc = g.ncell;
  const float rho = ff_of(W[c]).h, p = ff_of(W[4 * nc + c]).h;
  bool ok = rho >= 1e-30f && rho <= 1e30f && p >= 1e-30f && p <= 1e30f;
  const float irho = s_rcp(rho), c2 = ph.k.gamma.h * (p * irho);
  ok = ok && c2 >= 1e-37f && c2 <= 1e37f;
  const float cs = c2 * s_rsqrt(c2);
  float knu = 0.0f, best = 0.0f;
  if (ph.visc != FLUID_VISC_NONE) {
    const float T = ff_of(W[5 * nc + c]).h, x = T * ph.k.iT_ref.h;
    ok = ok && x >= 1e-30f && x <= 1e30f;
    float mu = ph.k.mu_ref.h;
    if (ph.visc == FLUID_VISC_POWER) mu *= __powf(x, ph.visc_e32);
    else if (ph.visc == FLUID_VISC_SUTHERLAND) mu = ph.k.mu_TS.h * (x * x) * s_rsqrt(x) * s_rcp(T + ph.k.suth_S.h);
    knu = ph.k.dt_visc.h * mu * irho;
  }
  for (int d = 0; d < g.ndim; ++d) {
    const float id = ff_of(g.idx[d][ci[d]]).h, u = fabsf(ff_of(W[(1 + d) * nc + c]).h);
    ok = ok && u <= 1e30f;
    best = fmaxf(best, fmaxf((u + cs) * id, knu * id * id));
  }
  return ok && best <= 1e36f ? best : __int_as_float(0x7f800000);
}

// Per-block maxima of the rate go to `partial`; the last block to finish reduces them and stores dt (no
// second launch).  nparts 0: a fixed dt, one block.  The ticket wraps to 0 at the last block, so nothing has
// to reset it for the next call.
// The FP64 rates bind (about 60 FP64-pipe instructions per cell), so a block first finds its largest
// FP32 rate and forms in FP64 only the cells within 1e-3 of it: the maximum is among them, bit
// for bit (TGV 128^3: 228 us with every cell in FP64 and the second launch).
__device__ __forceinline__ void k_dt_body(const double* __restrict__ W, const Geo& g, const Phys& ph, double* partial,
                                          int nparts, Ctl* ctl, double* dt_out, int clip, double t_end, uint3 bid,
                                          uint3 gdim) {
  __shared__ double sm[kDtBlock / 32];
  __shared__ unsigned last;
  double best = 0.0;
  if (nparts > 0) {
    const int total = g.n[0] * g.n[1] * g.n[2];
    const int t0 = bid.x * blockDim.x + threadIdx.x, stride = gdim.x * blockDim.x;
    float mine = 0.0f;
    for (int t = t0; t < total; t += stride) mine = fmaxf(mine, cell_rate32(W, g, ph, t));
    const float limit = block_max(mine, reinterpret_cast<float*>(sm)) * 0.999f;
    // an infinite limit: some value is outside the FP32 range, so every cell is formed in FP64
    const bool all = !(limit <= 1e36f);
    if (all || mine >= limit)
      for (int t = t0; t < total; t += stride)
        if (all || cell_rate32(W, g, ph, t) >= limit) best = fmax(best, cell_rate(W, g, ph, t));
    best = block_max(best, sm);
    if (threadIdx.x == 0) {
      __stcg(partial + bid.x, best);
      __threadfence();
      last = atomicInc(&ctl->ticket, nparts - 1) == (unsigned)(nparts - 1);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    best = 0.0;
    for (int i = threadIdx.x; i < nparts; i += blockDim.x) best = fmax(best, __ldcg(partial + i));
    best = block_max(best, sm);
  }
  if (threadIdx.x == 0) dt_store(best, ph, ctl, dt_out, clip, t_end);
}

__global__ void __launch_bounds__(kDtBlock) k_dt(const double* W, const __grid_constant__ Geo g,
                                                 const __grid_constant__ Phys ph, double* partial, int nparts,
                                                 Ctl* ctl, double* dt_out, int clip, double t_end) {
  step_wait();
  k_dt_body(W, g, ph, partial, nparts, ctl, dt_out, clip, t_end, blockIdx, gridDim);
}

// Halo exchange of a block decomposition: element t of the buffer [5][3][e2][e1] (t1 < t2 the axes
// other than A; e_b = p_b below A, n_b above A, starting at 0 resp. h_b) and the padded cell it
// maps to: layer l of face (A, side) is h + l / n + l (interior layers, packed) or l / h + n + l
// (halo layers, unpacked).
__global__ void k_halo_copy(double* __restrict__ U, double* __restrict__ buf, Geo g, int A,
                            int side, int unpack, long long total) {
  const int t1 = A == 0 ? 1 : 0, t2 = A == 2 ? 1 : 2;
  const int e1 = t1 < A ? g.p[t1] : g.n[t1], o1 = t1 < A ? 0 : g.h[t1];
  const int e2 = t2 < A ? g.p[t2] : g.n[t2], o2 = t2 < A ? 0 : g.h[t2];
  const int h = g.h[A], n = g.n[A];
  const int l0 = unpack ? (side == 0 ? 0 : h + n) : (side == 0 ? h : n);
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    long long r = t;
    const int i1 = (int)(r % e1);
    r /= e1;
    const int i2 = (int)(r % e2);
    r /= e2;
    const int l = (int)(r % 3);
    const int v = (int)(r / 3);
    int c[3];
    c[A] = l0 + l;
    c[t1] = o1 + i1;
    c[t2] = o2 + i2;
    const long long cell = (long long)v * g.ncell + c[0] + (long long)c[1] * g.sy + (long long)c[2] * g.sz;
    if (unpack) U[cell] = buf[t];
    else buf[t] = U[cell];
  }
}

__global__ void k_prim_to_cons(const double* W, double* U, int nc, Phys ph) {
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < nc; c += gridDim.x * blockDim.x) {
    const double r = W[c], u = W[nc + c], v = W[2 * nc + c], w = W[3 * nc + c], p = W[4 * nc + c];
    const double E = p * ph.igm1 + 0.5 * r * (u * u + v * v + w * w);
    U[c] = r;
    U[nc + c] = r * u;
    U[2 * nc + c] = r * v;
    U[3 * nc + c] = r * w;
    U[4 * nc + c] = E;
  }
}

__global__ void k_wall_velocity(const double* __restrict__ phi, double* __restrict__ vw,
                                const double* __restrict__ xc, int p, int h, int begin, int count,
                                double amp, double two_pi_kappa) {
  for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < p; a += gridDim.x * blockDim.x) {
    const int i = a - h - begin;
    vw[a] = (i >= 0 && i < count) ? amp * phi[i] * sin(two_pi_kappa * xc[a]) : 0.0;
  }
}

// ------------------------------------------------------------------------------------------------
// batched kernels of the serving loop (see BatchTable): each block walks virtual blocks of all the
// bucket's solves and runs the standalone body with the solve's data, block index and grid size
// ------------------------------------------------------------------------------------------------
template <bool MIXED>
__global__ void __launch_bounds__(128) kb_prim(const BatchTable* __restrict__ t) {
  FL_BATCH_LOOP(BK_PRIM)
  if (S.steps > 0) k_prim_bc_body<MIXED>(S.U, S.W, S.W32, S.g, S.ph, S.bc, S.ctl, bid, gdim);
  FL_BATCH_END
}

__global__ void __launch_bounds__(kDtBlock) kb_dt(const BatchTable* __restrict__ t, int step) {
  FL_BATCH_LOOP(BK_DT)
  if (step < S.steps)
    k_dt_body(S.W, S.g, S.ph, S.partial, S.nparts, S.ctl, nullptr, 1, S.t_end, bid, gdim);
  FL_BATCH_END
}

__global__ void __launch_bounds__(256) kb_grad(const BatchTable* __restrict__ t, int step) {
  FL_BATCH_LOOP(BK_GRAD)
  if (step < S.steps) k_grad_body<4>(S.W, S.G, S.g, bid, gdim);
  FL_BATCH_END
}

template <bool MIXED>
__global__ void __launch_bounds__(128) kb_stage_prim(const BatchTable* __restrict__ t, int stage, int step) {
  FL_BATCH_LOOP(BK_STAGEP)
  if (step < S.steps)
    k_stage_prim_body<MIXED>(stage, S.U, stage == 1 ? S.U : S.A, S.R, stage == 3 ? S.U : S.A, S.W,
                             S.W32, S.g, S.ph, S.ctl, S.t_end, bid, gdim);
  FL_BATCH_END
}

template <bool MIXED>
__global__ void __launch_bounds__(256) kb_halo(const BatchTable* __restrict__ t, int step) {
  FL_BATCH_LOOP(BK_HALO)
  if (step < S.steps) {
    const long long total = (long long)S.g.p[0] * S.g.p[1] * S.g.p[2] -
                            (long long)S.g.n[0] * S.g.n[1] * S.g.n[2];
    k_halo_prim_body<MIXED>(S.W, S.W32, S.g, S.ph, S.bc, S.ctl, total, bid, gdim);
  }
  FL_BATCH_END
}

__global__ void __launch_bounds__(256) kb_stage(const BatchTable* __restrict__ t, int step) {
  FL_BATCH_LOOP(BK_STAGE)
  if (step < S.steps) k_stage_body(3, S.U, S.A, S.R, S.U, S.W, S.W32, S.g, S.ph, S.ctl, S.t_end, 0.0, bid, gdim);
  FL_BATCH_END
}

cudaError_t launch_batch_faces(const BatchTable* dev, int step, int weno, bool visc,
                               cudaStream_t st) {
  for (int D = 0; D < 3; ++D) {
    const cudaError_t e = weno == FLUID_WENO_JS ? launch_batch_face_js(dev, D, step, visc, st)
                                                : launch_batch_face_z(dev, D, step, visc, st);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace

void batch_plan(BatchTable& t) {
  auto ceil_div = [](long long a, long long b) { return (a + b - 1) / b; };
  for (int k = 0; k < BK_COUNT; ++k) t.prefix[k][0] = 0;
  for (int i = 0; i < t.nslots; ++i) {
    BatchSlot& S = t.slot[i];
    const Geo& g = S.g;
    for (int k = 0; k < BK_COUNT; ++k) S.vgrid[k][0] = S.vgrid[k][1] = S.vgrid[k][2] = 1;
    auto set = [&](int k, long long x, long long y = 1, long long z = 1) {
      S.vgrid[k][0] = (int)x;
      S.vgrid[k][1] = (int)y;
      S.vgrid[k][2] = (int)z;
    };
    const long long nint = (long long)g.n[0] * g.n[1] * g.n[2];
    const long long npad = (long long)g.p[0] * g.p[1] * g.p[2];
    set(BK_PRIM, ceil_div(g.p[0], 128), std::min(g.p[1], 65535), std::min(g.p[2], 65535));
    set(BK_DT, S.nparts > 0 ? S.nparts : 1);
    const bool visc = S.ph.visc != FLUID_VISC_NONE;
    long long gt = 1;
    for (int a = 0; a < 3; ++a) gt *= g.n[a] + (a < g.ndim ? 4 : 0);   // order-4 stencils, both paths
    set(BK_GRAD, visc ? ceil_div(gt, 256) : 0);
    for (int D = 0; D < 3; ++D) {
      if (D >= g.ndim) set(BK_FACE0 + D, 0);
      else if (D == 0) set(BK_FACE0, tile_cols<0>(g), tile_rows<0>(g));
      else if (D == 1) set(BK_FACE1, tile_cols<1>(g), tile_rows<1>(g));
      else set(BK_FACE2, tile_cols<2>(g), tile_rows<2>(g));
    }
    set(BK_STAGEP, ceil_div(g.n[0], 128), std::min((g.n[1] + 1) / 2, 65535), std::min(g.n[2], 65535));
    set(BK_HALO, ceil_div(npad - nint, 256));
    set(BK_STAGE, ceil_div(nint, 256));
    for (int k = 0; k < BK_COUNT; ++k)
      t.prefix[k][i + 1] = t.prefix[k][i] + (long long)S.vgrid[k][0] * S.vgrid[k][1] * S.vgrid[k][2];
  }
}

cudaError_t launch_batch_chunk(const BatchTable* dev, int chunk, bool mixed, int weno, bool visc,
                               cudaStream_t st) {
  static const int gp = batch_grid(kb_prim<false>, 128), gpm = batch_grid(kb_prim<true>, 128);
  static const int gd = batch_grid(kb_dt, kDtBlock);
  static const int gg = batch_grid(kb_grad, 256);
  static const int gsp = batch_grid(kb_stage_prim<false>, 128), gspm = batch_grid(kb_stage_prim<true>, 128);
  static const int gh = batch_grid(kb_halo<false>, 256), ghm = batch_grid(kb_halo<true>, 256);
  static const int gs = batch_grid(kb_stage, 256);
  cudaError_t e;
  if (mixed) (kb_prim<true><<<gpm, 128, 0, st>>>(dev), ++t_launches);
  else (kb_prim<false><<<gp, 128, 0, st>>>(dev), ++t_launches);
  for (int k = 0; k < chunk; ++k) {
    if (mixed) {
      if ((e = launch_batch_mixed(dev, BMX_DT, k, st)) != cudaSuccess) return e;
    } else {
      (kb_dt<<<gd, kDtBlock, 0, st>>>(dev, k), ++t_launches);
    }
    for (int stage = 1; stage <= 3; ++stage) {
      if (mixed) {
        if (visc && (e = launch_batch_mixed(dev, BMX_GRAD, k, st)) != cudaSuccess) return e;
        for (int D = 0; D < 3; ++D)
          if ((e = launch_batch_mixed_faces(dev, D, k, weno, visc, st)) != cudaSuccess) return e;
      } else {
        if (visc) (kb_grad<<<gg, 256, 0, st>>>(dev, k), ++t_launches);
        if ((e = launch_batch_faces(dev, k, weno, visc, st)) != cudaSuccess) return e;
      }
      if (stage < 3 || k + 1 < chunk) {
        if (mixed) {
          (kb_stage_prim<true><<<gspm, 128, 0, st>>>(dev, stage, k), ++t_launches);
          (kb_halo<true><<<ghm, 256, 0, st>>>(dev, k), ++t_launches);
        } else {
          (kb_stage_prim<false><<<gsp, 128, 0, st>>>(dev, stage, k), ++t_launches);
          (kb_halo<false><<<gh, 256, 0, st>>>(dev, k), ++t_launches);
        }
      } else {
        (kb_stage<<<gs, 256, 0, st>>>(dev, k), ++t_launches);
      }
    }
  }
  return cudaGetLastError();
}

double* seam_buffer(int D, const Geo& g, int seg, SeamBuf fb) {
  const long long lines = (long long)g.n[D == 0 ? 1 : 0] * g.n[D == 2 ? 1 : 2];
  const long long nseg = (g.n[D] + seg - 1) / seg;
  return (fb.p != nullptr && nseg > 1 && lines * nseg <= fb.cap) ? fb.p : nullptr;
}

cudaError_t launch_face_seam(int D, const double* FB, double* R, const Geo& g, int seg, cudaStream_t st) {
  const long long lines = (long long)g.n[D == 0 ? 1 : 0] * g.n[D == 2 ? 1 : 2];
  const long long items = lines * ((g.n[D] + seg - 1) / seg - 1);
  const int grid = grid_for(items, 256);
  if (D == 0) launch_step(k_face_seam<0>, grid, 256, 0, st, FB, R, g, seg);
  else if (D == 1) launch_step(k_face_seam<1>, grid, 256, 0, st, FB, R, g, seg);
  else launch_step(k_face_seam<2>, grid, 256, 0, st, FB, R, g, seg);
  return cudaGetLastError();
}

int face_grid(int D, const Geo& g, int block, int seg) {
  const long long lines = (long long)g.n[D == 0 ? 1 : 0] * g.n[D == 2 ? 1 : 2];
  return grid_for(lines * ((g.n[D] + seg - 1) / seg), block);
}

cudaError_t launch_prim_bc(const double* U, double* W, float* W32, const Geo& g, const Phys& ph,
                           const BC& bc, Ctl* ctl, cudaStream_t st) {
  // a padded row in nb near-equal chunks of whole warps, at most 256 threads each
  const int nb = (g.p[0] + 255) / 256;
  const int block = ((g.p[0] + nb - 1) / nb + 31) / 32 * 32;
  const dim3 grid((g.p[0] + block - 1) / block, g.p[1] < 65535 ? g.p[1] : 65535,
                  g.p[2] < 65535 ? g.p[2] : 65535);
  if (W32) launch_step(k_prim_bc<true>, grid, block, 0, st, U, W, W32, g, ph, bc, ctl);
  else launch_step(k_prim_bc<false>, grid, block, 0, st, U, W, W32, g, ph, bc, ctl);
  return cudaGetLastError();
}

cudaError_t launch_grad(const double* W, double* G, const Geo& g, const Phys& ph, cudaStream_t st) {
  const int m = ph.visc_order == 6 ? 3 : 2;
  long long total = 1;
  for (int a = 0; a < 3; ++a) total *= g.n[a] + (a < g.ndim ? 2 * m : 0);
  if (m == 3) launch_step(k_grad<6>, grid_for(total, 256), 256, 0, st, W, G, g);
  else launch_step(k_grad<4>, grid_for(total, 256), 256, 0, st, W, G, g);
  return cudaGetLastError();
}

cudaError_t launch_face(int D, const double* W, const double* G, double* R, const Geo& g,
                        const Phys& ph, int block, int seg, SeamBuf fb, cudaStream_t st) {
  if (ph.weno == FLUID_TENO6A) return launch_face_teno(D, W, G, R, g, ph, st);
  if (ph.weno == FLUID_WENO_JS) return launch_face_js(D, W, G, R, g, ph, block, seg, fb, st);
  return launch_face_z(D, W, G, R, g, ph, block, seg, fb, st);
}

long long seam_capacity(const Geo& g) {
  long long cap = 0;
  for (int D = 0; D < g.ndim; ++D) {
    const long long lines = (long long)g.n[D == 0 ? 1 : 0] * g.n[D == 2 ? 1 : 2];
    const long long items = lines * ((g.n[D] + kSeamMinSeg - 1) / kSeamMinSeg);
    if (items > cap) cap = items;
  }
  return cap;
}

cudaError_t launch_source(double* R, const double* W, const float* W32, const Geo& g, const Phys& ph,
                          cudaStream_t st) {
  const long long total = (long long)g.n[0] * g.n[1] * g.n[2];
  launch_step(k_source, grid_for(total, 256), 256, 0, st, R, W, W32, g, ph);
  return cudaGetLastError();
}

cudaError_t launch_stage(int stage, const double* Un, const double* Us, const double* R, double* Ud,
                         const double* W, const float* W32, const Geo& g, const Phys& ph, Ctl* ctl,
                         double t_end, cudaStream_t st, double dt_arg) {
  const long long total = (long long)g.n[0] * g.n[1] * g.n[2];
  launch_step(k_stage, grid_for(total, 256), 256, 0, st, stage, Un, Us, R, Ud, W, W32, g, ph, ctl, t_end, dt_arg);
  return cudaGetLastError();
}

cudaError_t launch_stage_prim(int stage, const double* Un, const double* Us, const double* R,
                              double* Ud, double* W, float* W32, const Geo& g, const Phys& ph,
                              const BC& bc, Ctl* ctl, double t_end, cudaStream_t st) {
  // interior rows in nb near-equal chunks of whole warps, at most 256 threads each
  const int nb = (g.n[0] + 255) / 256;
  const int block = ((g.n[0] + nb - 1) / nb + 31) / 32 * 32;
  const int j2 = (g.n[1] + 1) / 2;                                     // row pairs
  const dim3 grid((g.n[0] + block - 1) / block, j2 < 65535 ? j2 : 65535, g.n[2] < 65535 ? g.n[2] : 65535);
  if (W32) launch_step(k_stage_prim<true>, grid, block, 0, st, stage, Un, Us, R, Ud, W, W32, g, ph, ctl, t_end);
  else launch_step(k_stage_prim<false>, grid, block, 0, st, stage, Un, Us, R, Ud, W, W32, g, ph, ctl, t_end);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_halo_prim(W, W32, g, ph, bc, ctl, st);
}

cudaError_t launch_halo_prim(double* W, float* W32, const Geo& g, const Phys& ph, const BC& bc, Ctl* ctl,
                             cudaStream_t st) {
  const long long total = (long long)g.p[0] * g.p[1] * g.p[2] - (long long)g.n[0] * g.n[1] * g.n[2];
  if (total <= 0) return cudaSuccess;
  if (W32) launch_step(k_halo_prim<true>, grid_for(total, 256), 256, 0, st, W, W32, g, ph, bc, ctl, total);
  else launch_step(k_halo_prim<false>, grid_for(total, 256), 256, 0, st, W, W32, g, ph, bc, ctl, total);
  return cudaGetLastError();
}

size_t halo_count(const Geo& g, int A) {
  size_t cnt = 5 * 3;
  for (int b = 0; b < 3; ++b)
    if (b != A) cnt *= (size_t)(b < A ? g.p[b] : g.n[b]);
  return cnt;
}

cudaError_t launch_halo_copy(double* U, double* buf, const Geo& g, int A, int side, bool unpack,
                             cudaStream_t st) {
  const long long total = (long long)halo_count(g, A);
  (k_halo_copy<<<grid_for(total, 256), 256, 0, st>>>(U, buf, g, A, side, unpack ? 1 : 0, total),
   ++t_launches);
  return cudaGetLastError();
}

int dt_partial_count(const Geo& g) {
  const long long total = (long long)g.n[0] * g.n[1] * g.n[2];
  long long b = (total + kDtBlock - 1) / kDtBlock;
  if (b > 152 * 8) b = 152 * 8;
  return (int)(b < 1 ? 1 : b);
}

cudaError_t launch_dt(const double* W, const Geo& g, const Phys& ph, double* partial, int nparts, Ctl* ctl,
                      double* dt_out, int clip_to_ctl, double t_end, cudaStream_t st) {
  const int n = ph.dt_fixed > 0.0 ? 0 : nparts;
  launch_step(k_dt, n > 0 ? n : 1, kDtBlock, 0, st, W, g, ph, partial, n, ctl, dt_out, clip_to_ctl, t_end);
  return cudaGetLastError();
}

cudaError_t launch_prim_to_cons(const double* W, double* U, int ncell, const Phys& ph,
                                cudaStream_t st) {
  (k_prim_to_cons<<<grid_for(ncell, 256), 256, 0, st>>>(W, U, ncell, ph), ++t_launches);
  return cudaGetLastError();
}

cudaError_t launch_wall_velocity(const double* phi, double* vw, const double* xc, int p, int h,
                                 int begin, int count, double amp, double two_pi_kappa,
                                 cudaStream_t st) {
  (k_wall_velocity<<<grid_for(p, 128), 128, 0, st>>>(phi, vw, xc, p, h, begin, count, amp,
                                                    two_pi_kappa), ++t_launches);
  return cudaGetLastError();
}

}  // namespace fl
