// Internal definitions shared by the solver's CUDA translation units (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/fluid.h"
#include "ff_math.cuh"

struct fluid_solver;

namespace fl {

constexpr int NV = 5;   // conservative variables (rho, rho u, rho v, rho w, E)
constexpr int NW = 6;   // primitive scratch (rho, u, v, w, p, T)
constexpr int NG = 9;   // velocity-gradient scratch, component c * 3 + b = d u_c / d x_b

// flag bits of Ctl::flags
constexpr unsigned FLAG_NONFINITE = 1u;
constexpr unsigned FLAG_GHOST_T = 2u;
constexpr unsigned FLAG_STAGING = 4u;   // the bulk-copy check's wait ran out (k_bulk_probe; never in Ctl::flags)

// Grid geometry: padded sizes, strides and per-axis 1-D metric arrays (device, length p[a]).
struct Geo {
  int ndim;
  int n[3], h[3], p[3];
  int sy, sz;      // strides (cells) of y and z; x stride is 1
  int ncell;       // p0 p1 p2: stride between variables
  const double* xc[3];   // cell centres
  const double* dx[3];   // cell widths
  const double* idx[3];  // 1 / widths
  const double* mc[3];   // d(index)/dx at centres
  const double* mf[3];   // d(index)/dx at face a+1/2
  const float* mf32[3];  // FP32 copy of mf (mixed path only, else null)
  const float* mc32[3];  // FP32 copy of mc (mixed path only, else null)
  const float* idx32[3]; // FP32 copy of idx (mixed path only, else null)
};

// The constants that the two-float terms of the FP64 face kernels use (set_ff)
struct PhysFF {
  ff gamma, gm1, igm1, gg, iR, eps4, mu_ref, mu_TS, iT_ref, suth_S, lam_fac, dt_visc, visc_exp, re;   // gg = gamma / (gamma - 1), mu_TS = mu_ref (T_ref + S), re = 2 sqrt(eps)
};

struct Phys {
  double gamma, gm1, igm1, R, iR, cp, Pr, lam_fac;
  double mu_ref, T_ref, iT_ref, visc_exp, suth_S;
  int visc_p, visc_q;  // power law: visc_exp = visc_p / visc_q (small integers), else visc_q = 0
  float visc_e32;      // visc_exp in FP32
  int visc_hw_lo, visc_hw_hi;   // high-word bounds of the fast range of fl_pow_rational
  int visc, weno;
  int visc_order;     // central differences of the dissipative fluxes: 4 or 6
  double eps;
  double f[3];
  int has_force;
  double cfl, dt_fixed, dt_visc_k;
  PhysFF k;         // two-float copies
};

struct BC {
  int kind[3][2];
  double Tw[3][2];
  const double* inflow[3][2];   // primitive profile [5][T2][T1] (device) or null
  int porous_axis, porous_side, porous_t1;
  const double* vw;             // transpiration velocity per padded index of axis porous_t1
};

// Device-resident step control: solver time, last dt, sticky error flags.
struct Ctl {
  double t, dt;
  unsigned flags;
  unsigned ticket;     // blocks of the current CFL reduction that have finished
};

// a plain load, also in kernels that begin before the writer of *p has ended (launch_step)
template <class T>
__device__ __forceinline__ T ld(const T* p) {
  return *p;
}

__device__ __forceinline__ bool finite_bits(double x) {
  return ((__double2hiint(x) >> 20) & 0x7ff) != 0x7ff;
}

// Primitives of the mixed path: W32 = [2 NW][ncell] floats, rows v and NW + v the two floats of
// primitive v.
__device__ __forceinline__ ff load_pair(const float* __restrict__ W32, int nc, int v, int cell) {
  return ff{W32[v * nc + cell], W32[(NW + v) * nc + cell]};
}
__device__ __forceinline__ void store_pair(float* __restrict__ W32, int nc, int v, int cell, ff w) {
  W32[v * nc + cell] = w.h;
  W32[(NW + v) * nc + cell] = w.l;
}

// One RK3 stage: stage 1 Un + dt r; stage 2 3/4 Un + 1/4 (Us + dt r); stage 3 1/3 Un + 2/3 (Us + dt r).
// The last two share their operations with the factors chosen first (a choice between the formulas
// executes both).
__device__ __forceinline__ void stage_combine(int stage, double dt, const double un[5], const double us[5],
                                              const double r[5], double out[5]) {
  if (stage == 1) {
#pragma unroll
    for (int v = 0; v < 5; ++v) out[v] = fma(dt, r[v], un[v]);
  } else {
    const double c0 = stage == 2 ? 0.75 : 1.0 / 3.0, c1 = stage == 2 ? 0.25 : 2.0 / 3.0;
#pragma unroll
    for (int v = 0; v < 5; ++v) out[v] = fma(c0, un[v], __dmul_rn(c1, fma(dt, r[v], us[v])));
  }
}

constexpr int kDtBlock = 256;   // threads of a CFL block
template <class T>
__device__ __forceinline__ T block_max(T v, T* sm) {
  for (int o = 16; o > 0; o >>= 1) {
    const T w = __shfl_down_sync(0xffffffffu, v, o);
    v = v > w ? v : w;
  }
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  v = sm[0];
  for (int i = 1; i < kDtBlock / 32; ++i) v = v > sm[i] ? v : sm[i];
  return v;
}

// dt = cfl / max(partial rates) (or dt_fixed); clip: clip so that t does not pass t_end and
// store in ctl->dt; otherwise write *dt_out.
__device__ __forceinline__ void dt_store(double best, const Phys& ph, Ctl* ctl, double* dt_out, int clip,
                                         double t_end) {
  double dt = ph.dt_fixed > 0.0 ? ph.dt_fixed : ph.cfl / best;
  if (!clip) {
    *dt_out = dt;
    return;
  }
  if (t_end > 0.0) {
    if (ctl->t >= t_end) dt = 0.0;
    else if (ctl->t + dt > t_end) dt = t_end - ctl->t;
  }
  ctl->dt = dt;
}

__host__ __device__ __forceinline__ double viscosity(double T, const Phys& ph) {
  if (ph.visc == FLUID_VISC_CONSTANT) return ph.mu_ref;
  const double r = T * ph.iT_ref;
  if (ph.visc == FLUID_VISC_POWER) {
    if (ph.visc_q > 0)
      return ph.mu_ref * fl_pow_rational(r, ph.visc_p, ph.visc_q, ph.visc_e32, ph.visc_hw_lo, ph.visc_hw_hi);
    return ph.mu_ref * exp(ph.visc_exp * log(r));
  }
  // Sutherland
  return ph.mu_ref * (r * fl_sqrt(r)) * (ph.T_ref + ph.suth_S) * fl_rcp(T + ph.suth_S);
}

// d mu / d T of the same laws, given mu = viscosity(T, ph): power law e mu / T; Sutherland
// (mu = C r^{3/2} / (T + S), C = mu_ref (T_ref + S)) mu (1.5 / T - 1 / (T + S))
__host__ __device__ __forceinline__ double viscosity_dT(double T, double mu, const Phys& ph) {
  if (ph.visc == FLUID_VISC_CONSTANT) return 0.0;
  if (ph.visc == FLUID_VISC_POWER) return ph.visc_exp * mu * fl_rcp(T);
  return mu * (1.5 * fl_rcp(T) - fl_rcp(T + ph.suth_S));
}

// The power-law exponent as p / q with 0 < p, q <= 16 when it is one to within a few ulp (0.7 is
// 7/10), for fl_pow_rational; q = 0 otherwise.  Also sets the FP32 copy.
inline void set_power_law(Phys& ph, double e) {
  ph.visc_exp = e;
  ph.visc_e32 = (float)e;
  ph.visc_p = ph.visc_q = 0;
  ph.visc_hw_lo = ph.visc_hw_hi = 0;
  for (int q = 1; q <= 16; ++q) {
    const double pq = e * q;
    const int p = (int)(pq + 0.5);
    if (p >= 1 && p <= 16 && fabs((double)p / q - e) <= 4.0 * 2.220446049250313e-16 * fabs(e)) {
      ph.visc_p = p;
      ph.visc_q = q;
      // |log2 x| < B keeps the FP32 estimate and x^p normal
      int B = 49;
      while (B > 1 && (B * e >= 125.0 || B * p >= 1021)) --B;
      ph.visc_hw_lo = (1023 - B) << 20;
      ph.visc_hw_hi = (1023 + B) << 20;
      return;
    }
  }
}

// The factor of the cell differences in the forward faces' indicators: with 2^16 the default epsilon of 1e-40
// and the squares beside it keep all bits of a pair (4 epsilon becomes 2^-99), and differences up to 2^33
// stay below the limit of the indicators (cell_values).
constexpr float kIndScale = 65536.0f;

// The ff constants of Phys (after its other members are set).  The indicators' 4 epsilon is kept at
// 2^-152 or above, so that its reciprocal stays an FP32 number: smaller values only act where every
// difference of the stencil is below 2^-76, under the rounding of the smallest states the ff path takes
// (2^-72 at 1.9e-6).
inline void set_ff(Phys& ph) {
  ph.k.gamma = ff_of(ph.gamma);
  ph.k.gm1 = ff_of(ph.gm1);
  ph.k.igm1 = ff_of(ph.igm1);
  ph.k.gg = ff_of(ph.gamma * ph.igm1);
  ph.k.iR = ff_of(ph.iR);
  const double e4 = 4.0 * ph.eps * ((double)kIndScale * kIndScale);
  ph.k.eps4 = ff_of(e4 < 7.52316384526264e-37 ? 7.52316384526264e-37 : e4);
  ph.k.mu_ref = ff_of(ph.mu_ref);
  ph.k.mu_TS = ff_of(ph.mu_ref * (ph.T_ref + ph.suth_S));
  ph.k.iT_ref = ff_of(ph.iT_ref);
  ph.k.suth_S = ff_of(ph.suth_S);
  ph.k.lam_fac = ff_of(ph.lam_fac);
  ph.k.dt_visc = ff_of(ph.dt_visc_k);
  ph.k.visc_exp = ff_of(ph.visc_exp);
  ph.k.re = ff_of(2.0 * sqrt(ph.eps));
}

// Configuration check shared by the entry points: NULL if valid, else a static message.
const char* config_error(const fluid_config* c);

// Kernels the launchers below have enqueued from this host thread (each launch site adds one); the
// solver's profiler counts the kernels of a bracketed call by the difference.
inline thread_local long long t_launches = 0;

// The kernels of a step follow one another on one stream, and on small grids the gap between two of
// them is as long as the kernel.  They are launched with programmatic stream serialisation: the
// next kernel is set up while the last blocks of this one run, and waits (step_wait, the first
// statement of every kernel launched this way) until this one has finished and its writes are
// visible.  A launch that follows or precedes anything else on the stream is ordered as usual.  Shock
// tube of 200 cells, 20 steps of 10 launches: 2.28 -> 1.91 ms (with the CFL reduction as one kernel);
// step adjoint of 96 x 48 and 512 x 128 cells: 427 -> 374 and 600 -> 533 us.
// Such a kernel begins before the kernel that writes its input has ended.  The read-only load path (__ldg, or
// what the compiler makes of a const __restrict__ kernel parameter) is defined only for data that no one
// writes during the kernel's lifetime, and the compiler may move loads through a __restrict__ parameter ahead of
// the wait.  So the pointer parameters of these kernels are not __restrict__, and what another kernel
// wrote is read by plain loads (ld); only what the set-up wrote once (metrics) may take __ldg.
// The batches' kernels, which fill the GPU, are launched plainly: eight served solves took 8.3 ms so,
// 9.9 ms with the overlap.
template <class... P, class... A>
void launch_step(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &at;
  c.numAttrs = 1;
  (void)cudaLaunchKernelEx(&c, kernel, static_cast<A&&>(args)...);   // cudaGetLastError has the error
  ++t_launches;
}
__device__ __forceinline__ void step_wait() {
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// ---- launchers implemented in kernels_fp64.cu --------------------------------------------------
// W32 (mixed path only, else null): the primitives go there as pairs (load_pair) instead of to W
cudaError_t launch_prim_bc(const double* U, double* W, float* W32, const Geo& g, const Phys& ph,
                           const BC& bc, Ctl* ctl, cudaStream_t st);
cudaError_t launch_grad(const double* W, double* G, const Geo& g, const Phys& ph, cudaStream_t st);
// blocks of the marching FP64 face kernels: one thread per segment of `seg` cells along D
int face_grid(int D, const Geo& g, int block, int seg);
// Seam buffer of the FP64 face kernels: 10 doubles per segment item (lines x segments of a launch),
// cap items; a launch whose segments are shorter than kSeamMinSeg or that does not fit runs without
// it (same result).  {nullptr, 0} turns it off.
struct SeamBuf {
  double* p;
  long long cap;
};
constexpr int kSeamMinSeg = 4;
long long seam_capacity(const Geo& g);   // items for segments of kSeamMinSeg cells on every axis
// the buffer for a launch of segments of `seg` cells along D, or null when it runs without
double* seam_buffer(int D, const Geo& g, int seg, SeamBuf fb);
// the first cells of the segments after each line's first, from the fluxes in FB
cudaError_t launch_face_seam(int D, const double* FB, double* R, const Geo& g, int seg, cudaStream_t st);
// ---- WENO5 face kernels (face_launch.cuh, one translation unit per scheme) ----------------------
cudaError_t launch_face_js(int D, const double* W, const double* G, double* R, const Geo& g,
                           const Phys& ph, int block, int seg, SeamBuf fb, cudaStream_t st);
cudaError_t launch_face_z(int D, const double* W, const double* G, double* R, const Geo& g,
                          const Phys& ph, int block, int seg, SeamBuf fb, cudaStream_t st);
cudaError_t launch_face(int D, const double* W, const double* G, double* R, const Geo& g,
                        const Phys& ph, int block, int seg, SeamBuf fb, cudaStream_t st);
// the velocities of the body force's work come from W32 when given, else from W (also below)
cudaError_t launch_source(double* R, const double* W, const float* W32, const Geo& g, const Phys& ph,
                          cudaStream_t st);
// dt_arg > 0 replaces the solver's dt (used by the adjoint's stage recomputation)
cudaError_t launch_stage(int stage, const double* Un, const double* Us, const double* R, double* Ud,
                         const double* W, const float* W32, const Geo& g, const Phys& ph, Ctl* ctl,
                         double t_end, cudaStream_t st, double dt_arg = 0.0);
// stage `stage` of RK3 into Ud with the solver's dt, then the primitives of Ud into W (into W32 when
// that is given) for every padded cell, equal to launch_prim_bc(Ud, ...) on the result
cudaError_t launch_stage_prim(int stage, const double* Un, const double* Us, const double* R,
                              double* Ud, double* W, float* W32, const Geo& g, const Phys& ph,
                              const BC& bc, Ctl* ctl, double t_end, cudaStream_t st);
// the halo cells of W (of W32 when that is given) from its interior, as launch_stage_prim's second pass
cudaError_t launch_halo_prim(double* W, float* W32, const Geo& g, const Phys& ph, const BC& bc, Ctl* ctl,
                             cudaStream_t st);
// dt from the primitives: into ctl->dt, clipped to t_end (clip_to_ctl), or into *dt_out
cudaError_t launch_dt(const double* W, const Geo& g, const Phys& ph, double* partial, int nparts, Ctl* ctl,
                      double* dt_out, int clip_to_ctl, double t_end, cudaStream_t st);
int dt_partial_count(const Geo& g);
// ---- TENO6-A face kernels implemented in kernels_teno.cu ----------------------------------------
cudaError_t launch_face_teno(int D, const double* W, const double* G, double* R, const Geo& g,
                             const Phys& ph, cudaStream_t st);
// ---- mixed-precision launchers implemented in kernels_mixed.cu --------------------------------
cudaError_t launch_face_mixed(int D, const float* W32, const float* G32, double* R, const Geo& g,
                              const Phys& ph, cudaStream_t st);
// Stage output of the last axis's face kernel when the stage is fused into it: Ud = stage `stage`
// of RK3 from Un, Us and the completed right-hand side, and the primitives of Ud written to a second
// W32, since the kernel still reads the current one.  prims = false (the last stage of a call)
// writes Ud only.
struct StageOut {
  int stage;
  int prims;
  const double* Un;
  const double* Us;
  double* Ud;
  float* W32;
  Ctl* ctl;
  double t_end;
};
// the face kernel of the last axis (ndim - 1) accumulating into R's values of the other axes,
// fused with the stage combination and the primitives of its result (interior cells; the halo
// cells of the new W32 follow with launch_halo_prim)
cudaError_t launch_face_mixed_stage(const float* W32, const float* G32, const double* R, const Geo& g,
                                    const Phys& ph, const StageOut& so, cudaStream_t st);
cudaError_t launch_grad32(const float* W32, float* G32, const Geo& g, cudaStream_t st);
// check of the bulk-staging helpers (fluid_check_bulk_staging)
cudaError_t launch_bulk_probe(const float* src, float* dst, int nrows, unsigned extra_tx,
                              unsigned* flags, cudaStream_t st);
cudaError_t launch_dt32(const float* W32, const Geo& g, const Phys& ph, double* partial, int nparts, Ctl* ctl,
                        double* dt_out, int clip_to_ctl, double t_end, cudaStream_t st);

// ---- adjoint launchers implemented in kernels_adjoint.cu ----------------------------------------
cudaError_t launch_adj_faces(const double* W, const double* G, const double* mu, double* CW,
                             double* CG, double* gW, double* gG, const Geo& g, const Phys& ph,
                             cudaStream_t st);
cudaError_t launch_adj_source(const double* mu, double* gW, const Geo& g, const Phys& ph, cudaStream_t st);
cudaError_t launch_adj_bc(const double* W, double* gW, double* gvw_col, const Geo& g,
                          const Phys& ph, const BC& bc, cudaStream_t st);
cudaError_t launch_adj_prim(const double* U, const double* gW, double* gU, const Geo& g,
                            const Phys& ph, cudaStream_t st);
cudaError_t launch_adj_phi(const double* gvw_col, const double* xc, double* gphi, int p_t1,
                           int h_t1, int ext_t2, int begin, int count, double amp,
                           double two_pi_kappa, cudaStream_t st);
int wall_loss_parts(const Geo& g, int A);
cudaError_t launch_wall_loss(const double* W, double* part, int nparts, double* J, double* gT2,
                             const Geo& g, const Phys& ph, int A, int side, double Tw,
                             cudaStream_t st);
cudaError_t launch_wall_fluxes(const double* W, double* qw, double* tw, const Geo& g, const Phys& ph,
                               int A, int side, double Tw, cudaStream_t st);
cudaError_t launch_wall_loss_grad(const double* U, const double* gT2, double* dJdU, const Geo& g,
                                  const Phys& ph, int A, int side, cudaStream_t st);
cudaError_t launch_lincomb(double* out, double c0, const double* x0, double c1, const double* x1,
                           double c2, const double* x2, double c3, const double* x3, const Geo& g,
                           cudaStream_t st);

cudaError_t launch_prim_to_cons(const double* W, double* U, int ncell, const Phys& ph,
                                cudaStream_t st);
// block decomposition: doubles of one packed halo buffer of axis A, and the copy between the three
// layers next to face (A, side) and the buffer (unpack: buffer -> halo layers; else interior
// layers -> buffer)
size_t halo_count(const Geo& g, int A);
cudaError_t launch_halo_copy(double* U, double* buf, const Geo& g, int A, int side, bool unpack,
                             cudaStream_t st);
cudaError_t launch_wall_velocity(const double* phi, double* vw, const double* xc, int p, int h,
                                 int begin, int count, double amp, double two_pi_kappa,
                                 cudaStream_t st);

// ---- batched launches of the serving loop ------------------------------------------------------
// One launch advances every solve of a bucket: the kernel's blocks walk the "virtual blocks" of all
// solves (each solve's own launch grid of that kernel, laid end to end), and every virtual block
// runs the standalone kernel's body with the solve's data and its own block index and grid size,
// so each solve computes exactly what its standalone launches compute.  Solves of any grid size
// (and 2-D with 3-D) share a bucket; the grids of the launches are fixed, so a chunk of steps is
// captured once per bucket in a CUDA graph and the table below, in device memory, is rewritten
// between chunks as solves are admitted and retire.
constexpr int kBatchMax = 64;   // solves per bucket
enum BatchKernel {
  BK_PRIM = 0, BK_DT, BK_GRAD, BK_FACE0, BK_FACE1, BK_FACE2,
  BK_STAGEP, BK_HALO, BK_STAGE, BK_COUNT
};
struct BatchSlot {
  Geo g;
  Phys ph;
  BC bc;
  double* U;          // state (advanced in place)
  double* A;          // stage state
  double* R;          // right-hand side
  double* W;          // primitives (FP64)
  double* G;          // FP64 gradients (FP64 viscous)
  float* W32;         // primitives (mixed)
  float* G32;         // FP32 gradients (mixed viscous)
  double* partial;    // CFL partial maxima
  int nparts;         // their count (0 with a fixed dt)
  Ctl* ctl;
  double t_end;
  int steps;          // steps of the current chunk; the solve idles at later steps
  int vgrid[BK_COUNT][3];
};
struct BatchTable {
  int nslots;
  int pad;
  long long prefix[BK_COUNT][kBatchMax + 1];   // virtual blocks before each solve, per kernel
  BatchSlot slot[kBatchMax];
};
// the solve of virtual block vb of kernel k (binary search of the prefix)
__device__ __forceinline__ int batch_slot(const BatchTable* __restrict__ t, int k, long long vb) {
  int lo = 0, hi = t->nslots - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (t->prefix[k][mid] <= vb) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}
__device__ __forceinline__ uint3 batch_bid(const int vg[3], long long lb) {
  uint3 b;
  b.x = (unsigned)(lb % vg[0]);
  b.y = (unsigned)((lb / vg[0]) % vg[1]);
  b.z = (unsigned)(lb / ((long long)vg[0] * vg[1]));
  return b;
}
#define FL_BATCH_LOOP(K)                                                        \
  const long long total_ = t->prefix[K][t->nslots];                             \
  for (long long vb = blockIdx.x; vb < total_; vb += gridDim.x) {                \
    const int si_ = batch_slot(t, K, vb);                                       \
    const BatchSlot& S = t->slot[si_];                                          \
    const uint3 bid = batch_bid(S.vgrid[K], vb - t->prefix[K][si_]);            \
    const uint3 gdim = make_uint3(S.vgrid[K][0], S.vgrid[K][1], S.vgrid[K][2]);
#define FL_BATCH_END \
    __syncthreads(); \
  }
// blocks of a batched launch: as many as fit the GPU at once (each walks virtual blocks)
template <class K>
int batch_grid(K kernel, int block, size_t smem = 0) {
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, smem) != cudaSuccess || per_sm < 1)
    per_sm = 1;
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return per_sm * sms;
}
// the batched WENO5 FP64 face kernels of one axis, per scheme
cudaError_t launch_batch_face_js(const BatchTable* dev, int D, int step, bool visc, cudaStream_t st);
cudaError_t launch_batch_face_z(const BatchTable* dev, int D, int step, bool visc, cudaStream_t st);
// fluid_create with stream-ordered allocations on st (cudaMallocAsync): set-up copies are enqueued
// on st and nothing synchronises; fluid_destroy of such a solver frees on st without waiting
int solver_create_async(const fluid_config* cfg, cudaStream_t st, fluid_solver** out);
// a solver's part of a batch (its geometry, physics, boundaries and scratch, state U, t_end); false
// when its configuration has no batched kernels (TENO6-A, sixth-order stencils, exchange faces)
bool batch_slot_of(fluid_solver* s, double* U, double t_end, BatchSlot& out);
// fill slot.vgrid and the prefixes for the solves of t (their Geo and Phys set)
void batch_plan(BatchTable& t);
// enqueue the batched kernels of `chunk` RK3 steps (what fluid_step(U, chunk) does for every solve)
cudaError_t launch_batch_chunk(const BatchTable* dev, int chunk, bool mixed, int weno, bool visc,
                               cudaStream_t st);
// the mixed path's batched gradient and CFL kernels, and its face kernels (kernels_mixed.cu)
enum { BMX_GRAD = 0, BMX_DT = 1 };
cudaError_t launch_batch_mixed(const BatchTable* dev, int kind, int step, cudaStream_t st);
cudaError_t launch_batch_mixed_faces(const BatchTable* dev, int D, int step, int weno, bool visc,
                                     cudaStream_t st);

}  // namespace fl
