// Launches of the WENO5 face kernels (face_kernels.cuh) of one scheme; included by the translation
// unit of that scheme.
#pragma once

#include "face_kernels.cuh"

namespace fl {

namespace {

template <int D, int SCHEME, bool VISC>
__global__ void __launch_bounds__(128) k_face(const double* __restrict__ W, const double* __restrict__ G,
                                              double* __restrict__ R, double* __restrict__ FB,
                                              const __grid_constant__ Geo g, const __grid_constant__ Phys ph,
                                              int seg) {
  step_wait();
  k_face_body<D, SCHEME, VISC>(W, G, R, FB, g, ph, seg, blockIdx, gridDim);
}

template <int D, int SCHEME, bool VISC>
__global__ void __launch_bounds__(TileShape<D>::threads, TileShape<D>::blocks) k_face_tile(
    const double* __restrict__ W, const double* __restrict__ G, double* __restrict__ R,
    const __grid_constant__ Geo g, const __grid_constant__ Phys ph) {
  step_wait();
  extern __shared__ __align__(16) unsigned char raw[];
  const int cols = tile_cols<D>(g);                        // neighbouring blocks: neighbouring columns
  k_face_tile_body<D, SCHEME, VISC>(W, G, R, g, ph,
                                    *reinterpret_cast<TileShared<TileShape<D>::threads>*>(raw),
                                    blockIdx.x % cols, blockIdx.x / cols);
}

template <int D, int SCHEME, bool VISC>
cudaError_t launch_tile(const double* W, const double* G, double* R, const Geo& g, const Phys& ph,
                        cudaStream_t st) {
  constexpr int n = TileShape<D>::threads;
  constexpr size_t smem = sizeof(TileShared<n>);
  const cudaError_t e = cudaFuncSetAttribute(k_face_tile<D, SCHEME, VISC>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const unsigned grid = (unsigned)(tile_rows<D>(g) * tile_cols<D>(g));
  launch_step(k_face_tile<D, SCHEME, VISC>, grid, n, smem, st, W, G, R, g, ph);
  return cudaGetLastError();
}

template <int SCHEME, bool VISC>
cudaError_t launch_scheme(int D, const double* W, const double* G, double* R, const Geo& g, const Phys& ph,
                          int block, int seg, SeamBuf fb, cudaStream_t st) {
  if (seg <= 0) {
    if (D == 0) return launch_tile<0, SCHEME, VISC>(W, G, R, g, ph, st);
    if (D == 1) return launch_tile<1, SCHEME, VISC>(W, G, R, g, ph, st);
    return launch_tile<2, SCHEME, VISC>(W, G, R, g, ph, st);
  }
  int grid;
  face_shape(D, g, block, seg, grid);
  double* FB = seam_buffer(D, g, seg, fb);
  if (D == 0) launch_step(k_face<0, SCHEME, VISC>, grid, block, 0, st, W, G, R, FB, g, ph, seg);
  else if (D == 1) launch_step(k_face<1, SCHEME, VISC>, grid, block, 0, st, W, G, R, FB, g, ph, seg);
  else launch_step(k_face<2, SCHEME, VISC>, grid, block, 0, st, W, G, R, FB, g, ph, seg);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || !FB) return e;
  return launch_face_seam(D, FB, R, g, seg, st);
}

}  // namespace

}  // namespace fl
