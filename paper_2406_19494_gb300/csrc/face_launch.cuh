// Launches of the WENO5 face kernels (face_kernels.cuh) of one scheme; included by the translation
// unit of that scheme.
#pragma once

#include "face_kernels.cuh"

namespace fl {

namespace {

// launches of at most this many tiles (one per SM of this GPU) take the small ones along y and z (SmallTile has
// both sides measured)
constexpr long long kSmallTiles = 152;

template <int D, int SCHEME, bool VISC>
__global__ void __launch_bounds__(128) k_face(const double* W, const double* G,
                                              double* R, double* FB,
                                              const __grid_constant__ Geo g, const __grid_constant__ Phys ph,
                                              int seg) {
  step_wait();
  k_face_body<D, SCHEME, VISC>(W, G, R, FB, g, ph, seg, blockIdx, gridDim);
}

template <int D, int SCHEME, bool VISC, class S = TileShape<D>>
__global__ void __launch_bounds__(S::threads, S::blocks) k_face_tile(
    const double* W, const double* G, double* R,
    const __grid_constant__ Geo g, const __grid_constant__ Phys ph) {
  step_wait();
  extern __shared__ __align__(16) unsigned char raw[];
  const int cols = tile_cols<D, S>(g);                     // neighbouring blocks: neighbouring columns
  k_face_tile_body<D, SCHEME, VISC, S>(W, G, R, g, ph, *reinterpret_cast<TileShared<S::threads>*>(raw),
                                       blockIdx.x % cols, blockIdx.x / cols);
}

template <int D, int SCHEME, bool VISC, class S = TileShape<D>>
cudaError_t launch_tile(const double* W, const double* G, double* R, const Geo& g, const Phys& ph,
                        cudaStream_t st) {
  constexpr int n = S::threads;
  constexpr size_t smem = sizeof(TileShared<n>);
  const long long tiles = tile_rows<D, S>(g) * tile_cols<D, S>(g);
  if constexpr (D > 0 && n == TileShape<D>::threads)
    if (tiles <= kSmallTiles) return launch_tile<D, SCHEME, VISC, SmallTile>(W, G, R, g, ph, st);
  const cudaError_t e = cudaFuncSetAttribute(k_face_tile<D, SCHEME, VISC, S>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  launch_step(k_face_tile<D, SCHEME, VISC, S>, (unsigned)tiles, n, smem, st, W, G, R, g, ph);
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
  if (block <= 0) block = 128;
  const int grid = face_grid(D, g, block, seg);
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
