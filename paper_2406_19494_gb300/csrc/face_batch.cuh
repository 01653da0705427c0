// Batched launches of the WENO5 face kernels (face_kernels.cuh) of one scheme: blocks walk the
// virtual blocks of a bucket's solves (BatchTable).  Included by the translation unit of the scheme.
#pragma once

#include "face_kernels.cuh"

namespace fl {

namespace {

template <int D, int SCHEME, bool VISC>
__global__ void __launch_bounds__(TileShape<D>::threads, TileShape<D>::blocks) kb_face(const BatchTable* __restrict__ t, int step) {
  extern __shared__ __align__(16) unsigned char raw[];
  FL_BATCH_LOOP(BK_FACE0 + D)
  (void)gdim;
  if (step < S.steps)
    k_face_tile_body<D, SCHEME, VISC>(S.W, S.G, S.R, S.g, S.ph,
                                      *reinterpret_cast<TileShared<TileShape<D>::threads>*>(raw), bid.x, bid.y);
  FL_BATCH_END
}

template <int D, int SCHEME, bool VISC>
cudaError_t launch_batch_d(const BatchTable* dev, int step, cudaStream_t st) {
  constexpr int n = TileShape<D>::threads;
  constexpr size_t smem = sizeof(TileShared<n>);
  // the attribute is per device
  const cudaError_t e = cudaFuncSetAttribute(kb_face<D, SCHEME, VISC>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  static const int grid = batch_grid(kb_face<D, SCHEME, VISC>, n, smem);
  (kb_face<D, SCHEME, VISC><<<grid, n, smem, st>>>(dev, step), ++t_launches);
  return cudaGetLastError();
}

template <int SCHEME, bool VISC>
cudaError_t launch_batch(const BatchTable* dev, int D, int step, cudaStream_t st) {
  if (D == 0) return launch_batch_d<0, SCHEME, VISC>(dev, step, st);
  if (D == 1) return launch_batch_d<1, SCHEME, VISC>(dev, step, st);
  return launch_batch_d<2, SCHEME, VISC>(dev, step, st);
}

}  // namespace

}  // namespace fl
