// WENO5-Z face kernels of the FP64 path for the serving loop's batches.
#include "face_batch.cuh"

namespace fl {

cudaError_t launch_batch_face_z(const BatchTable* dev, int D, int step, bool visc, cudaStream_t st) {
  return visc ? launch_batch<FLUID_WENO_Z, true>(dev, D, step, st) : launch_batch<FLUID_WENO_Z, false>(dev, D, step, st);
}

}  // namespace fl
