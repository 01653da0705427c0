// WENO5-JS face kernels of the FP64 path.
#include "face_launch.cuh"

namespace fl {

cudaError_t launch_face_js(int D, const double* W, const double* G, double* R, const Geo& g,
                          const Phys& ph, int block, int seg, SeamBuf fb, cudaStream_t st) {
  if (ph.visc == FLUID_VISC_NONE)
    return launch_scheme<FLUID_WENO_JS, false>(D, W, G, R, g, ph, block, seg, fb, st);
  return launch_scheme<FLUID_WENO_JS, true>(D, W, G, R, g, ph, block, seg, fb, st);
}

}  // namespace fl
