// k_render for F32 blocks.
#include "render_kernel.cuh"

namespace lrvol {

cudaError_t launch_render_f32(const RenderParams &prm, int degree, int f, bool trace, cudaStream_t s) {
  return trace ? launch_render_s<LRVOL_STORE_F32, true>(prm, degree, f, s)
               : launch_render_s<LRVOL_STORE_F32, false>(prm, degree, f, s);
}

}  // namespace lrvol
