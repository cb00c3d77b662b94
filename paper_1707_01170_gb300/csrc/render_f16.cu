// k_render for F16 blocks.
#include "render_kernel.cuh"

namespace lrvol {

cudaError_t launch_render_f16(const RenderParams &prm, int degree, int f, bool trace, cudaStream_t s) {
  return trace ? launch_render_s<LRVOL_STORE_F16, true>(prm, degree, f, s)
               : launch_render_s<LRVOL_STORE_F16, false>(prm, degree, f, s);
}

}  // namespace lrvol
