// kernels_tile_general_f32_b.cu -- the small lattices' general kernel, float, Scheme B.
#include "kernels_tile_general.cuh"

namespace lbm {

cudaError_t launch_tile_general_f32_b(const lbm_solver *s, int src, const double *records, int steps, bool prepare,
                                        cudaStream_t st)
{
    LBM_TILE_G_CASES(float, false)
}

}  // namespace lbm
