// kernels_tile_general_f64_a.cu -- the small lattices' general kernel, double, Scheme A.
#include "kernels_tile_general.cuh"

namespace lbm {

cudaError_t launch_tile_general_f64_a(const lbm_solver *s, int src, const double *records, int steps, bool prepare,
                                        cudaStream_t st)
{
    LBM_TILE_G_CASES(double, true)
}

}  // namespace lbm
