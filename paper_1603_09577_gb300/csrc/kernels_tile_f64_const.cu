// kernels_tile_f64_const.cu -- the small lattices' kernel, double storage, constant tensor.
#include "kernels_tile.cuh"

namespace lbm {

cudaError_t launch_tile_f64_const(const lbm_solver *s, int src, int steps, bool prepare, cudaStream_t st)
{
    LBM_TILE_FAMILIES(double, false)
}

}  // namespace lbm
