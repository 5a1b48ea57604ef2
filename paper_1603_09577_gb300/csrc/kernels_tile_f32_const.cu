// kernels_tile_f32_const.cu -- the small lattices' kernel, float storage, constant tensor.
#include "kernels_tile.cuh"

namespace lbm {

cudaError_t launch_tile_f32_const(const lbm_solver *s, int src, int steps, bool prepare, cudaStream_t st)
{
    LBM_TILE_FAMILIES(float, false)
}

}  // namespace lbm
