// kernels_tile_f32_kfield.cu -- the small lattices' kernel, float storage, per-node tensor field.
#include "kernels_tile.cuh"

namespace lbm {

cudaError_t launch_tile_f32_kfield(const lbm_solver *s, int src, int steps, bool prepare, cudaStream_t st)
{
    LBM_TILE_FAMILIES(float, true)
}

}  // namespace lbm
