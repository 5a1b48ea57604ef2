// kernels_march_kfield.cu -- the marching kernel's instantiations: per-node tensor field (a source decided at run time).
#include "kernels_march.cuh"

namespace lbm {

cudaError_t launch_march_kfield(const lbm_solver *s, int src, bool prepare, cudaStream_t st)
{
#define LBM_GO(CV, DF) march_t<CV, DF, 2, true>(s, src, prepare, st)
    LBM_MARCH_FAMILIES(LBM_GO)
#undef LBM_GO
}

}  // namespace lbm
