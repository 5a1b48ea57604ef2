// kernels_march_free.cu -- the marching kernel's instantiations: constant tensor, no source.
#include "kernels_march.cuh"

namespace lbm {

cudaError_t launch_march_free(const lbm_solver *s, int src, bool prepare, cudaStream_t st)
{
#define LBM_GO(CV, DF) march_t<CV, DF, 0, false>(s, src, prepare, st)
    LBM_MARCH_FAMILIES(LBM_GO)
#undef LBM_GO
}

}  // namespace lbm
