// kernels_ensemble4.cu -- the ensemble with four time steps per sweep through HBM: one
// launch covers the strips of every instance, each marched as in kernels_march.cuh
// (FP32 storage, periodic walls, constant K per instance).
//
// The instances' constants cannot sit in the argument space, where packed
// instructions would read them; a block brings its instance's constants through
// shared memory into registers, and a lane marches two pairs of columns so that
// they serve twice: 128 registers, four blocks of four warps per SM.
//
// 128 instances of 64 to 1024 nodes a side, 100 steps (GB300): 20.9 -> 14.56 ms
// against the two-step 30 x 30 tiles.
#include "kernels_march.cuh"
#include "lbm_ensemble.h"

namespace lbm {

constexpr int kE4T = 4, kE4KW = 1, kE4P = 2, kE4Stage = 2, kE4Blocks = 4;
using E4 = March<kE4T, kE4KW, kE4P, kE4Stage>;
static_assert(E4::kOut == kEns4Cols, "strips of the work list");
constexpr int kE4Const = sizeof(Coll<float>) / sizeof(float);
constexpr int kE4Smem = E4::kSmem + ((kE4Const * 4 + 15) & ~15);

template <int CONV, int DIFF>
__global__ void __launch_bounds__(E4::kThreads, kE4Blocks)
k_ens_march(const EnsInst *__restrict__ inst, const int4 *__restrict__ items, int parity)
{
    extern __shared__ __align__(16) float sm_e4[];
    const int4 it = __ldg(items + blockIdx.x);
    const EnsInst &I = inst[it.x];
    float *consts = sm_e4 + E4::kSmem / sizeof(float);
    for (int i = threadIdx.x; i < kE4Const; i += E4::kThreads) consts[i] = reinterpret_cast<const float *>(&I.k)[i];
    __syncthreads();
    Coll<F2> kc;
#pragma unroll
    for (int i = 0; i < kE4Const; ++i) {                 // (volatile: the constants are to stay in registers)
        float v;
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"((unsigned)__cvta_generic_to_shared(consts + i)));
        reinterpret_cast<F2 *>(&kc)[i] = F2(v);
    }
    MarchArgs a;
    a.src = parity ? I.pop[1] : I.pop[0];
    a.dst = parity ? I.pop[0] : I.pop[1];
    a.Afield = nullptr;
    a.plane = I.plane;
    a.pitch = (int)I.pitch;
    a.nx = I.nx;
    a.ny = I.ny;
    a.abb_x = a.abb_y = 0;
    a.has_src = 0;
    a.give_up = 0;
    a.err = I.err;
    const bool cols = it.y - kE4T < 0 || it.y - (kE4T - 1) + E4::kW >= a.nx || it.y - kE4T + E4::kInW > a.pitch;
    if (cols) march_strip<CONV, DIFF, 0, false, kE4T, kE4KW, kE4P, kE4Stage, true>(a, kc, sm_e4, it.y, it.z, it.w, true, false);
    else march_strip<CONV, DIFF, 0, false, kE4T, kE4KW, kE4P, kE4Stage, false>(a, kc, sm_e4, it.y, it.z, it.w, false, false);
}

template <int CONV, int DIFF>
static cudaError_t ens4_t(const lbm_ensemble_s *e, bool prepare, cudaStream_t st)
{
    static SmemOptIn once;
    const cudaError_t err = opt_in_smem((const void *)k_ens_march<CONV, DIFF>, kE4Smem, once);
    if (err != cudaSuccess || prepare) return err;
    k_ens_march<CONV, DIFF><<<e->nitems4, E4::kThreads, kE4Smem, st>>>(e->d_inst, e->d_items4, e->parity);
    return cudaGetLastError();
}

cudaError_t ens_launch_step4(const lbm_ensemble_s *e, bool prepare, cudaStream_t st)
{
    switch (e->family) {
    case 0: return ens4_t<0, 0>(e, prepare, st);
    case 1: return ens4_t<0, 1>(e, prepare, st);
    case 2: return ens4_t<0, 2>(e, prepare, st);
    case 3: return ens4_t<1, 0>(e, prepare, st);
    case 4: return ens4_t<1, 1>(e, prepare, st);
    case 5: return ens4_t<1, 2>(e, prepare, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace lbm
