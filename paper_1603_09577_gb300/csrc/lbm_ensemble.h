// lbm_ensemble.h -- internal state of a batched ensemble of independent lattices.
#pragma once

#include "lbm_internal.h"

namespace lbm {

constexpr int kEnsTile = 32;        // tile width (nodes along x)
constexpr int kEnsRows = 8;         // tile height: one node per thread
constexpr int kEnsThreads = kEnsTile * kEnsRows;

// Per-instance data read by the kernels (device table).
struct __align__(16) EnsInst {
    float *pop[2];          // A/B population buffers (9 planes each)
    long long pitch, plane;
    long long phi_off;      // offset of this instance in the packed phi arrays
    int nx, ny;
    Coll<float> k;          // constants of the collision (lbm_relax.cuh)
    float ux, uy, uxx, uxy, uyy;
    int *err;               // checked builds: shared index-fault word
};

__device__ __forceinline__ Params<float> ens_params(const EnsInst &I)
{
    Params<float> p;
    p.nx = I.nx; p.ny = I.ny; p.pitch = I.pitch; p.plane = I.plane;
    p.abb_x = 0; p.abb_y = 0;
    p.k = I.k;
    p.ux = I.ux; p.uy = I.uy; p.uxx = I.uxx; p.uxy = I.uxy; p.uyy = I.uyy;
    p.r0 = 0.f; p.r1 = 0.f; p.half_r0 = 0.f; p.inv_den = 1.f; p.inv_post = 1.f;
    p.has_src = 0;
    for (int i = 0; i < 4; ++i) p.phi_wall[i] = 0.f;
    p.Afield = nullptr;
    p.err = I.err;
    return p;
}

}  // namespace lbm

struct lbm_ensemble_s {
    int count = 0, family = 0, ntiles = 0, grid = 0, parity = 0;
    int spp = 1;                    // time steps per persistent launch (1 or 2)
    int ntiles2 = 0, grid2 = 0;     // 30 x 30 tiles of the two-step kernel
    int ntiles2p = 0, grid2p = 0;   // 62 x 14 pair tiles of the two-step kernel
    int shape2 = 0;                 // two-step tiles: 0 30 x 30 (one node per thread), 1 62 x 14 (two)
    int persistent2 = 0;            // two-step launch: 0 a block per tile, 1 persistent with a fixed
                                    // stride, 2 persistent with tiles claimed from a counter
    int nitems4 = 0;                // strips of the four-step sweeps; 0: an instance is too small for them
    int4 *d_items4 = nullptr;       // instance, first column, rows from .. to
    int4 *d_tiles2 = nullptr;
    int4 *d_tiles2p = nullptr;
    int *d_claim = nullptr;         // tile counter and departed-block counter of mode 2
    lbm::EnsInst *d_inst = nullptr;
    int4 *d_tiles = nullptr;
    int *tile_begin = nullptr;      // host: first tile of each instance (count + 1)
    long long total_nodes = 0;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    int graph_steps = 0, graph_parity = 0;
    int *err = nullptr;             // index-fault word of checked builds
    double *partials = nullptr;     // per-tile statistics (8 doubles per 32 x 8 tile)
    int *d_tile_begin = nullptr;    // device copy of tile_begin
};

namespace lbm {
cudaError_t ens_launch_step(const lbm_ensemble_s *e, int t_begin, int t_end, int blocks, cudaStream_t st);
cudaError_t ens_launch_step2(const lbm_ensemble_s *e, cudaStream_t st);
// four steps over the strips of every instance (kernels_ensemble4.cu)
cudaError_t ens_launch_step4(const lbm_ensemble_s *e, bool prepare, cudaStream_t st);
constexpr int kEns4Cols = 120;      // output columns of a strip
int ens2_occupancy_blocks(int family, int shape);
constexpr int kEns2Tile = 30;       // two-step tiles: 30 x 30 outputs
constexpr int kEns2PCols = 62;      // two-step pair tiles: 62 x 14 outputs
constexpr int kEns2PRows = 14;
cudaError_t ens_launch_init(const lbm_ensemble_s *e, const void *phi, int in_prec, cudaStream_t st);
cudaError_t ens_launch_get_phi(const lbm_ensemble_s *e, void *out, int out_prec, cudaStream_t st);
// the eight statistics of every instance into out (count x 8 doubles)
cudaError_t ens_launch_reduce(const lbm_ensemble_s *e, const double *ref, double *out, cudaStream_t st);
int ens_occupancy_blocks(int family);
}  // namespace lbm
