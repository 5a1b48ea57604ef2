// lbm_internal.h -- host-side solver state, workspace layout and the kernel
// launchers shared by the translation units of liblbm.
#pragma once

#include <cuda_runtime.h>
#include <stddef.h>

#include <atomic>
#include <string>

#include "lbm.h"
#include "lbm_relax.cuh"

namespace lbm {

constexpr int kReduceBlocks = 1024;     // fixed: deterministic reduction order
constexpr int kReduceThreads = 256;
constexpr int kPitchAlign = 64;         // row pitch in elements (>= 128 B rows)

struct Layout {
    long long pitch = 0, plane = 0;
    size_t esize = 0, csize = 0;
    size_t off_pop[2] = {0, 0}, off_phi[2] = {0, 0};
    size_t off_afield = 0, off_staging = 0, off_partials = 0, off_flag = 0, off_check = 0, off_err = 0, off_cnt = 0;
    size_t pop_bytes = 0, phi_bytes = 0, total = 0;
};

int make_layout(const lbm_desc *d, Layout *L);

}  // namespace lbm

namespace lbm {

constexpr int kTileMaxT = 8;        // most steps of a launch over a small lattice's tiles

// The launches that a lattice can take and their estimated times (route.cu). The tiling
// of the small lattices' kernels: W x H tiles, at most T steps per launch; us: the
// estimated time of a step (1e30: no tiling fits). The search takes 15 to 100 us of host
// time and depends on the sizes, the walls, the precision, the path and the device only, not on
// the coefficients: a program that changes them as it goes searches once. T = 0: not planned yet.
struct TilePlan {
    int W = 0, H = 0, T = 0;
    double us = 0.0;
    bool general = false;           // for the general path's kernel
    int sms = 0;                    // for a device of so many SMs
    double launch[kTileMaxT + 1] = {};              // us of a launch of so many steps over the tiles
    double one = 0.0, two = 0.0, four = 0.0;        // FP32, Scheme B: us of the other kernels' launches
    bool nodes = false;             // two steps: 30 x 30 node tiles, not 62 x 14 pair tiles
};

// The launches of a call, in the order they run
struct Route {
    int tiles = 0;      // small lattices' tiles, which share their steps as evenly as they can
    int fours = 0;      // sweeps of four steps (the marching kernel)
    int pairs = 0;      // sweeps of two steps over pair tiles
    int twos = 0;       // sweeps of two steps by another kernel: the one that the descriptor
                        // names, or on the path left to the library 30 x 30 node tiles
    int ones = 0;       // single steps
};

}  // namespace lbm

struct lbm_solver {
    lbm_desc d;
    lbm_coeffs c;
    lbm::Layout L;
    int coeffs_set = 0, phi_set = 0, kfield_set = 0;
    char *ws = nullptr;
    size_t ws_bytes = 0;
    void *pop[2] = {nullptr, nullptr};
    float *phi[2] = {nullptr, nullptr};
    void *afield = nullptr;
    void *staging = nullptr;
    double *partials = nullptr;
    int *flag = nullptr;
    double *check = nullptr;        // 8 doubles: reduction output of lbm_check_finite
    int *err = nullptr;             // index-fault word of checked builds
    int cur = 0;
    int give_up = 0;                // 1: the four-step sweeps take every copy for late (a test)
    int fixed = 0;                  // 1: the kernels that the descriptor names, whatever the size
    int sms = 0;                    // SMs of the device, read at the first step
    lbm::TilePlan plan;
    // the kernels' parameters in the compute type of `prec`, made by lbm_set_coeffs (made at
    // every launch they took 0.1 us of host time of 2.1)
    lbm::Params<float> pf{};
    lbm::Params<double> pd{};
    long long t = 0;
    // Dirichlet records of the extrapolated axes (caller-owned device memory)
    const double *dir_vals = nullptr;
    int dir_nrec = 0;
    long long *dir_counter = nullptr;   // device: steps since the records' count restarted
    int dir_reset = 0;                  // 1: clear dir_counter before the next step
    int dir_off = 0;                    // place of the next sweep's first step within its lbm_step call
    // adjoint (caller-provided second workspace)
    char *adj = nullptr;
    void *lam[2] = {nullptr, nullptr};
    double *gA = nullptr;
    double *adj_partials = nullptr;
    int adj_cur = 0, adj_active = 0;
};

namespace lbm {

// Per-device record of a kernel's opt-in to more than 48 KB of dynamic shared
// memory. The flags are atomic, so first launches from several host threads do
// not race on them (cudaFuncSetAttribute is idempotent and may then run twice).
// The opt-in happens at the first launch on a device, which must therefore come
// before any stream capture on that device.
struct SmemOptIn {
    std::atomic<int> done[64];
};
cudaError_t opt_in_smem(const void *kernel, int bytes, SmemOptIn &flags);

void set_error(const std::string &msg);
int fail(int code, const std::string &msg);
int cuda_check(cudaError_t e, const char *what);

// kernel parameters in the compute type of the solver
template <class C>
const Params<C> &make_params(const lbm_solver *s);
template <> inline const Params<float> &make_params<float>(const lbm_solver *s) { return s->pf; }
template <> inline const Params<double> &make_params<double>(const lbm_solver *s) { return s->pd; }

// Family key of the step launchers: conv * 3 + diff, or 6 + diff for the linear
// family without a flux (conv 0 with u = 0), which runs the collision without
// the flux terms (kConvNone).
inline int step_key(const lbm_solver *s)
{
    if (s->c.conv == 0 && s->c.u[0] == 0.0 && s->c.u[1] == 0.0 && s->c.diff >= 0 && s->c.diff <= 2)
        return 6 + s->c.diff;
    return s->c.conv * 3 + s->c.diff;
}

// the prescaled rates, source factors and block of the collision (Params),
// from the rates s0..s8 and the block A (computed in double, rounded once)
template <class C>
inline void set_scaled_rates(const double s[9], double A3, double A35, double A5, Params<C> *p)
{
    const double h1 = 1.0 - 0.5 * s[1], h2 = 1.0 - 0.5 * s[2], h4 = 1.0 - 0.5 * s[4], h6 = 1.0 - 0.5 * s[6];
    p->se1 = (C)(s[1] / 36.0); p->se2 = (C)(s[2] / 36.0);
    p->sq4 = (C)(s[4] / 12.0); p->sq6 = (C)(s[6] / 12.0);
    p->sp7 = (C)(s[7] / 4.0); p->sp8 = (C)(s[8] / 4.0);
    p->he1 = (C)(-2.0 * h1 / 36.0); p->he2 = (C)(h2 / 36.0);
    p->hq4 = (C)(-h4 / 12.0); p->hq6 = (C)(-h6 / 12.0);
    p->a3s = (C)(A3 / 6.0); p->a35s = (C)(A35 / 6.0); p->a5s = (C)(A5 / 6.0);
    p->c3s = (C)(1.0 / 6.0 - A3 / 12.0); p->c35s = (C)(-A35 / 12.0); p->c5s = (C)(1.0 / 6.0 - A5 / 12.0);
}

// the constants of relax() for the coefficients c and the block A
inline Coll<double> make_coll(const lbm_coeffs &c, double A3, double A35, double A5)
{
    Coll<double> k;
    const double *s = c.s;
    const double ux = c.u[0], uy = c.u[1], uu = ux * ux + uy * uy;
    const double h1 = 1.0 - 0.5 * s[1], h2 = 1.0 - 0.5 * s[2], h4 = 1.0 - 0.5 * s[4], h6 = 1.0 - 0.5 * s[6];
    const bool quad = c.conv == 1;                    // B = a phi^2/2, C = a a phi^3/3
    k.nse1 = -s[1] / 36.0; k.nse2 = -s[2] / 36.0;
    k.sq4 = s[4] / 6.0; k.nsq4 = -s[4] / 12.0; k.sq6 = s[6] / 6.0; k.nsq6 = -s[6] / 12.0;
    k.sp7 = s[7] / 4.0; k.nsp7 = -k.sp7; k.sp8 = s[8] / 4.0; k.nsp8 = -k.sp8;
    k.na3 = -A3 / 6.0; k.na35 = -A35 / 6.0; k.na5 = -A5 / 6.0;
    k.ke1 = quad ? -2.0 : 3.0 * uu - 2.0;
    k.nkp1 = quad ? -1.0 : 3.0 * uu - 1.0;
    k.ke3 = (quad ? uu : 0.0) + (c.diff == 2 ? 2.0 / 3.0 : 0.0);
    const double half = quad ? 0.5 : 1.0, third = quad ? 1.0 / 3.0 : 1.0;
    k.bx = half * ux; k.by = half * uy;
    k.nbx = -k.bx; k.nby = -k.by;
    k.nkxx = -third * (ux * ux - uy * uy);
    k.nkxy = -third * ux * uy;
    k.inv_den = 1.0 / (1.0 - 0.5 * c.r1);
    k.phi0 = 0.5 * c.r0 * k.inv_den;
    k.r0 = c.r0 / 9.0; k.r1 = c.r1 / 9.0;             // the source's factors below are per R/9
    k.nhe1 = 2.0 * h1 / 4.0; k.he2 = h2 / 4.0;
    k.hqx = -0.75 * h4 * ux; k.hqy = -0.75 * h6 * uy;
    k.hqx2 = 1.5 * h4 * ux; k.hqy2 = 1.5 * h6 * uy;
    k.jsx = 9.0 * ((1.0 / 6.0 - A3 / 12.0) * ux - A35 / 12.0 * uy);
    k.jsy = 9.0 * (-A35 / 12.0 * ux + (1.0 / 6.0 - A5 / 12.0) * uy);
    k.ux9 = 9.0 * ux; k.uy9 = 9.0 * uy; k.sixth = 1.0 / 6.0; k.nsixth = -1.0 / 6.0;
    k.four = 4.0; k.mtwo = -2.0; k.half = 0.5;
    return k;
}

cudaError_t launch_init(const lbm_solver *s, const void *phi, int in_prec, cudaStream_t st);
cudaError_t launch_step(const lbm_solver *s, int src, cudaStream_t st);
// node tiles of two steps; rows: lbm_desc.block_rows (4: 30 x 30, else 30 x 62)
cudaError_t launch_step2(const lbm_solver *s, int src, int rows, cudaStream_t st);
cudaError_t launch_step2m(const lbm_solver *s, int src, cudaStream_t st);
cudaError_t launch_step2_tma(const lbm_solver *s, int src, cudaStream_t st);
// two steps per pass, two x-adjacent nodes per thread (kernel_variant 5)
cudaError_t launch_step2p_f32(const lbm_solver *s, int src, cudaStream_t st);
cudaError_t launch_step2p_bf16s(const lbm_solver *s, int src, cudaStream_t st);
cudaError_t launch_step_ptr(const lbm_solver *s, const void *src, void *dst, cudaStream_t st);
// general path (Scheme A, extrapolation walls, power-law flux): a step when
// phi0 is null, else the initialisation from phi0
cudaError_t launch_general_f64(const lbm_solver *s, int src, const double *bv, const void *phi0, int in_prec,
                               cudaStream_t st);
cudaError_t launch_general_f32(const lbm_solver *s, int src, const double *bv, const void *phi0, int in_prec,
                               cudaStream_t st);
// two general steps per pass (FP32); records: the caller's Dirichlet records
cudaError_t launch_step2_general(const lbm_solver *s, int src, const double *records, cudaStream_t st);
// advance the device record count by `by` steps (one thread, after a call's sweeps)
cudaError_t launch_tick(long long *counter, int by, cudaStream_t st);
// four steps per sweep of an FP32 lattice (kernels_march.cuh); prepare: only the
// kernel's attributes, so that a later first launch may happen under capture
cudaError_t launch_march_src(const lbm_solver *s, int src, bool prepare, cudaStream_t st);
cudaError_t launch_march_free(const lbm_solver *s, int src, bool prepare, cudaStream_t st);
cudaError_t launch_march_kfield(const lbm_solver *s, int src, bool prepare, cudaStream_t st);
// `steps` steps in one launch over the tiles of s->plan (kernels_tile.cuh)
TilePlan tile_plan(int nx, int ny, bool f64, bool general, int sms);
double tile_launch_us(int nx, int ny, int W, int H, int steps, bool f64, bool general, int sms);
// the route of nsteps steps on a device of `sms` SMs, and whether the launch is left to the library
bool general_path(const lbm_solver *s);
bool auto_path(const lbm_solver *s);
Route plan_route(lbm_solver *s, int nsteps, int sms);
// strips and chunks of the marching kernel's launch: blocks of H rows, four per SM
constexpr int kMarchBlocks = 4, kMarchOut = 120;
struct MarchGrid { int strips, chunks, H; };
MarchGrid march_grid(int nx, int ny, int sms);
#define LBM_DECLARE_TILE_GENERAL(NAME) \
    cudaError_t NAME(const lbm_solver *s, int src, const double *records, int steps, bool prepare, cudaStream_t st)
LBM_DECLARE_TILE_GENERAL(launch_tile_general_f32_a);
LBM_DECLARE_TILE_GENERAL(launch_tile_general_f32_b);
LBM_DECLARE_TILE_GENERAL(launch_tile_general_f64_a);
LBM_DECLARE_TILE_GENERAL(launch_tile_general_f64_b);
#undef LBM_DECLARE_TILE_GENERAL
cudaError_t launch_tile_f32_const(const lbm_solver *s, int src, int steps, bool prepare, cudaStream_t st);
cudaError_t launch_tile_f32_kfield(const lbm_solver *s, int src, int steps, bool prepare, cudaStream_t st);
cudaError_t launch_tile_f64_const(const lbm_solver *s, int src, int steps, bool prepare, cudaStream_t st);
cudaError_t launch_tile_f64_kfield(const lbm_solver *s, int src, int steps, bool prepare, cudaStream_t st);
bool step_v4_supported(const lbm_solver *s);
bool step_v4_preferred(const lbm_solver *s);
cudaError_t launch_step_v4(const lbm_solver *s, int src, cudaStream_t st);
cudaError_t launch_get_phi(const lbm_solver *s, void *out, int out_prec, cudaStream_t st);
cudaError_t launch_reduce(const lbm_solver *s, const double *ref, double *out, cudaStream_t st);
cudaError_t launch_kfield(const lbm_solver *s, const double *K, cudaStream_t st);
// the eight deterministic FP64 statistics of a plain FP64 field (partials:
// kReduceBlocks * 8 doubles)
cudaError_t launch_reduce_field(const double *field, long long n, const double *ref, double *partials, double *out,
                                cudaStream_t st);

int adjoint_blocks(const lbm_solver *s);
cudaError_t launch_adjoint_begin(const lbm_solver *s, const void *dphi, int in_prec, void *lam, cudaStream_t st);
cudaError_t launch_adjoint_step(const lbm_solver *s, const void *F, const void *lam_in, void *lam_out, double *gA,
                                double *partials, cudaStream_t st);
cudaError_t launch_adjoint_end(const lbm_solver *s, const void *phi0, int in_prec, const void *lam, const double *gA,
                               double *dphi0, double *dK, double *du, double *partials, cudaStream_t st);

}  // namespace lbm
