// kernels_tile_general.cuh -- several time steps per launch for small lattices of the
// general path: Scheme A (Remark II) or B, the power-law flux, affine and Fisher
// sources, the tensor diffusion function, and periodic, anti-bounce-back or
// extrapolated walls with a Dirichlet record per step. The tiles are those of
// kernels_tile.cuh, one node per lane; Scheme A's phi(t_n) is a tenth plane of the
// region. An extrapolated node takes its inward neighbour's pull, two nodes inward at
// most: tiles are at least two nodes wide and high, and the last one of an axis ends at
// its last node (it overlaps its neighbour and writes the shared nodes with the same
// values). One body serves all steps of a launch, so that a state does not depend on
// how a call is split into launches.
//
// What bounds it: the latency of a step's chain on a nearly empty SM. 301^2 FP32
// (Burgers-Fisher, 400 steps): 2474 -> 1513 us against two-step 30 x 30 tiles, of which
// there are 121 for 152 SMs.
#pragma once

#include "kernels_general.cuh"
#include "kernels_tile.cuh"

namespace lbm {

constexpr int kTileGThreads = 512;
template <class R> constexpr int kTileGPlane = kTileSmem / (20 * (int)sizeof(R));

template <class R>
struct TileGArgs {
    Params<R> p;
    const R *src, *src_phi;
    R *dst, *dst_phi;
    const double *records;
    const long long *rec_cnt;
    int nrec, rec_off;
    int W, H, T;
};

template <class R, int CONV, int DIFF, bool SA>
__global__ void __launch_bounds__(kTileGThreads, 1)
k_tile_g(const __grid_constant__ TileGArgs<R> a)
{
    extern __shared__ __align__(16) unsigned char sm_g[];
    constexpr int PS = kTileGPlane<R>;
    const Params<R> &p = a.p;
    const int T = a.T, RX = a.W + 2 * (T - 1), X0 = min((int)blockIdx.x * a.W, p.nx - a.W), Y0 = min((int)blockIdx.y * a.H, p.ny - a.H);
    R *buf = reinterpret_cast<R *>(sm_g) + kTilePad / 2;
    const unsigned inv = 0xffffffffu / (unsigned)RX + 1;
    for (int l = 1; l <= T; ++l) {
        const R *in = buf + (l & 1) * 10 * PS;
        R *out = buf + ((l & 1) ^ 1) * 10 * PS;
        const int ilo = l - 1, ihi = a.W + 2 * (T - 1) - (l - 1), jhi = a.H + 2 * (T - 1) - (l - 1);
        for (int n = ilo * RX + threadIdx.x; n < jhi * RX; n += blockDim.x) {
            const int j = (int)__umulhi((unsigned)n, inv), i = n - j * RX;
            if (i < ilo || i >= ihi) continue;
            int x = X0 - (T - 1) + i, y = Y0 - (T - 1) + j;
            if ((p.abb_x || p.nee_x) && (x < 0 || x >= p.nx)) continue;      // no such node
            if ((p.abb_y || p.nee_y) && (y < 0 || y >= p.ny)) continue;
            if ((unsigned)x >= (unsigned)p.nx) x = tile_wrap(x, p.nx);
            if ((unsigned)y >= (unsigned)p.ny) y = tile_wrap(y, p.ny);
            LBM_CHK(x, p.nx, p.err, kErrX);
            LBM_CHK(y, p.ny, p.err, kErrY);
            const long long own = (long long)y * p.pitch + x;
            const bool ex = p.nee_x && (x == 0 || x == p.nx - 1), ey = p.nee_y && (y == 0 || y == p.ny - 1);
            // the node whose pull this one takes: itself, or its inward neighbour
            const int dx = ex ? (x == 0 ? 1 : -1) : 0, dy = ey ? (y == 0 ? 1 : -1) : 0;
            R f[9], prev = R(0);
            if (l == 1) {
                pull_wrap<sizeof(R) == 8 ? LBM_F64 : LBM_F32>(p, a.src, x + dx, y + dy, f);
                if (SA) prev = a.src_phi[own];
            } else {
                const int c = (j + dy) * RX + i + dx;
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    int s = c - cy(k) * RX - cx(k);
                    LBM_CHK(s, PS, p.err, kErrShared);
                    f[k] = in[k * PS + s];
                }
                if (SA) prev = in[9 * PS + j * RX + i];
            }
            if (ex || ey) {
                R sum = f[0];
#pragma unroll
                for (int k = 1; k < 9; ++k) sum += f[k];
                const R phif = SA ? sum : (sum + p.half_r0) * p.inv_den;
                const double *bv = record_of(a.records, a.rec_cnt, a.nrec, 2 * (p.nx + p.ny), a.rec_off + l - 1);
                const double vb = ex ? bv[x == 0 ? y : p.ny + y] : bv[2 * p.ny + (y == 0 ? x : p.nx + x)];
                R eb[9], ef[9];
                feq_stored<R, CONV, DIFF, SA>(p, (R)vb, eb);
                feq_stored<R, CONV, DIFF, SA>(p, phif, ef);
#pragma unroll
                for (int k = 0; k < 9; ++k) f[k] = eb[k] + (f[k] - ef[k]);
            } else if ((p.abb_x && (x == 0 || x == p.nx - 1)) || (p.abb_y && (y == 0 || y == p.ny - 1))) {
#pragma unroll
                for (int k = 1; k < 9; ++k) {
                    const int xs = x - cx(k), ys = y - cy(k);
                    const bool ox = p.abb_x && (xs < 0 || xs >= p.nx), oy = p.abb_y && (ys < 0 || ys >= p.ny);
                    if (ox || oy) {
                        const R wx = xs < 0 ? p.phi_wall[0] : p.phi_wall[1], wy = ys < 0 ? p.phi_wall[2] : p.phi_wall[3];
                        const R phiw = (ox && oy) ? R(0.5) * (wx + wy) : (ox ? wx : wy);
                        const R back = l == 1 ? __ldg(a.src + opp(k) * p.plane + own) : in[opp(k) * PS + j * RX + i];
                        f[k] = wall_term<R, CONV, DIFF>(p, k, phiw) - back;
                    }
                }
            }
            R A3 = p.A3, A35 = p.A35, A5 = p.A5, phi;
            if (p.Afield) {
                A3 = __ldg(p.Afield + own);
                A35 = __ldg(p.Afield + p.plane + own);
                A5 = __ldg(p.Afield + 2 * p.plane + own);
            }
            if (SA) collide_a<R, CONV, DIFF>(p, f, A3, A35, A5, prev, phi);
            else collide<R, CONV, DIFF>(p, f, A3, A35, A5, phi);
            if (l < T) {
                R *o = out + j * RX + i;
#pragma unroll
                for (int k = 0; k < 9; ++k) o[k * PS] = f[k];
                if (SA) o[9 * PS] = phi;
            } else {
#pragma unroll
                for (int k = 0; k < 9; ++k) a.dst[k * p.plane + own] = f[k];
                if (SA) a.dst_phi[own] = phi;
            }
        }
        __syncthreads();
    }
}

template <class R, int CONV, int DIFF, bool SA>
static cudaError_t tile_g_t(const lbm_solver *s, int src, const double *records, int steps, bool prepare, cudaStream_t st)
{
    static SmemOptIn once;
    const cudaError_t e = opt_in_smem((const void *)k_tile_g<R, CONV, DIFF, SA>, kTileSmem, once);
    if (e != cudaSuccess || prepare) return e;
    TileGArgs<R> a;
    a.p = make_params<R>(s);
    a.src = (const R *)s->pop[src];
    a.src_phi = (const R *)s->phi[src];
    a.dst = (R *)s->pop[src ^ 1];
    a.dst_phi = (R *)s->phi[src ^ 1];
    a.records = records;
    a.rec_cnt = s->dir_counter;
    a.nrec = s->dir_nrec;
    a.rec_off = s->dir_off;
    a.W = s->plan.W;
    a.H = s->plan.H;
    a.T = steps;
    int threads = kTileGThreads;
    if (sizeof(R) == 4 && steps == 1) {
        // a single FP32 step needs no halo and is bound by latency: a node per thread, six to
        // eight blocks per SM (400^2 6.2 us against 7.9 over the plan's tiles, one block per SM)
        a.W = std::min(32, s->d.nx);
        a.H = std::min(4, s->d.ny);
        threads = 128;
    }
    const dim3 grid((s->d.nx + a.W - 1) / a.W, (s->d.ny + a.H - 1) / a.H);
    k_tile_g<R, CONV, DIFF, SA><<<grid, threads, steps > 1 ? kTileSmem : 0, st>>>(a);
    return cudaGetLastError();
}

// families of the general path but the C-free variant
#define LBM_TILE_G_CASES(R, SA)                                                                   \
    switch (s->c.conv * 4 + s->c.diff) {                                                          \
    case 0: return tile_g_t<R, 0, 0, SA>(s, src, records, steps, prepare, st);                    \
    case 1: return tile_g_t<R, 0, 1, SA>(s, src, records, steps, prepare, st);                    \
    case 2: return tile_g_t<R, 0, 2, SA>(s, src, records, steps, prepare, st);                    \
    case 3: return tile_g_t<R, 0, 3, SA>(s, src, records, steps, prepare, st);                    \
    case 4: return tile_g_t<R, 1, 0, SA>(s, src, records, steps, prepare, st);                    \
    case 5: return tile_g_t<R, 1, 1, SA>(s, src, records, steps, prepare, st);                    \
    case 6: return tile_g_t<R, 1, 2, SA>(s, src, records, steps, prepare, st);                    \
    case 7: return tile_g_t<R, 1, 3, SA>(s, src, records, steps, prepare, st);                    \
    case 8: return tile_g_t<R, 2, 0, SA>(s, src, records, steps, prepare, st);                    \
    case 9: return tile_g_t<R, 2, 1, SA>(s, src, records, steps, prepare, st);                    \
    case 10: return tile_g_t<R, 2, 2, SA>(s, src, records, steps, prepare, st);                   \
    case 11: return tile_g_t<R, 2, 3, SA>(s, src, records, steps, prepare, st);                   \
    }                                                                                             \
    return cudaErrorInvalidValue;

}  // namespace lbm
