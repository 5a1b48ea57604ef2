// kernels_tile.cuh -- up to kTileMaxT fused time steps per launch for small lattices
// (Scheme B): FP64, and FP32 with two x-adjacent nodes per packed instruction. FP64
// lattices too large for a second step per launch take it too, one step per launch
// (route.cu has both sides measured).
//
// A launch on a small lattice costs more than its arithmetic: the host's part, the
// gap to the next launch and the latency of the pulls. Here a block owns a W x H
// tile and recomputes a halo of T - 1 nodes around it, so that T steps need no
// exchange: step 1 pulls the region from global memory (L2), the following ones
// pull from shared memory (two buffers in turn, one barrier per step) and shrink
// by one node a side, the last one writes the tile. The tile count is made to fit
// the SMs, and T and the tile to the least estimated time (tile_plan).
//
// What bounds it: FP32, the latency of a step's chain (barrier, pulls, collision)
// and of the first pulls; FP64, the pipe, whose quarter of an SM takes a warp's
// collision 2.2 us. Measured (GB300, us per step, before -> now): FP32 100^2 3.5 ->
// 1.06, 200^2 3.6 -> 1.31, 400^2 4.14 -> 2.18 (one step per launch 5.4); FP64 128^2
// 8.28 -> 5.21, 64^2 8.28 -> 3.50. With each item on a thread of its own path (early
// exits, wall branches) the 400^2 took 2.59.
#pragma once

#include <algorithm>

#include "lbm_internal.h"

namespace lbm {

template <class R> struct TileVec;                   // arithmetic type and nodes per item
template <> struct TileVec<float> { using V = F2; static constexpr int N = 2, kThreads = 768; };
template <> struct TileVec<double> { using V = double; static constexpr int N = 1, kThreads = 512; };

template <class R>
struct TileArgs {
    Coll<typename TileVec<R>::V> k;
    const R *src;
    R *dst;
    const R *Afield;
    long long plane, pitch;
    int nx, ny, W, H, T;
    int abb_x, abb_y, has_src;
    R wt[8][3];
    int *err;
};

// shared memory: two buffers of nine planes, 225 KB; a plane has room for a column
// either side of the region
constexpr int kTileSmem = 230400, kTilePad = 4;
template <class R> constexpr int kTilePlane = kTileSmem / (18 * (int)sizeof(R));

// region of a tile: RX columns (a multiple of the nodes per item), RY rows
template <class R> __host__ __device__ __forceinline__ int tile_rx(int W, int T)
{
    constexpr int N = TileVec<R>::N;
    const int rx = (W + 2 * (T - 1) + N - 1) / N * N;
    return rx < 2 * N ? 2 * N : rx;                  // two items a row at least: the division by a multiply
}

__device__ __forceinline__ int tile_wrap(int v, int n)
{
    v %= n;
    return v < 0 ? v + n : v;
}

__device__ __forceinline__ double part(double v, int) { return v; }
__device__ __forceinline__ float part(F2 v, int h) { return h ? v.v.y : v.v.x; }
__device__ __forceinline__ void set_part(double &v, int, double a) { v = a; }
__device__ __forceinline__ void set_part(F2 &v, int h, float a) { (h ? v.v.y : v.v.x) = a; }

// Step l of a block's tile. FIRST: pulls from global memory, else from the region
// `in` left by step l - 1; the last step writes the tile, the others the region `out`.
// WALLS: the block has nodes at anti-bounce-back walls (a branch to them would make
// every item move its populations to the registers where the branches meet). All
// lanes of a warp run every item, those without one on the last cell: in convergent
// code the collision's constants come from uniform registers.
template <class R, int CONV, int DIFF, bool KF, bool WALLS, bool FIRST>
__device__ __forceinline__ void tile_step(const TileArgs<R> &a, int l, const R *in, R *out, int X0, int Y0, int RX,
                                          int per_row, unsigned inv, int warp, int lane)
{
    using V = typename TileVec<R>::V;
    constexpr int N = TileVec<R>::N, kThreads = TileVec<R>::kThreads, PS = kTilePlane<R>;
    const int T = a.T, X1 = min(X0 + a.W, a.nx), Y1 = min(Y0 + a.H, a.ny);    // outputs [X0, X1) x [Y0, Y1)
    // the nodes this step is for: the tile and T - l around it
    const int ilo = l - 1, ihi = X1 - X0 + 2 * (T - 1) - (l - 1), jlo = l - 1, jhi = Y1 - Y0 + 2 * (T - 1) - (l - 1);
    const int end = jhi * per_row;
    for (int base = jlo * per_row + warp * 32; base < end; base += kThreads) {
        const int n = min(base + lane, end - 1);
        const int j = (int)__umulhi((unsigned)n, inv), i = (n - j * per_row) * N;   // region cell
        const int x = X0 - (T - 1) + i, y = Y0 - (T - 1) + j;
        bool mine = base + lane < end && i + N > ilo && i < ihi;
        if (WALLS) {                                                // nodes beyond a wall do not exist
            if (a.abb_y) mine = mine && y >= 0 && y < a.ny;
            if (a.abb_x) mine = mine && x + N > 0 && x < a.nx;
        }
        int xw[N] = {}, yw = 0;
        if (FIRST || KF) {
            yw = a.abb_y ? min(max(y, 0), a.ny - 1) : tile_wrap(y, a.ny);
#pragma unroll
            for (int h = 0; h < N; ++h) {
                xw[h] = a.abb_x ? min(max(x + h, 0), a.nx - 1) : tile_wrap(x + h, a.nx);
                LBM_CHK(xw[h], a.nx, a.err, kErrX);
            }
            LBM_CHK(yw, a.ny, a.err, kErrY);
        }
        V g[9];
        const R *s0 = in + j * RX + i;
        if (FIRST) {
            const int ym = yw == 0 ? (a.abb_y ? 0 : a.ny - 1) : yw - 1, yp = yw == a.ny - 1 ? (a.abb_y ? yw : 0) : yw + 1;
            const long long row[3] = {ym * a.pitch, yw * a.pitch, yp * a.pitch};
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const R *s = a.src + k * a.plane + row[1 - cy(k)];
#pragma unroll
                for (int h = 0; h < N; ++h) {
                    int xs = xw[h] - cx(k);
                    if (cx(k) > 0) xs = xs < 0 ? (a.abb_x ? 0 : a.nx - 1) : xs;
                    if (cx(k) < 0) xs = xs >= a.nx ? (a.abb_x ? a.nx - 1 : 0) : xs;
                    set_part(g[k], h, __ldg(s + xs));
                }
            }
        } else {
            // (what lies beyond a row's ends goes to nodes that no later step uses)
            const R *sr[3] = {s0 - RX, s0, s0 + RX};
#pragma unroll
            for (int k = 0; k < 9; ++k) {
                const R *s = sr[1 - cy(k)] + k * PS - cx(k);
                if constexpr (N == 2) {
                    if (cx(k) == 0) g[k] = F2(*reinterpret_cast<const float2 *>(s));
                    else g[k] = F2(s[0], s[1]);
                } else {
                    g[k] = s[0];
                }
            }
        }
        if (WALLS) {
            const bool south = a.abb_y && y == 0, north = a.abb_y && y == a.ny - 1;
#pragma unroll
            for (int h = 0; h < N; ++h) {
                const bool west = a.abb_x && x + h == 0, east = a.abb_x && x + h == a.nx - 1;
                if (west || east || south || north) {
#pragma unroll
                    for (int k = 1; k < 9; ++k) {
                        const bool ox = cx(k) != 0 && (cx(k) > 0 ? west : east);
                        const bool oy = cy(k) != 0 && (cy(k) > 0 ? south : north);
                        if (ox || oy) {
                            const R own = FIRST ? __ldg(a.src + opp(k) * a.plane + yw * a.pitch + xw[h]) : s0[opp(k) * PS + h];
                            set_part(g[k], h, vsub(a.wt[k - 1][(ox ? 1 : 0) + (oy ? 2 : 0) - 1], own));
                        }
                    }
                }
            }
        }
        V A3 = V(0.f), A35 = V(0.f), A5 = V(0.f), phi;
        if constexpr (KF) {
#pragma unroll
            for (int h = 0; h < N; ++h) {
                const long long o = yw * a.pitch + xw[h];
                set_part(A3, h, __ldg(a.Afield + o));
                set_part(A35, h, __ldg(a.Afield + a.plane + o));
                set_part(A5, h, __ldg(a.Afield + 2 * a.plane + o));
            }
        }
        relax<V, CONV, DIFF, KF>(a.k, a.has_src != 0, g, A3, A35, A5, phi);
        if (l < T) {
            R *o = out + j * RX + i;
            if (mine) {
#pragma unroll
                for (int k = 0; k < 9; ++k) {
                    if constexpr (N == 2) *reinterpret_cast<float2 *>(o + k * PS) = g[k].v;
                    else o[k * PS] = g[k];
                }
            }
        } else {
            R *o = a.dst + y * a.pitch + x;
#pragma unroll
            for (int h = 0; h < N; ++h)
                if (mine && x + h >= X0 && x + h < X1) {
#pragma unroll
                    for (int k = 0; k < 9; ++k) o[k * a.plane + h] = part(g[k], h);
                }
        }
    }
}

template <class R, int CONV, int DIFF, bool KF, bool WALLS>
__device__ __forceinline__ void tile_steps(const TileArgs<R> &a, R *buf, int X0, int Y0)
{
    constexpr int N = TileVec<R>::N, PS = kTilePlane<R>;
    const int T = a.T, RX = tile_rx<R>(a.W, T), per_row = RX / N;
    const unsigned inv = 0xffffffffu / (unsigned)per_row + 1;           // n / per_row by a multiply (n < 2^16)
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    tile_step<R, CONV, DIFF, KF, WALLS, true>(a, 1, buf, buf, X0, Y0, RX, per_row, inv, warp, lane);
    for (int l = 2; l <= T; ++l) {
        __syncthreads();
        R *in = buf + (l & 1) * 9 * PS, *out = buf + ((l & 1) ^ 1) * 9 * PS;
        tile_step<R, CONV, DIFF, KF, WALLS, false>(a, l, in, out, X0, Y0, RX, per_row, inv, warp, lane);
    }
}

template <class R, int CONV, int DIFF, bool KF>
__global__ void __launch_bounds__(TileVec<R>::kThreads, 1)
k_tile(const __grid_constant__ TileArgs<R> a)
{
    extern __shared__ __align__(16) unsigned char sm_t[];
    R *buf = reinterpret_cast<R *>(sm_t) + kTilePad / 2;
    const int X0 = blockIdx.x * a.W, Y0 = blockIdx.y * a.H;
    const bool walls = (a.abb_x && (X0 - a.T <= 0 || X0 + a.W + a.T >= a.nx)) ||
                       (a.abb_y && (Y0 - a.T <= 0 || Y0 + a.H + a.T >= a.ny));
    if (walls) tile_steps<R, CONV, DIFF, KF, true>(a, buf, X0, Y0);
    else tile_steps<R, CONV, DIFF, KF, false>(a, buf, X0, Y0);
}

template <class R, int CONV, int DIFF, bool KF>
static cudaError_t tile_t(const lbm_solver *s, int src, int steps, bool prepare, cudaStream_t st)
{
    static SmemOptIn once;
    const cudaError_t e = opt_in_smem((const void *)k_tile<R, CONV, DIFF, KF>, kTileSmem, once);
    if (e != cudaSuccess || prepare) return e;
    const Params<R> &p = make_params<R>(s);
    TileArgs<R> a;
    a.k = coll_cast<typename TileVec<R>::V>(p.k);
    a.src = (const R *)s->pop[src];
    a.dst = (R *)s->pop[src ^ 1];
    a.Afield = p.Afield;
    a.plane = p.plane;
    a.pitch = p.pitch;
    a.nx = p.nx;
    a.ny = p.ny;
    a.W = s->plan.W;
    a.H = s->plan.H;
    a.T = steps;
    a.abb_x = p.abb_x;
    a.abb_y = p.abb_y;
    a.has_src = p.has_src;
    for (int k = 0; k < 8; ++k)
        for (int z = 0; z < 3; ++z) a.wt[k][z] = p.wt[k][z];
    a.err = p.err;
    const dim3 grid((a.nx + a.W - 1) / a.W, (a.ny + a.H - 1) / a.H);
    k_tile<R, CONV, DIFF, KF><<<grid, TileVec<R>::kThreads, steps > 1 ? kTileSmem : 0, st>>>(a);
    return cudaGetLastError();
}

#define LBM_TILE_FAMILIES(R, KF)                                                       \
    switch (step_key(s)) {                                                             \
    case 0: return tile_t<R, 0, 0, KF>(s, src, steps, prepare, st);                    \
    case 1: return tile_t<R, 0, 1, KF>(s, src, steps, prepare, st);                    \
    case 2: return tile_t<R, 0, 2, KF>(s, src, steps, prepare, st);                    \
    case 3: return tile_t<R, 1, 0, KF>(s, src, steps, prepare, st);                    \
    case 4: return tile_t<R, 1, 1, KF>(s, src, steps, prepare, st);                    \
    case 5: return tile_t<R, 1, 2, KF>(s, src, steps, prepare, st);                    \
    case 6: return tile_t<R, kConvNone, 0, KF>(s, src, steps, prepare, st);            \
    case 7: return tile_t<R, kConvNone, 1, KF>(s, src, steps, prepare, st);            \
    case 8: return tile_t<R, kConvNone, 2, KF>(s, src, steps, prepare, st);            \
    }                                                                                  \
    return cudaErrorInvalidValue;

}  // namespace lbm
