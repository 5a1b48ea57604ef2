// kernels_march.cuh -- T fused stream-collide time steps (Eq. 34) per sweep
// through HBM for large FP32 grids: a systolic march of warps down a strip.
//
// A block owns a strip of 64 P KW columns and walks down its rows. Its warps are
// split into T levels of KW warps: level l holds the state after step l + 1, one
// row per iteration; a lane owns P pairs of x-adjacent nodes, each pair collided
// in packed FP32x2 arithmetic. Level 0 takes its rows from a staging area that
// asynchronous copies fill a few rows ahead, level T - 1 writes to global memory,
// and the levels between pass their rows through shared memory: each keeps a ring
// of the last four rows it finished. A row of level l needs the rows above and
// below it from level l - 1, so level l runs two rows behind level l - 1; then all
// levels of an iteration are independent and one barrier per iteration is enough.
//
// Cost: every population is read and written once per T steps (18 B per update
// for T = 4 in FP32). The strip gives up T - 1 columns on either side, and writes a
// multiple of four columns (120 of 128), and a chunk of H rows takes H + 3 (T - 1) iterations to
// fill and drain, in which the other blocks of the SM run.
//
// Alignment: level l's pairs start one column right of level l - 1's, so a pull
// with c_x != 0 always meets an aligned pair, and the pairs written by every level
// are aligned too. The pulls with c_x = 0 straddle two pairs; those three planes
// keep their even and odd columns apart, so that neither side has bank conflicts.
//
// What bounds it, 4096^2 FP32 with walls (GB300): warps wait for one another at the
// barrier and on their own dependent instructions (issue slots 55 %, FMA pipe 46 %
// busy, DRAM 53 %); 218,500 MLUPS against 149,500 of the two-step pair tiles, whose
// HBM traffic per update is twice as large. Measured on the way, same grid: level 0
// loading straight from global memory 150k (its latency is on every iteration's
// path), two pairs per lane with half the warps 209k, three blocks per SM with a
// deeper staging area 201k, strips of 64 columns 213k, six steps per sweep 152k.
#pragma once

#include <type_traits>

#include "lbm_internal.h"

namespace lbm {

struct MarchArgs {
    Coll<F2> k;
    const float *src;
    float *dst;
    const float *Afield;       // per-node blocks or null
    long long plane;
    int pitch, nx, ny;
    int H, strips, chunks;     // rows per block; blocks = strips x chunks
    int abb_x, abb_y;
    float wt[8][3];            // wall terms (Params)
    int has_src;
    int give_up;               // 1: level 0 takes its first row for late (a test of what follows)
    int *err;
};

// The one shape in use: four steps per sweep, strips of 128 columns, two warps per
// level, two staged rows; 64 registers and 55 KB of shared memory, four blocks per SM.
constexpr int kMarchT = 4, kMarchKW = 2, kMarchP = 1, kMarchStage = 2;

template <int T, int KW, int P, int STAGE> struct March {
    static constexpr int kThreads = 32 * KW * T;
    static constexpr int kW = 64 * P * KW, kPairs = kW / 2;
    // output columns: a multiple of 4, so that every strip's copies start on a 16-byte boundary
    static constexpr int kOut = (kW - 2 * (T - 1)) & ~3;
    // ring of a level: the planes with c_y = 1 keep four rows, the others three
    static constexpr int kRing = 30 * kW;
    // level 0's input: kStage rows of the nine planes, one pair wider, rounded to 16 bytes
    static constexpr int kStage = STAGE, kInW = kW + 4, kInSlot = 9 * kInW;
    static constexpr unsigned kInBytes = kInSlot * sizeof(float);
    static constexpr int kBars = 2 * STAGE;                            // floats taken by the mbarriers
    static constexpr int kSmem = ((T - 1) * kRing + kStage * kInSlot + kBars) * (int)sizeof(float);
    static_assert(T % 4 == 0, "the first column of a strip's copies is X0 - T");
};

__device__ __forceinline__ void march_bar_init(unsigned bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void march_expect(unsigned bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_copy(unsigned to, const float *from, unsigned bytes, unsigned bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(to),
                 "l"(from), "r"(bytes), "r"(bar)
                 : "memory");
}
// bounded wait for phase `parity`; false when the limit ran out
__device__ __forceinline__ bool march_wait(unsigned bar, unsigned parity, unsigned polls = 1u << 20)
{
    for (unsigned i = 0; i < polls; ++i) {
        unsigned done;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done)
                     : "r"(bar), "r"(parity)
                     : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void march_barrier(int threads) { asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory"); }

__device__ __forceinline__ void copy4(unsigned to, const float *from)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(to), "l"(from) : "memory");
}

__device__ __forceinline__ int wrap_index(int v, int n)
{
    v %= n;
    return v < 0 ? v + n : v;
}

// A ring's planes by c_y: first float of the class and place within it.
__device__ constexpr int ring_place(int k)
{
    return k < 5 ? (k == 0 || k == 2 || k == 4 ? 0 : (k == 1 ? 1 : 2)) : (k == 5 || k == 7 ? 1 : 2);
}
__device__ constexpr int ring_plane(int k, int w)
{
    return cy(k) > 0 ? 4 * ring_place(k) * w : (cy(k) == 0 ? (12 + 3 * ring_place(k)) * w : (21 + 3 * ring_place(k)) * w);
}
__device__ __forceinline__ int ring_next(int off, int rows, int w) { return off == (rows - 1) * w ? 0 : off + w; }

// Pair q's pull from a row of plane K, w columns wide (columns 2q + 1 - c_x and the
// next), the write of pair q, and the single column 2q + 1 + h.
template <int K> __device__ __forceinline__ F2 ring_pull(const float *row, int w, int q)
{
    if (cx(K) == 0) return F2(row[w / 2 + q], row[q + 1]);
    return F2(*reinterpret_cast<const float2 *>(row + 2 * q + 1 - cx(K)));
}
template <int K> __device__ __forceinline__ void ring_put(float *row, int w, int q, F2 v)
{
    if (cx(K) == 0) {
        row[q] = v.v.x;
        row[w / 2 + q] = v.v.y;
    } else {
        *reinterpret_cast<float2 *>(row + 2 * q) = v.v;
    }
}
__device__ __forceinline__ float ring_own(const float *row, int w, int q, int k, int h)
{
    if (cx(k) == 0) return h ? row[q + 1] : row[w / 2 + q];
    return row[2 * q + 1 + h];
}

template <int K = 0, class F> __device__ __forceinline__ void each_k(F f)
{
    f(std::integral_constant<int, K>());
    if constexpr (K < 8) each_k<K + 1>(f);
}

// One strip. EDGE: it touches the edges of the grid -- `cols`, its columns wrap or meet
// walls; `rows`, it has rows at anti-bounce-back walls.
template <int CONV, int DIFF, int SRC, bool KF, int T, int KW, int P, int ST, bool EDGE>
__device__ __forceinline__ void march_strip(const MarchArgs &a, const Coll<F2> &kc, float *sm, int X0, int Y0, int Y1,
                                            bool cols, bool rows)
{
    using M = March<T, KW, P, ST>;
    if (!EDGE) cols = rows = false;
    // (the shuffle tells the compiler that a warp takes one branch: the constants then sit in
    // uniform registers, where packed instructions read them)
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int lev = warp / KW, q0 = (warp - lev * KW) * 32 * P + lane;  // pairs q0 + 32 p
    const int xa = X0 - (T - 1) + lev + 2 * q0;         // columns xa + 64 p, xa + 64 p + 1
    // rows of this level
    int lo = Y0 - (T - 1 - lev), hi = Y1 - 1 + (T - 1 - lev);
    if (rows) {
        lo = max(lo, 0);
        hi = min(hi, a.ny - 1);
    }
    const int n_it = (Y1 - Y0) + 3 * (T - 1);
    const int r_first = Y0 - (T - 1) - 2 * lev;          // row of iteration 0
    float *stage = sm + (T - 1) * M::kRing;
    float *bars = stage + M::kStage * M::kInSlot;

    if (threadIdx.x == 0) {
        for (int j = 0; j < M::kStage; ++j) march_bar_init((unsigned)__cvta_generic_to_shared(bars + 2 * j));
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    march_barrier(M::kThreads);

    // the x-wall node of pair p, if any: side 1 west, -1 east, node wh
    auto xwall = [&](int p, int &side, int &wh) {
        const int x = xa + 64 * p;
        side = (x == 0 || x + 1 == 0) ? 1 : ((x == a.nx - 1 || x + 1 == a.nx - 1) ? -1 : 0);
        wh = (x == 0 || x == a.nx - 1) ? 0 : 1;
    };
    // anti-bounce-back of the pair's wall nodes; own(k, h): the node's population k before the step
    auto walls = [&](int r, int p, F2 g[9], auto own) {
        const bool south = a.abb_y && r == 0, north = a.abb_y && r == a.ny - 1;
        if (south || north) {
#pragma unroll
            for (int k = 1; k < 9; ++k)
                if (cy(k) != 0 && (cy(k) > 0 ? south : north))
                    g[k] = F2(__fsub_rn(a.wt[k - 1][1], own(opp(k), 0)), __fsub_rn(a.wt[k - 1][1], own(opp(k), 1)));
        }
        int side = 0, wh = 0;
        if (cols && a.abb_x) xwall(p, side, wh);
        if (side != 0) {
#pragma unroll
            for (int k = 1; k < 9; ++k) {
                if (cx(k) != 0 && cx(k) == side) {
                    const bool both = cy(k) != 0 && (cy(k) > 0 ? south : north);
                    const float v = __fsub_rn(both ? a.wt[k - 1][2] : a.wt[k - 1][0], own(opp(k), wh));
                    if (wh == 0) g[k].v.x = v;
                    else g[k].v.y = v;
                }
            }
        }
    };
    auto step = [&](int r, int p, F2 g[9]) {
        F2 A3, A35, A5, ph;
        if constexpr (KF) {
            const unsigned row = (unsigned)wrap_index(r, a.ny) * (unsigned)a.pitch;
            const unsigned i0 = row + wrap_index(xa + 64 * p, a.nx), i1 = row + wrap_index(xa + 64 * p + 1, a.nx);
            A3 = F2(__ldg(a.Afield + i0), __ldg(a.Afield + i1));
            A35 = F2(__ldg(a.Afield + a.plane + i0), __ldg(a.Afield + a.plane + i1));
            A5 = F2(__ldg(a.Afield + 2 * a.plane + i0), __ldg(a.Afield + 2 * a.plane + i1));
        }
        relax<F2, CONV, DIFF, KF, SRC>(kc, a.has_src != 0, g, A3, A35, A5, ph);
    };

    // Level 0's input. The nine planes' rows that row r pulls from (columns X0 - T and on) are
    // copied into slot (r - first row) % kStage, kStage - 1 iterations ahead, by the first warp of
    // level 1: one bulk copy per plane from lanes 0 to 8. With `cols` the bulk copies take the part
    // of the row that lies in the grid, in whole 16 bytes, and the few columns left of column 0 or
    // from the last full 16 bytes on (wrapped when x is periodic; behind a wall no node keeps
    // them) are copied one by one.
    const unsigned stage_s = (unsigned)__cvta_generic_to_shared(stage), bars_s = (unsigned)__cvta_generic_to_shared(bars);
    auto source_row = [&](int r, int cyk) {
        int y = r - cyk;
        if (rows) y = min(max(y, 0), a.ny - 1);
        else y = y < 0 ? y + a.ny : (y >= a.ny ? y - a.ny : y);
        LBM_CHK(y, a.ny, a.err, kErrY);
        return (unsigned)y * (unsigned)a.pitch;
    };
    const int w4 = M::kW;
    int s4 = 0, s3 = 0;                                  // this iteration's row in the rings, in floats

    if (lev == 0) {
        auto column = [&](int x) { return a.abb_x ? min(max(x, 0), a.nx - 1) : wrap_index(x, a.nx); };
        unsigned phases = 0;                             // bit j: the phase slot j's next row completes
        int use = 0, i = 0, r = r_first;
        const int n_run = a.give_up ? 0 : n_it;
        march_barrier(M::kThreads);
        for (; i < n_run; ++i, ++r) {
            if (r >= lo && r <= hi) {
                if (!march_wait(bars_s + 8 * use, (phases >> use) & 1)) break;
                phases ^= 1u << use;
                const float *in = stage + use * M::kInSlot + 2 * q0 + 1;
                F2 g[P][9];
#pragma unroll
                for (int p = 0; p < P; ++p)
                    each_k([&](auto K) {
                        const float *s = in + K * M::kInW + 64 * p - cx(K);
                        if (cx(K) == 0) g[p][K] = F2(s[0], s[1]);
                        else g[p][K] = F2(*reinterpret_cast<const float2 *>(s));
                    });
                if (EDGE) {
                    const unsigned own = source_row(r, 0);
#pragma unroll
                    for (int p = 0; p < P; ++p)
                        walls(r, p, g[p], [&](int k, int h) {
                            return __ldg(a.src + k * a.plane + own + column(xa + 64 * p + h));
                        });
                }
#pragma unroll
                for (int p = 0; p < P; ++p) step(r, p, g[p]);
#pragma unroll
                for (int p = 0; p < P; ++p)
                    each_k([&](auto K) {
                        ring_put<K>(sm + (cy(K) > 0 ? s4 : s3) + ring_plane(K, w4), w4, q0 + 32 * p, g[p][K]);
                    });
            }
            use = use == M::kStage - 1 ? 0 : use + 1;
            s4 = ring_next(s4, 4, w4);
            s3 = ring_next(s3, 3, w4);
            march_barrier(M::kThreads);
        }
        if (i < n_it && lane == 0) atomicOr(a.err, 16);  // a copy did not arrive in time
        for (; i < n_it; ++i, ++r) {                     // no result from what is not there: NaN from here on
            if (r >= lo && r <= hi) {                    // (the copies still end before their slots are filled again)
                march_wait(bars_s + 8 * use, (phases >> use) & 1, 1u << 12);
                phases ^= 1u << use;
            }
            for (int p = 0; p < P; ++p)
                each_k([&](auto K) {
                    ring_put<K>(sm + (cy(K) > 0 ? s4 : s3) + ring_plane(K, w4), w4, q0 + 32 * p, F2(__int_as_float(0x7fffffff)));
                });
            use = use == M::kStage - 1 ? 0 : use + 1;
            s4 = ring_next(s4, 4, w4);
            s3 = ring_next(s3, 3, w4);
            march_barrier(M::kThreads);
        }
    } else {
        const bool copier = warp == KW;
        auto plane_cy = [](int k) { return (k == 2 || k == 5 || k == 6) ? 1 : ((k == 4 || k == 7 || k == 8) ? -1 : 0); };
        const int xl = X0 - T;                           // first column pulled
        int xb = xl, nb = M::kInW;                       // columns of the bulk copies
        int left = 0, singles = 0;                       // columns copied one by one: left of the row, in all
        if (cols) {
            xb = max(xl, 0);
            nb = min(xl + M::kInW, a.nx & ~3) - xb;
            left = a.abb_x ? 0 : xb - xl;                // T or 0
            singles = left + max(min(xl + M::kW + 2, a.abb_x ? a.nx : a.nx + T) - (xb + nb), 0);
        }
        const int lcy = plane_cy(lane);
        // the n-th single copy: its place in a slot (bytes), its plane's c_y, and its source in row 0
        auto single = [&](int n, int &to, int &cyk) {
            const int c = n / 9, k = n - 9 * c, x = c < left ? xl + c : xb + nb + (c - left);
            int e = x - xl;
            LBM_CHK(e, M::kInW, a.err, kErrShared);
            to = (k * M::kInW + e) * 4;
            cyk = plane_cy(k);
            return a.src + k * a.plane + (x < 0 ? x + a.nx : (x >= a.nx ? x - a.nx : x));
        };
        int sto[2] = {-1, -1}, scy[2] = {0, 0};           // this lane's first two
        const float *sfrom[2] = {a.src, a.src};
        if (EDGE) {
#pragma unroll
            for (int j = 0; j < 2; ++j)
                if (lane + 32 * j < 9 * singles) sfrom[j] = single(lane + 32 * j, sto[j], scy[j]);
        }
        const int lo0 = rows ? max(Y0 - (T - 1), 0) : Y0 - (T - 1);
        const int hi0 = rows ? min(Y1 - 1 + (T - 1), a.ny - 1) : Y1 - 1 + (T - 1);
        auto copy = [&](int slot, int r) {               // row r of level 0
            if (r >= lo0 && r <= hi0) {
                const unsigned to = stage_s + slot * M::kInBytes;
                if (lane == 0) march_expect(bars_s + 8 * slot, 36u * nb);
                __syncwarp();
                if (lane < 9)
                    bulk_copy(to + (lane * M::kInW + xb - xl) * 4, a.src + lane * a.plane + source_row(r, lcy) + xb, 4 * nb,
                              bars_s + 8 * slot);
                if (EDGE) {
#pragma unroll
                    for (int j = 0; j < 2; ++j)
                        if (sto[j] >= 0) copy4(to + sto[j], sfrom[j] + source_row(r, scy[j]));
                    for (int n = lane + 64; n < 9 * singles; n += 32) {
                        int to_n, cy_n;
                        const float *from = single(n, to_n, cy_n);
                        copy4(to + to_n, from + source_row(r, cy_n));
                    }
                }
            }
            if (cols) asm volatile("cp.async.commit_group;" ::: "memory");
        };
        int fill = M::kStage - 1;
        if (copier) {
#pragma unroll
            for (int j = 0; j < M::kStage - 1; ++j) copy(j, Y0 - (T - 1) + j);
            if (cols) asm volatile("cp.async.wait_group %0;" ::"n"(M::kStage - 2) : "memory");
        }
        march_barrier(M::kThreads);
        const float *in = sm + (lev - 1) * M::kRing;
        float *out = sm + lev * M::kRing;
        for (int i = 0, r = r_first; i < n_it; ++i, ++r) {
            if (copier) {
                copy(fill, Y0 - (T - 1) + i + M::kStage - 1);
                fill = fill == M::kStage - 1 ? 0 : fill + 1;
            }
            // rows r - 1, r, r + 1 of level lev - 1 are those of iterations i - 3, i - 2, i - 1
            const int p4 = ring_next(s4, 4, w4), p3 = ring_next(s3, 3, w4), n3 = ring_next(p3, 3, w4);
            // the last `lev` pairs of a level have no sources: they compute on what follows in
            // shared memory, and nothing keeps their results
            if (r >= lo && r <= hi) {
                F2 g[P][9];
#pragma unroll
                for (int p = 0; p < P; ++p)
                    each_k([&](auto K) {
                        g[p][K] = ring_pull<K>(in + (cy(K) > 0 ? p4 : (cy(K) == 0 ? p3 : n3)) + ring_plane(K, w4), w4, q0 + 32 * p);
                    });
                if (EDGE) {
                    const int o4 = ring_next(p4, 4, w4);
#pragma unroll
                    for (int p = 0; p < P; ++p)
                        walls(r, p, g[p], [&](int k, int h) {
                            return ring_own(in + (cy(k) > 0 ? o4 : p3) + ring_plane(k, w4), w4, q0 + 32 * p, k, h);
                        });
                }
#pragma unroll
                for (int p = 0; p < P; ++p) step(r, p, g[p]);
                if (lev < T - 1) {
#pragma unroll
                    for (int p = 0; p < P; ++p)
                        each_k([&](auto K) {
                            ring_put<K>(out + (cy(K) > 0 ? s4 : s3) + ring_plane(K, w4), w4, q0 + 32 * p, g[p][K]);
                        });
                } else {
                    int yy = r;
                    LBM_CHK(yy, a.ny, a.err, kErrY);
#pragma unroll
                    for (int p = 0; p < P; ++p) {
                        int X = xa + 64 * p;
                        if (q0 + 32 * p < M::kOut / 2 && X < a.nx) {
                            LBM_CHK(X, a.nx, a.err, kErrX);
                            // a pair that starts at the last column of an odd row ends in the row's padding
                            float *o = a.dst + (unsigned)yy * (unsigned)a.pitch + X;
#pragma unroll
                            for (int k = 0; k < 9; ++k) __stcs(reinterpret_cast<float2 *>(o + k * a.plane), g[p][k].v);
                        }
                    }
                }
            }
            s4 = p4;
            s3 = p3;
            if (copier && cols) asm volatile("cp.async.wait_group %0;" ::"n"(M::kStage - 2) : "memory");   // row i + 1 is there
            march_barrier(M::kThreads);
        }
    }
}

// Two copies of the march: a branch to the walls inside the loop would make every
// row of every strip move its populations to the registers they meet again in.
template <int CONV, int DIFF, int SRC, bool KF, int T, int KW, int P, int ST, int MINB>
__global__ void __launch_bounds__(32 * KW * T, MINB)
k_march(const __grid_constant__ MarchArgs a)
{
    extern __shared__ __align__(16) float sm_m[];
    using M = March<T, KW, P, ST>;
    // strips one after another, the first and the last strip of the grid, whose blocks take
    // longest, ahead of the others
    const int order = blockIdx.x / a.chunks, chunk = blockIdx.x - order * a.chunks;
    const int strip = order == 0 ? 0 : (order == 1 ? a.strips - 1 : order - 1);
    const int X0 = strip * M::kOut, Y0 = chunk * a.H;
    const int Y1 = min(Y0 + a.H, a.ny);
    if (Y0 >= a.ny) return;
    // without cols no pull leaves the row, and the bulk copies end in the row or its padding
    const bool cols = X0 - T < 0 || X0 - (T - 1) + M::kW >= a.nx || X0 - T + M::kInW > a.pitch;
    const bool rows = a.abb_y && (Y0 - T < 0 || Y1 + T > a.ny);
    if (cols || rows) march_strip<CONV, DIFF, SRC, KF, T, KW, P, ST, true>(a, a.k, sm_m, X0, Y0, Y1, cols, rows);
    else march_strip<CONV, DIFF, SRC, KF, T, KW, P, ST, false>(a, a.k, sm_m, X0, Y0, Y1, false, false);
}

template <int CONV, int DIFF, int SRC, bool KF>
static cudaError_t march_t(const lbm_solver *s, int src, bool prepare, cudaStream_t st)
{
    using M = March<kMarchT, kMarchKW, kMarchP, kMarchStage>;
    const auto kernel = k_march<CONV, DIFF, SRC, KF, kMarchT, kMarchKW, kMarchP, kMarchStage, kMarchBlocks>;
    static SmemOptIn once;
    const cudaError_t e = opt_in_smem((const void *)kernel, M::kSmem, once);
    if (e != cudaSuccess || prepare) return e;
    const Params<float> &p = make_params<float>(s);
    MarchArgs a;
    a.k = coll_cast<F2>(p.k);
    a.src = (const float *)s->pop[src];
    a.dst = (float *)s->pop[src ^ 1];
    a.Afield = p.Afield;
    a.plane = p.plane;
    a.pitch = (int)p.pitch;
    a.nx = p.nx;
    a.ny = p.ny;
    a.abb_x = p.abb_x;
    a.abb_y = p.abb_y;
    for (int k = 0; k < 8; ++k)
        for (int z = 0; z < 3; ++z) a.wt[k][z] = p.wt[k][z];
    a.has_src = p.has_src;
    a.give_up = s->give_up;
    a.err = p.err;
    static_assert(M::kOut == kMarchOut, "strips of the launch's grid");
    const MarchGrid g = march_grid(p.nx, p.ny, s->sms);
    a.strips = g.strips;
    a.chunks = g.chunks;
    a.H = g.H;
    kernel<<<a.strips * a.chunks, M::kThreads, M::kSmem, st>>>(a);
    return cudaGetLastError();
}

#define LBM_MARCH_FAMILIES(CALL)                  \
    switch (step_key(s)) {                        \
    case 0: return CALL(0, 0);                    \
    case 1: return CALL(0, 1);                    \
    case 2: return CALL(0, 2);                    \
    case 3: return CALL(1, 0);                    \
    case 4: return CALL(1, 1);                    \
    case 5: return CALL(1, 2);                    \
    case 6: return CALL(kConvNone, 0);            \
    case 7: return CALL(kConvNone, 1);            \
    case 8: return CALL(kConvNone, 2);            \
    }                                             \
    return cudaErrorInvalidValue;

}  // namespace lbm
