// route.cu -- which kernels serve a call of lbm_step (host only).
//
// Where the descriptor leaves the launch to the library, the kernels of a precision
// return the same bits, so the route is a matter of time alone: each kernel's launch
// is estimated from the shape of the lattice, and a call takes the launches with the
// least sum. The estimates are fitted to measured launches (GB300, us, periodic /
// walls; step calls of 12 steps, k_march 96):
//
//   lattice        one step      pair tiles   30 x 30 tiles   k_march       k_tile, 4 steps
//   400^2          4.1 / 6.1     8.2 / 14.4     8.2 / 12.3       -             10.4 / 10.4
//   512^2          6.1 / 6.2    10.0 / 16.3     8.2 / 12.3       -             14.4 / 14.4
//   600^2          6.2 / 7.9    10.0 / 16.4     8.2 / 12.5       -             16.4 / 16.8
//   1000^2        10.3 / 12.3   16.4 / 22.6    15.2 / 20.2    26.6 / 27.8
//   2048^2        47.5 / 47.7   59.4 / 67.4    61.8 / 65.7    81.8 / 89.1
//   4096^2         178 / 178     209 / 220      229 / 232      285 / 288
//   64 x 16384    10.3 / 16.4   32.8 / 59.5    20.5 / 33.0       -
//   128 x 16384   24.8 / 26.7   44.6 / 73.8    35.6 / 46.6    79.8 / 88.1
//   2 x 300000     112 / 123     260 / 556      121 / 243        -
//   300000 x 5    17.1 / 18.5   47.2 / 86.2    89.2 / 150        -
//   65536 x 64    47.2 / 47.8   64.3 / 78.2    78.5 / 94.4    81.4 / 86.4
//
// Tiles of a fixed shape cost the same however few of their nodes a narrow lattice
// fills, and tiles at walls about twice as much. A rule on the node count alone (pair
// tiles everywhere else, tiles of one step for single steps) had made 64 x 16384 with
// walls 1.8, 2 x 300000 2.1 and single steps on 600^2 1.6 times slower than one step
// per launch.
#include <algorithm>

#include "lbm_internal.h"

namespace lbm {

// the general kernel serves Scheme A, extrapolation walls and the power-law flux
bool general_path(const lbm_solver *s)
{
    return s->d.scheme == LBM_SCHEME_A || s->d.bc_x == LBM_NEE || s->d.bc_y == LBM_NEE || s->c.conv >= 2 ||
           s->c.diff == 3;
}

// Lattices of Scheme B whose launch is left to the library: FP64 and FP32 with
// kernel_variant 0 and no block shape, or FP32 with the pair kernels' small tiles
// (kernel_variant 5, block_rows 4). The kernels of a precision agree bit for bit,
// whatever the split into sweeps; only with a per-node tensor in FP32 and one step per
// pass do the one-step kernels differ in the last bit, so that they alone run there.
bool auto_path(const lbm_solver *s)
{
    if (s->fixed) return false;
    if (s->d.prec == LBM_F64) return s->d.kernel_variant == 0 && s->d.block_rows == 0;
    return s->d.prec == LBM_F32 && !(s->d.per_cell_K && s->d.steps_per_pass == 1) &&
           ((s->d.kernel_variant == 0 && s->d.block_rows == 0) || (s->d.kernel_variant == 5 && s->d.block_rows == 4));
}

// Strips of the marching kernel and their chunks: one wave of four blocks per SM, or up
// to three where the chunks stay 48 rows or more (a chunk takes 9 iterations beyond its
// rows). 4096^2: 1824 blocks 218.5k MLUPS, 608 204.4k, 4000 211.1k; 1024^2 (chunks of 15
// rows): 608 blocks 154k, 304 112.7k.
MarchGrid march_grid(int nx, int ny, int sms)
{
    const int wave = sms * kMarchBlocks;
    MarchGrid g;
    g.strips = (nx + kMarchOut - 1) / kMarchOut;
    long long waves = (long long)g.strips * ny / (48LL * wave);
    waves = waves < 1 ? 1 : (waves > 3 ? 3 : waves);
    const int chunks = std::max((int)(waves * wave / g.strips), 1);
    g.H = (ny + chunks - 1) / chunks;
    g.chunks = (ny + g.H - 1) / g.H;
    return g;
}

// Whether sweeps of four steps by the marching kernel can serve this lattice. They need
// strips and chunks for the whole chip: from about 2^18 nodes on.
static bool march_fits(const lbm_solver *s)
{
    return s->d.nx >= 128 && s->d.ny >= 64 && (long long)s->d.nx * s->d.ny >= (1LL << 18) && s->L.plane < (1LL << 31);
}

// tiles of tx x ty nodes, and those of them that touch a wall (0.4 for one in y, whose branch
// is the same for all lanes of a row)
static void count_tiles(const lbm_solver *s, int tx, int ty, double *all, double *edge)
{
    const double gx = (s->d.nx + tx - 1) / tx, gy = (s->d.ny + ty - 1) / ty;
    const double ix = s->d.bc_x == LBM_ABB ? std::max(gx - 2, 0.0) : gx, iy = s->d.bc_y == LBM_ABB ? std::max(gy - 2, 0.0) : gy;
    *all = gx * gy;
    *edge = (gx - ix) * gy + 0.4 * ix * (gy - iy);
}

// the estimates of the FP32 kernels (the table above)
static void estimate(const lbm_solver *s, int sms, TilePlan *p)
{
    double n, e;
    count_tiles(s, 32, 8, &n, &e);
    // 18 planes in sectors of 32 bytes: from about 115 MB on the step comes from HBM
    const bool hbm = (double)s->d.ny * ((s->d.nx + 7) / 8) * 32.0 * 18.0 > 115e6;
    p->one = std::max(4.1, 3.4 + (hbm ? 2.7e-3 : 2.0e-3) * n + (e > 0 ? 0.9 + std::min(5.0, 1e-3 * e) : 0.0));
    count_tiles(s, 62, 14, &n, &e);
    const double pair = std::max(8.0, 4.0 + 10.5e-3 * n) + (e > 0 ? 5.5 + 9e-3 * e : 0.0);
    count_tiles(s, 30, 30, &n, &e);
    const double node = std::max(8.0, 3.5 + 12.2e-3 * n) + (e > 0 ? 4.0 + 7e-3 * e : 0.0);
    p->nodes = node < pair;
    p->two = std::min(node, pair);
    if (hbm) p->us = 1e30;              // no small lattice: tiles of 2 x 300000 take 91 us per step
    // tile_launch_us weighs tilings; against other kernels a launch takes 10 % less, but its pulls
    // and stores besides, and more at walls. Estimated / measured, periodic: 400^2 2 steps 8.4 / 8.2,
    // 4 11.3 / 10.4, 6 15.0 / 14.4; 512^2 10.4 / 10.3, 14.5 / 14.4, 19.6 / 16.4; 800^2 3 steps 23.7 / 22.6;
    // 64 x 16384 2 steps 27.9 / 26.7
    for (double &us : p->launch) us = (0.4 + 0.9 * us + 10e-6 * (double)s->d.nx * s->d.ny) * (e > 0 ? 1.06 : 1.0);
    p->four = 1e30;
    if (march_fits(s)) {
        const MarchGrid g = march_grid(s->d.nx, s->d.ny, sms);
        const int wave = sms * kMarchBlocks, waves = (g.strips * g.chunks + wave - 1) / wave;
        const bool walls = s->d.bc_x == LBM_ABB || s->d.bc_y == LBM_ABB;
        p->four = 1.0 + waves * (g.H + 9) * (g.strips <= 3 ? 1.27 : 1.1) * (walls ? 1.05 : 1.0);
    }
}

static void need_plan(lbm_solver *s, bool general, int sms)
{
    if (s->plan.T != 0 && s->plan.general == general && s->plan.sms == sms) return;
    const bool f64 = s->d.prec == LBM_F64;
    s->plan = tile_plan(s->d.nx, s->d.ny, f64, general, sms);
    s->plan.general = general;
    s->plan.sms = sms;
    if (s->plan.us < 1e29)
        for (int n = 1; n <= s->plan.T; ++n)
            s->plan.launch[n] = tile_launch_us(s->d.nx, s->d.ny, s->plan.W, s->plan.H, n, f64, general, sms);
    if (!f64 && !general) estimate(s, sms, &s->plan);
    if (!f64 && general) {               // one step: 32 x 4 tiles; several: 30 % more at walls
        const double blocks = (double)((s->d.nx + 31) / 32) * ((s->d.ny + 3) / 4);
        const bool walls = s->d.bc_x != LBM_PERIODIC || s->d.bc_y != LBM_PERIODIC;
        for (double &us : s->plan.launch) us *= walls ? 1.3 : 1.0;
        s->plan.launch[1] = std::max(4.1, (walls ? 4.6 : 3.4) + 1.6e-3 * blocks);
    }
}

// launches of a call, modulo 2: as with steps_per_pass steps each (n, or n/2 + n%2), so that
// a captured call that ended on the buffer it started from still does
static int launch_parity(const lbm_solver *s, int nsteps)
{
    return (s->d.steps_per_pass == 2 ? nsteps / 2 + nsteps % 2 : nsteps) & 1;
}

// The number of launches over the plan's tiles, odd or even as `parity`, and in *us their
// time: nsteps shared as evenly as can be, at least `least` in each. 0: there is none.
static int tile_launches(const lbm_solver *s, int nsteps, int parity, int least, double *us)
{
    const TilePlan &p = s->plan;
    int best = 0;
    *us = 1e30;
    if (p.us >= 1e29 || nsteps < 1) return 0;
    const int fewest = (nsteps + p.T - 1) / p.T;
    for (int n = fewest; n <= nsteps && nsteps / n >= least && n < fewest + 8; ++n) {
        if ((n & 1) != parity) continue;
        const int lo = nsteps / n, more = nsteps - lo * n;
        const double t = (n - more) * p.launch[lo] + (more ? more * p.launch[lo + 1] : 0.0);
        if (t < *us) { *us = t; best = n; }
    }
    return best;
}

// The general path's small lattices (the C-free variant runs one step per launch). All
// calls of a lattice take the same kernel, tiles or not: its bits differ from the other
// general kernels' in the last place. Measured on a power-law flux, us per step in calls of
// 20 (the kernels of the descriptor -> tiles), Scheme A:
//   FP32, one step per pass    60^2      301^2     400^2     500^2     600^2
//     extrapolated walls    4.6 -> 1.6  6.2 -> 3.7  6.3 -> 4.7  8.3 -> 6.3  8.5 -> 9.1
//     periodic              4.1 -> 1.6  4.5 -> 2.9  6.2 -> 3.7  6.2 -> 5.3
//   FP32, two steps per pass
//     extrapolated walls    6.2 -> 1.6  6.2 -> 3.7  7.4 -> 4.7  7.4 -> 6.3  7.3 -> 9.1
//     periodic              4.1 -> 1.6  4.1 -> 2.9  5.0 -> 3.7  5.1 -> 5.3
//   FP64, extrapolated      24.6 -> 10.4  55 -> 43  81 -> 72  104 -> 96
// A periodic lattice with two steps per pass keeps its two-step kernel from 130,000 nodes
// on (Scheme A 170,000), where a call of two steps (400^2 Scheme B 8.2 us) is one launch over
// the tiles (10.3). Not mended by this choice: calls of one or two single steps on periodic
// lattices, 301^2 Scheme A 4.5 -> 6.1 and 500^2 6.2 -> 8.2 us per step, where longer calls gain. FP64 Scheme B
// without walls keeps the one-step kernel where one step per launch over the tiles takes as
// many turns of the FP64 pipe: 250^2 20.5 us against 22.6.
static bool tile_general_wanted(lbm_solver *s, int sms)
{
    if (s->fixed || s->d.kernel_variant != 0 || s->d.block_rows != 0 || s->c.cfree || s->d.prec == LBM_BF16S || s->c.conv > 2)
        return false;
    const long long n = (long long)s->d.nx * s->d.ny;
    const bool f64 = s->d.prec == LBM_F64, periodic = s->d.bc_x == LBM_PERIODIC && s->d.bc_y == LBM_PERIODIC;
    if (n > (f64 ? 500000 : 250000)) return false;
    if (periodic && s->d.steps_per_pass == 2 && n > (s->d.scheme == LBM_SCHEME_A ? 170000 : 130000)) return false;
    need_plan(s, true, sms);
    if (s->plan.us >= 1e29 || (!f64 && s->plan.T < 2)) return false;
    if (f64 && periodic && s->d.scheme == LBM_SCHEME_B && s->plan.T == 1) {
        const int blocks = ((s->d.nx + 31) / 32) * ((s->d.ny + 7) / 8), warps = (s->plan.W * s->plan.H + 31) / 32;
        return (warps + 3) / 4 < 2 * ((blocks + sms - 1) / sms);
    }
    return true;
}

// FP32 on the path left to the library: the tiles with up to two single steps after them (a
// launch of one step is the one-step kernel's: on 600^2 6.2 us, over the tiles 10.2), or
// sweeps of four, of two and single steps.
static Route plan_f32(const lbm_solver *s, int nsteps)
{
    const TilePlan &p = s->plan;
    Route best;
    double least = 1e30;
    const int fours[3] = {p.four < 1e29 ? nsteps / 4 : 0, p.four < 1e29 ? nsteps / 4 - 1 : 0, 0};
    for (int f : fours) {
        if (f < 0) continue;
        const int pairs = (nsteps - 4 * f) / 2, twos[3] = {pairs, pairs - 1, 0};
        for (int t : twos) {
            if (t < 0) continue;
            const int one = nsteps - 4 * f - 2 * t;
            if (((f + t + one) & 1) != launch_parity(s, nsteps)) continue;
            const double us = f * (f ? p.four : 0.0) + t * p.two + one * p.one;
            if (us < least) {
                least = us;
                best = Route();
                best.fours = f;
                (p.nodes ? best.twos : best.pairs) = t;
                best.ones = one;
            }
        }
    }
    for (int one = 0; one <= 2; ++one) {
        double us;
        const int tiles = tile_launches(s, nsteps - one, launch_parity(s, nsteps) ^ (one & 1), 2, &us);
        if (one) us += one * p.one + 3.0;         // only where the tiles alone are clearly longer
        if (!tiles || us >= least) continue;
        least = us;
        best = Route();
        best.tiles = tiles;
        best.ones = one;
    }
    return best;
}

Route plan_route(lbm_solver *s, int nsteps, int sms)
{
    Route r;
    if (general_path(s)) {
        double us;
        if (tile_general_wanted(s, sms)) r.tiles = tile_launches(s, nsteps, launch_parity(s, nsteps), 1, &us);
        else if (s->d.steps_per_pass == 2) { r.twos = nsteps / 2; r.ones = nsteps % 2; }
        else r.ones = nsteps;
        return r;
    }
    if (!auto_path(s)) {
        if (s->d.steps_per_pass == 2) {
            (s->d.kernel_variant == 5 ? r.pairs : r.twos) = nsteps / 2;
            r.ones = nsteps % 2;
        } else {
            r.ones = nsteps;
        }
        return r;
    }
    need_plan(s, false, sms);
    if (s->d.prec == LBM_F32) return plan_f32(s, nsteps);
    // FP64: the tiles wherever one fits (up to some 39 M nodes), with one step per launch on
    // large lattices too, where they are a one-step kernel with fewer and larger blocks. us per
    // step of the one-step kernel -> tiles, linear periodic / cubic diffusion with walls and
    // source: 128^2 8.2 -> 5.3 / 10.2 -> 6.3, 301^2 18.4 -> 16.4 / 21.5 -> 18.4, 512^2 39.0 -> 39.8 /
    // 45.1 -> 43.1, 1000^2 144.2 -> 139.3 / 159.6 -> 149.7, 2048^2 563.5 -> 556.4 / 620 -> 597, 4096^2
    // 2233 -> 2206 / 2455 -> 2343; 2 x 300000 1274 -> 129, 33 x 8000 75.9 -> 39.1, 1023 x 777 with
    // walls 114.9 -> 116.7, 2048^2 linear with walls 565.5 -> 568.6.
    double us;
    r.tiles = tile_launches(s, nsteps, launch_parity(s, nsteps), 1, &us);
    if (!r.tiles) r.ones = nsteps;
    return r;
}

}  // namespace lbm
