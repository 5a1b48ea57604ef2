// tile_plan.cu -- tiles and steps per launch of the small lattices' kernel.
#include "kernels_tile_general.cuh"

namespace lbm {

// Estimated time of a launch of `steps` steps over W x H tiles. A launch takes some
// microseconds until its first results (gap to the launch before it, pulls from L2); a
// step takes a latency, plus FP32: the issue time of the region's warps; FP64: 2.2 us for every
// four warps (68 to 78 operations of 64 cycles, one warp per quarter of the SM).
// Fitted to measured launches (us): FP32 100^2 T = 8 8.5, 400^2 T = 4 10.4, T = 8 17.4, 600^2
// T = 4 16.7, T = 8 32; FP64 64^2 T = 3 10.5, 128^2 T = 2 10.4, T = 4 24.9, 200^2 T = 2 18.6. On
// large FP64 lattices, where blocks overlap, it is some 15 % low (2048^2 478, measured 557):
// it then only chooses the tiles, not whether they run (route.cu).
double tile_launch_us(int nx, int ny, int W, int H, int steps, bool f64, bool general, int sms)
{
    const int N = f64 || general ? 1 : 2, RY = H + 2 * (steps - 1);
    const int RX = f64 || general ? tile_rx<double>(W, steps) : tile_rx<float>(W, steps);
    const int blocks = ((nx + W - 1) / W) * ((ny + H - 1) / H), n_waves = (blocks + sms - 1) / sms;
    double t = 0.0;
    for (int l = 1; l <= steps; ++l) {                       // rows drop out whole, columns do not
        const int warps = (RX / N * (RY - 2 * (l - 1)) + 31) / 32;
        if (general) t += f64 ? 0.3 + 4.6 * ((warps + 3) / 4) : 0.4 + 0.06 * warps;
        else t += f64 ? 0.2 + 2.2 * ((warps + 3) / 4) : 0.25 + 0.055 * warps;
    }
    return (f64 ? 3.0 : 4.5) + n_waves * t;
}

// The least estimated time per step over T and the tilings that give every SM at
// most one block (or a few waves of them).
TilePlan tile_plan(int nx, int ny, bool f64, bool general, int sms)
{
    TilePlan best;
    best.W = nx; best.H = ny; best.T = 1; best.us = 1e30;          // no tiling fits: never the fastest
    for (int T = 1; T <= kTileMaxT; ++T)
        for (int bx = 1; bx <= nx && bx <= 4 * sms; ++bx) {
            const int W = (nx + bx - 1) / bx;
            if ((nx + W - 1) / W != bx || (general && W < 2)) continue;
            for (int waves = 1; waves <= 4; ++waves) {
                const int by = std::min(general ? ny / 2 : ny, waves * sms / bx);
                if (by < 1) continue;
                const int H = (ny + by - 1) / by;
                const int RX = f64 || general ? tile_rx<double>(W, T) : tile_rx<float>(W, T), RY = H + 2 * (T - 1);
                const int plane = general ? (f64 ? kTileGPlane<double> : kTileGPlane<float>)
                                          : (f64 ? kTilePlane<double> : kTilePlane<float>);
                if ((long long)RX * RY + kTilePad > (T > 1 ? plane : 65536)) continue;
                const double us = tile_launch_us(nx, ny, W, H, T, f64, general, sms) / T;
                if (us < best.us) { best.W = W; best.H = H; best.T = T; best.us = us; }
            }
        }
    return best;
}

}  // namespace lbm
