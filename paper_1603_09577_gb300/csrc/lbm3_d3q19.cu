// lbm3_d3q19.cu -- the three-dimensional (D3Q19) fused stream-collide step,
// its initialisation and read-out, and the lbm3_* C ABI (include/lbm3.h).
//
// One thread per node, x fastest (warps of 32 along x), a grid of
// (x tiles, y tiles, z). Every step pulls the 19 populations f_k(x) =
// f*_k(x - c_k) with periodic wrap (19 reads and 19 writes per update: 152 B
// in FP32), replaces the links that cross an anti-bounce-back wall at wall
// nodes, then collides in the projector form of the moment reading (see
// lbm3.h): feq of Eq. 3 per direction, the flux block acting on j - B, and the
// Scheme B source.
#include <math.h>
#include <string.h>

#include <new>
#include <string>

#include <cuda_bf16.h>

#include "lbm3.h"
#include "lbm_internal.h"

#include "lbm3_relax.cuh"

namespace lbm {

// SRC: there is a source (BF16S decides at run time). FP64 is bound by its pipe and held to
// 64 registers, four blocks per SM; FP32 to 40, six blocks. With both forms of relax3() in
// one kernel and 80 registers in FP64 (three blocks), against now (us per step): 256 x 256 x
// 128 FP64 cubic diffusion with a source 2044 -> 1968, without 1937 -> 1905; 59 x 74 x 27
// with a source 42.7 -> 41.0; 64^3 FP32 8.2 -> 6.5.
template <int PREC, int CONV, int DIFF, bool WALLS, bool OFF32, bool SRC>
__global__ void __launch_bounds__(256, PREC == LBM_F64 ? 4 : (PREC == LBM_F32 ? 6 : 0))
k_step3(const StepParams3<PREC, WALLS> p, const Planes3<typename St3<PREC>::T> pl)
{
    using S = St3<PREC>;
    using T = typename S::C;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= p.nx || y >= p.ny) return;
    const unsigned own = ((unsigned)z * (unsigned)p.ny + (unsigned)y) * (unsigned)p.pitch + (unsigned)x;
    T f[19];
    pull3_node<PREC, CONV, DIFF, WALLS, OFF32>(p, pl, x, y, z, own, f);
    T phi = T(0), mass = T(0);
    if constexpr (PREC != LBM_BF16S) {
        relax3<T, CONV, DIFF, SRC>(p.k, f);
    } else {
        collide3<CONV, DIFF, T>(p, f, phi, mass);
    }
    store3<PREC, OFF32>(pl, own, f, phi, mass);
}

template <int PREC, int CONV, int DIFF>
__global__ void __launch_bounds__(256)
k_init3(const Params3<typename St3<PREC>::C> p, const void *__restrict__ phi_in, int in_prec,
        const Planes3<typename St3<PREC>::T> pl)
{
    using T = typename St3<PREC>::C;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= p.nx || y >= p.ny) return;
    const long long in = ((long long)z * p.ny + y) * p.nx + x;
    const T phi0 = in_prec == LBM_F64 ? T(((const double *)phi_in)[in]) : T(((const float *)phi_in)[in]);
    // fbar = feq(phi0) - R_k/2 (Eq. 40, 33), then one collision, which in exact arithmetic
    // leaves feq + R_k/2 (the moments are off equilibrium by -R_k/2 alone): FP64 and FP32
    // store that, over pairs of opposite velocities (some 70 operations in place of 600)
    T f[19];
    if constexpr (PREC != LBM_BF16S) {
        const T beta = CONV == 1 ? T(0.5) * phi0 * phi0 : phi0, bp = CONV == 1 ? phi0 : T(1);
        const T cphi = CONV == 1 ? phi0 * phi0 * phi0 * T(1.0 / 3.0) : phi0;
        const T iso = DIFF == 0 ? T(0) : (DIFF == 1 ? phi0 * phi0 * T(1.0 / 6.0) : phi0 * phi0 * phi0 * T(1.0 / 9.0));
        const T hR = p.has_src ? T(0.5) * (p.r1 * phi0 + p.r0) : T(0);
        const T X = phi0 - T(4.5) * (p.u2_3 * cphi + iso) + hR, t = beta + bp * hR;
        const T b18 = X * T(1.0 / 18.0) + T(0.25) * iso, b36 = X * T(1.0 / 36.0) + T(0.25) * iso;
        const T Ux = p.u6[0] * t, Uy = p.u6[1] * t, Uz = p.u6[2] * t, Vx = p.u12[0] * t, Vy = p.u12[1] * t, Vz = p.u12[2] * t;
        auto pair = [&](int k, T e, T o) {
            f[k] = e + o;
            f[k + 1] = e - o;
        };
        f[0] = X * T(1.0 / 3.0);
        pair(1, T(0.25) * p.uu[0] * cphi + b18, Ux);
        pair(3, T(0.25) * p.uu[3] * cphi + b18, Uy);
        pair(5, T(0.25) * p.uu[5] * cphi + b18, Uz);
        pair(7, (T(0.125) * (p.uu[0] + p.uu[3]) + T(0.25) * p.uu[1]) * cphi + b36, Vx + Vy);
        pair(9, (T(0.125) * (p.uu[0] + p.uu[3]) - T(0.25) * p.uu[1]) * cphi + b36, Vx - Vy);
        pair(11, (T(0.125) * (p.uu[0] + p.uu[5]) + T(0.25) * p.uu[2]) * cphi + b36, Vx + Vz);
        pair(13, (T(0.125) * (p.uu[0] + p.uu[5]) - T(0.25) * p.uu[2]) * cphi + b36, Vz - Vx);
        pair(15, (T(0.125) * (p.uu[3] + p.uu[5]) + T(0.25) * p.uu[4]) * cphi + b36, Vy + Vz);
        pair(17, (T(0.125) * (p.uu[3] + p.uu[5]) - T(0.25) * p.uu[4]) * cphi + b36, Vy - Vz);
    } else {
        const Coef3<CONV, DIFF, T> q(p, phi0);
#pragma unroll
        for (int k = 0; k < 19; ++k) f[k] = q.feq(k, phi0) - T(0.5) * q.source(k);
    }
    T phi = phi0, mass = T(0);
    if constexpr (PREC == LBM_BF16S) collide3<CONV, DIFF, T>(p, f, phi, mass);
    const unsigned own = ((unsigned)z * (unsigned)p.ny + (unsigned)y) * (unsigned)p.pitch + (unsigned)x;
    store3<PREC, false>(pl, own, f, phi, mass);
}

// phi(t_n) = (sum fbar* - r0/2) / (1 + r1/2) into an FP64 or FP32 field
template <int PREC>
__global__ void __launch_bounds__(256)
k_get_phi3(const Params3<typename St3<PREC>::C> p, const typename St3<PREC>::T *__restrict__ f,
           const float *__restrict__ h, void *__restrict__ out, int out_prec)
{
    using S = St3<PREC>;
    using T = typename S::C;
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z;
    if (x >= p.nx || y >= p.ny) return;
    const long long own = ((long long)z * p.ny + y) * p.pitch + x;
    T s = T(0);
#pragma unroll
    for (int k = 0; k < 19; ++k) s += S::ld(f + k * p.plane, own, h, own, w3<T>(k));
    const double v = (double)((s - p.half_r0) * p.inv_post);
    const long long o = ((long long)z * p.ny + y) * p.nx + x;
    if (out_prec == LBM_F64) ((double *)out)[o] = v;
    else ((float *)out)[o] = (float)v;
}

}  // namespace lbm

struct lbm3_solver {
    lbm3_desc d;
    lbm3_coeffs c;
    int coeffs_set = 0, phi_set = 0;
    long long pitch = 0, plane = 0;
    size_t esize = 0;
    void *pop[2] = {nullptr, nullptr};
    float *hpl[2] = {nullptr, nullptr};   // BF16S shift planes
    double *staging = nullptr;
    double *partials = nullptr;
    int *err = nullptr;
    int cur = 0;
    size_t state_bytes = 0;               // populations, then the BF16S shift plane (contiguous)
    double G[6] = {0, 0, 0, 0, 0, 0};
    // the kernels' parameters in the compute type of `prec`, made by lbm3_set_coeffs
    // (made at every launch they took 2 us of host time, as long as the launch itself)
    lbm::Params3W<float> pf{};
    lbm::Params3W<double> pd{};
};

namespace lbm {
namespace {

size_t up256(size_t x) { return (x + 255) & ~size_t(255); }

int check_desc3(const lbm3_desc *d)
{
    if (!d) return fail(LBM_EINVAL, "null lbm3_desc");
    if (d->nx < 2 || d->ny < 2 || d->nz < 2) return fail(LBM_EINVAL, "nx, ny and nz must be >= 2");
    if ((long long)d->nx * d->ny * d->nz > (1LL << 31)) return fail(LBM_EINVAL, "grid larger than 2^31 nodes");
    // node indices within a plane (rows padded to the pitch) are 32-bit
    const long long pitch = ((long long)d->nx + kPitchAlign - 1) / kPitchAlign * kPitchAlign;
    if (pitch * d->ny * d->nz > (1LL << 31) - 1) return fail(LBM_EINVAL, "population plane larger than 2^31 - 1 elements");
    if (d->prec != LBM_F64 && d->prec != LBM_F32 && d->prec != LBM_BF16S)
        return fail(LBM_EINVAL, "D3Q19 storage is LBM_F64, LBM_F32 or LBM_BF16S");
    const int b = d->block_rows;
    if (!(b == 0 || b == 1 || b == 2 || b == 4 || b == 8)) return fail(LBM_EINVAL, "block_rows must be 0, 1, 2, 4 or 8");
    if (d->ny > 65535 * 8 || d->nz > 65535) return fail(LBM_EINVAL, "ny or nz exceeds the launch grid");
    for (int a = 0; a < 3; ++a)
        if (d->bc[a] != LBM_PERIODIC && d->bc[a] != LBM_ABB)
            return fail(LBM_EINVAL, "D3Q19 boundaries are LBM_PERIODIC or LBM_ABB per axis");
    for (int i = 0; i < 6; ++i)
        if (!isfinite(d->phi_wall[i])) return fail(LBM_EINVAL, "non-finite wall value");
    return LBM_OK;
}

struct Layout3 {
    long long pitch, plane;
    size_t esize, pop_bytes, h_bytes, off_stage, off_part, off_err, total;
};

Layout3 layout3(const lbm3_desc *d)
{
    Layout3 L;
    L.pitch = ((long long)d->nx + kPitchAlign - 1) / kPitchAlign * kPitchAlign;
    L.plane = L.pitch * d->ny * d->nz;
    L.esize = d->prec == LBM_F64 ? 8 : (d->prec == LBM_F32 ? 4 : 2);
    L.pop_bytes = up256(19 * (size_t)L.plane * L.esize);
    L.h_bytes = d->prec == LBM_BF16S ? up256((size_t)L.plane * 4) : 0;
    L.off_stage = 2 * (L.pop_bytes + L.h_bytes);
    L.off_part = L.off_stage + up256((size_t)d->nx * d->ny * d->nz * 8);
    L.off_err = L.off_part + up256((size_t)kReduceBlocks * 8 * sizeof(double));
    L.total = L.off_err + 256;
    return L;
}

// Eq. 26 in 3-D: A = (K / (d c_s^2) + I/2)^-1 (Cholesky test of K, adjugate inverse)
bool relax_block3(const double K[6], double A[6])
{
    const double kxx = K[0], kxy = K[1], kxz = K[2], kyy = K[3], kyz = K[4], kzz = K[5];
    const double m1 = kxx, m2 = kxx * kyy - kxy * kxy;
    const double m3 = kxx * (kyy * kzz - kyz * kyz) - kxy * (kxy * kzz - kyz * kxz) + kxz * (kxy * kyz - kyy * kxz);
    if (!(m1 > 0.0 && m2 > 0.0 && m3 > 0.0)) return false;
    const double a = 3 * kxx + 0.5, b = 3 * kxy, c = 3 * kxz, d = 3 * kyy + 0.5, e = 3 * kyz, f = 3 * kzz + 0.5;
    const double det = a * (d * f - e * e) - b * (b * f - e * c) + c * (b * e - d * c);
    A[0] = (d * f - e * e) / det;    // xx
    A[1] = (c * e - b * f) / det;    // xy
    A[2] = (b * e - c * d) / det;    // xz
    A[3] = (a * f - c * c) / det;    // yy
    A[4] = (b * c - a * e) / det;    // yz
    A[5] = (a * d - b * b) / det;    // zz
    return true;
}

Coll3<double> make_coll3(const lbm3_solver *s)
{
    Coll3<double> k{};
    const double se = s->c.se, *u = s->c.u, u2_3 = (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]) / 3.0;
    const bool quad = s->c.conv == 1;                 // B = a phi^2/2, C = a a phi^3/3
    const double half = quad ? 0.5 : 1.0, third = quad ? 1.0 / 3.0 : 1.0;
    const int pa[3] = {0, 0, 1}, pb[3] = {1, 2, 2};   // planes xy, xz, yz
    k.omse = 1.0 - se;
    for (int i = 0; i < 6; ++i) k.nG[i] = -0.1 * s->G[i];
    for (int a = 0; a < 3; ++a) {
        k.nb[a] = -half * u[a];
        k.ph[a] = 0.5 * u[a];
        k.u6[a] = u[a] / 6.0;
        k.u12[a] = u[a] / 12.0;
        k.ea[a] = third * 0.25 * se * u[a] * u[a];
        const double sq = u[pa[a]] * u[pa[a]] + u[pb[a]] * u[pb[a]], cr = u[pa[a]] * u[pb[a]];
        k.ep[a] = third * (0.125 * se * sq + 0.25 * se * cr);
        k.em[a] = third * (0.125 * se * sq - 0.25 * se * cr);
    }
    k.tb = half * se;
    k.hse = 1.0 - 0.5 * se;
    k.xs = quad ? se : se - 4.5 * se * u2_3;
    k.xc = quad ? -1.5 * se * u2_3 : 0.0;
    k.xi = s->c.diff == 1 ? -0.75 * se : (s->c.diff == 2 ? -0.5 * se : 0.0);
    k.qi = s->c.diff == 1 ? se / 24.0 : (s->c.diff == 2 ? se / 36.0 : 0.0);
    k.i18 = 1.0 / 18.0; k.i36 = 1.0 / 36.0; k.i3 = 1.0 / 3.0;
    k.inv_den = 1.0 / (1.0 - 0.5 * s->c.r1);
    k.phi0 = 0.5 * s->c.r0 * k.inv_den;
    k.r0 = s->c.r0; k.r1 = s->c.r1;
    if (!quad) {                                      // R = r0 + r1 phi: the source joins the moments' other terms in phi
        for (int a = 0; a < 3; ++a) {
            k.nb[a] += k.ph[a] * k.r1;
            k.pc[a] = k.ph[a] * k.r0;
        }
        k.tb += k.hse * k.r1;
        k.hr0 = k.hse * k.r0;
    }
    return k;
}

template <class T>
const Params3W<T> &params3(const lbm3_solver *s);
template <> inline const Params3W<float> &params3<float>(const lbm3_solver *s) { return s->pf; }
template <> inline const Params3W<double> &params3<double>(const lbm3_solver *s) { return s->pd; }

template <class T>
Params3W<T> compute_params3(const lbm3_solver *s)
{
    Params3W<T> p{};
    p.nx = s->d.nx; p.ny = s->d.ny; p.nz = s->d.nz;
    p.pitch = s->pitch; p.plane = s->plane;
    p.se = (T)s->c.se;
    p.hse = (T)(1.0 - 0.5 * s->c.se);
    p.omse = (T)(1.0 - s->c.se);
    p.q18 = (T)(0.25 * s->c.se);
    p.q36 = (T)(0.125 * s->c.se);
    for (int i = 0; i < 6; ++i) p.G[i] = (T)(0.1 * s->G[i]);
    const double *u = s->c.u;
    p.ux = (T)u[0]; p.uy = (T)u[1]; p.uz = (T)u[2];
    p.uu[0] = (T)(u[0] * u[0]); p.uu[1] = (T)(u[0] * u[1]); p.uu[2] = (T)(u[0] * u[2]);
    p.uu[3] = (T)(u[1] * u[1]); p.uu[4] = (T)(u[1] * u[2]); p.uu[5] = (T)(u[2] * u[2]);
    p.u2_3 = (T)((u[0] * u[0] + u[1] * u[1] + u[2] * u[2]) / 3.0);
    const double q18 = 0.25 * s->c.se, q36 = 0.125 * s->c.se;
    const int pa[3] = {0, 0, 1}, pb[3] = {1, 2, 2};   // planes xy, xz, yz
    for (int a = 0; a < 3; ++a) {
        p.u6[a] = (T)(u[a] / 6.0);
        p.u12[a] = (T)(u[a] / 12.0);
        p.ea[a] = (T)(q18 * u[a] * u[a]);
        const double sq = u[pa[a]] * u[pa[a]] + u[pb[a]] * u[pb[a]], cr = u[pa[a]] * u[pb[a]];
        p.ep[a] = (T)(q36 * sq + q18 * cr);
        p.em[a] = (T)(q36 * sq - q18 * cr);
    }
    p.r0 = (T)s->c.r0; p.r1 = (T)s->c.r1;
    p.half_r0 = (T)(0.5 * s->c.r0);
    p.inv_den = (T)(1.0 / (1.0 - 0.5 * s->c.r1));
    p.inv_post = (T)(1.0 / (1.0 + 0.5 * s->c.r1));
    p.has_src = s->c.r0 != 0.0 || s->c.r1 != 0.0;
    for (int a = 0; a < 3; ++a) p.abb[a] = s->d.bc[a] == LBM_ABB;
    p.any_abb = p.abb[0] || p.abb[1] || p.abb[2];
    for (int i = 0; i < 6; ++i) p.phi_wall[i] = (T)s->d.phi_wall[i];
    p.err = s->err;
    p.k = coll3_cast<T>(make_coll3(s));
    if (!p.any_abb || s->d.prec == LBM_BF16S) return p;        // BF16S forms the wall terms itself
    for (int k = 1; k < 19; ++k)
        for (int set = 1; set < 8; ++set) {
            double tot = 0.0;
            int cnt = 0;
            const int ck[3] = {c3x(k), c3y(k), c3z(k)};
            for (int a = 0; a < 3; ++a)
                if (set >> a & 1) {
                    tot += s->d.phi_wall[2 * a + (ck[a] > 0 ? 0 : 1)];
                    ++cnt;
                }
            const double phi = tot / cnt, cphi = s->c.conv ? phi * phi * phi / 3.0 : phi;
            const double iso = s->c.diff == 0 ? 0.0 : (s->c.diff == 1 ? phi * phi / 6.0 : phi * phi * phi / 9.0);
            const double cu = ck[0] * u[0] + ck[1] * u[1] + ck[2] * u[2];
            const int c2 = ck[0] * ck[0] + ck[1] * ck[1] + ck[2] * ck[2];
            const double tr3 = (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]) / 3.0 * cphi + iso;
            p.wt[k - 1][set - 1] = (T)(2.0 * w3<double>(k) * (phi + 4.5 * (cu * cu * cphi + c2 * iso - tr3)));
        }
    return p;
}

dim3 block3(const lbm3_solver *s) { return dim3(32, s->d.block_rows > 0 ? s->d.block_rows : 8); }
dim3 grid3(const lbm3_solver *s)
{
    const dim3 b = block3(s);
    return dim3((s->d.nx + 31) / 32, (s->d.ny + b.y - 1) / b.y, s->d.nz);
}

template <class T>
Planes3<T> planes3(const lbm3_solver *s)
{
    Planes3<T> pl;
    const T *src = (const T *)s->pop[s->cur];
    T *dst = (T *)s->pop[s->cur ^ 1];
    for (int k = 0; k < 19; ++k) {
        pl.src[k] = src + k * s->plane;
        pl.dst[k] = dst + k * s->plane;
        pl.poff[k] = (unsigned)(k * s->plane);   // used only when 19 * plane < 2^32
    }
    pl.src0 = src;
    pl.dst0 = dst;
    pl.src_h = s->hpl[s->cur];
    pl.dst_h = s->hpl[s->cur ^ 1];
    return pl;
}

template <int PREC, int CONV, int DIFF>
cudaError_t launch3_t(const lbm3_solver *s, const void *phi0, int in_prec, cudaStream_t st)
{
    using T = typename St3<PREC>::T;
    const auto &p = params3<typename St3<PREC>::C>(s);
    if (phi0) {
        // the initial state goes to the current buffer
        Planes3<T> pl = planes3<T>(s);
        for (int k = 0; k < 19; ++k) pl.dst[k] = (T *)pl.src[k];
        pl.dst_h = s->hpl[s->cur];
        k_init3<PREC, CONV, DIFF><<<grid3(s), block3(s), 0, st>>>(p, phi0, in_prec, pl);
    } else {
        const bool off32 = 19 * s->plane < (1LL << 32);
        const Planes3<T> pl = planes3<T>(s);
        auto launch = [&](auto walls, auto o32) {
            constexpr bool W = decltype(walls)::value, O = decltype(o32)::value;
            if (PREC != LBM_BF16S && p.has_src) k_step3<PREC, CONV, DIFF, W, O, PREC != LBM_BF16S><<<grid3(s), block3(s), 0, st>>>(p, pl);
            else k_step3<PREC, CONV, DIFF, W, O, false><<<grid3(s), block3(s), 0, st>>>(p, pl);
        };
        if (p.any_abb && off32) launch(std::true_type(), std::true_type());
        else if (p.any_abb) launch(std::true_type(), std::false_type());
        else if (off32) launch(std::false_type(), std::true_type());
        else launch(std::false_type(), std::false_type());
    }
    return cudaGetLastError();
}

template <int PREC>
cudaError_t launch3_p(const lbm3_solver *s, const void *phi0, int in_prec, cudaStream_t st)
{
    switch (s->c.conv * 3 + s->c.diff) {
    case 0: return launch3_t<PREC, 0, 0>(s, phi0, in_prec, st);
    case 1: return launch3_t<PREC, 0, 1>(s, phi0, in_prec, st);
    case 2: return launch3_t<PREC, 0, 2>(s, phi0, in_prec, st);
    case 3: return launch3_t<PREC, 1, 0>(s, phi0, in_prec, st);
    case 4: return launch3_t<PREC, 1, 1>(s, phi0, in_prec, st);
    case 5: return launch3_t<PREC, 1, 2>(s, phi0, in_prec, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch3(const lbm3_solver *s, const void *phi0, int in_prec, cudaStream_t st)
{
    switch (s->d.prec) {
    case LBM_F64: return launch3_p<LBM_F64>(s, phi0, in_prec, st);
    case LBM_F32: return launch3_p<LBM_F32>(s, phi0, in_prec, st);
    case LBM_BF16S: return launch3_p<LBM_BF16S>(s, phi0, in_prec, st);
    }
    return cudaErrorInvalidValue;
}

// ---- FP32: two steps per sweep ------------------------------------------------
// Blocks: the 30 x 14 columns of the lattice, cut along z into chunks of 16 planes (a
// chunk costs two more); measured with wall code in, 256^3: 16 323.8 us per step, 8 331.0,
// 32 328.7, 43 324.6.
template <int CONV, int DIFF, bool SRC>
cudaError_t sweep3_t(const lbm3_solver *s, bool prepare, cudaStream_t st)
{
    constexpr int TY = 14, MINB = 2;
    static SmemOptIn once;
    const cudaError_t e = opt_in_smem((const void *)k_sweep3<CONV, DIFF, SRC, TY, MINB>, S3<TY>::kSmem, once);
    if (e != cudaSuccess || prepare) return e;
    const Params3<float> &p = params3<float>(s);
    Sweep3Args a;
    a.k = coll3_cast<F2>(p.k);
    a.src = (const float *)s->pop[s->cur];
    a.dst = (float *)s->pop[s->cur ^ 1];
    a.plane = p.plane;
    a.pitch = (int)p.pitch;
    a.nx = p.nx; a.ny = p.ny; a.nz = p.nz;
    a.err = p.err;
    const int bx = (p.nx + kS3X - 1) / kS3X, by = (p.ny + TY - 1) / TY;
    a.H = 16;
    k_sweep3<CONV, DIFF, SRC, TY, MINB><<<dim3(bx, by, (p.nz + a.H - 1) / a.H), S3<TY>::kThreads, S3<TY>::kSmem, st>>>(a);
    return cudaGetLastError();
}

cudaError_t launch_sweep3(const lbm3_solver *s, bool prepare, cudaStream_t st)
{
    const bool src = s->c.r0 != 0.0 || s->c.r1 != 0.0;
#define LBM_S3(CV, DF) \
    case CV * 3 + DF: return src ? sweep3_t<CV, DF, true>(s, prepare, st) : sweep3_t<CV, DF, false>(s, prepare, st);
    switch (s->c.conv * 3 + s->c.diff) {
        LBM_S3(0, 0)
        LBM_S3(0, 1)
        LBM_S3(0, 2)
        LBM_S3(1, 0)
        LBM_S3(1, 1)
        LBM_S3(1, 2)
    }
#undef LBM_S3
    return cudaErrorInvalidValue;
}

// FP32, periodic, launch left to the library (block_rows 0), large enough (the figures
// stand at the kernel), 32-bit byte offsets within a slab, and estimated faster. A plane of a
// 30 x 14 column costs a block the same time but for its traffic, however little of it a
// flat or narrow lattice fills, and a chunk of 16 planes the first step on two more; a one-step
// warp of 32 nodes costs what HBM takes, more on rows that are no multiple of it (ns). us per step of single
// steps / sweeps: 256^3 376 / 274, 64 x 64 x 1024 96 / 89, 31 x 31 x 4400 162 / 128, 8 x 9 x 65535 399 / 265,
// 61 x 29 x 2400 129 / 118, 96 x 15 x 3000 101 / 118, 32 x 15 x 8800 99 / 149, 4096 x 2 x 512 96 / 255.
bool sweep3_wanted(const lbm3_solver *s)
{
    if (!(s->d.prec == LBM_F32 && s->d.block_rows == 0 && s->d.bc[0] == LBM_PERIODIC && s->d.bc[1] == LBM_PERIODIC &&
          s->d.bc[2] == LBM_PERIODIC && (long long)s->d.nx * s->d.ny * s->d.nz >= (1LL << 22) &&
          s->pitch * s->d.ny < (1LL << 29) && (s->d.ny + 13) / 14 <= 65535))
        return false;
    const double columns = (double)((s->d.nx + kS3X - 1) / kS3X) * ((s->d.ny + 13) / 14);
    const double fill = (double)s->d.nx * s->d.ny / (columns * kS3X * 14);
    const double sweep = 1.05 * columns * (s->d.nz * (6.3 + 5.6 * fill) + 12.0 * ((s->d.nz + 15) / 16));
    const double warps = (double)((s->d.nx + 31) / 32) * s->d.ny * s->d.nz;
    const double ones = 2.0 * warps * (s->d.nx < 64 && s->d.nx % 32 ? 0.95 : 0.74);
    return sweep < ones;
}

template <int PREC>
cudaError_t get_phi3_p(const lbm3_solver *s, void *out, int out_prec, cudaStream_t st)
{
    using T = typename St3<PREC>::T;
    k_get_phi3<PREC><<<grid3(s), block3(s), 0, st>>>(params3<typename St3<PREC>::C>(s), (const T *)s->pop[s->cur],
                                                     s->hpl[s->cur], out, out_prec);
    return cudaGetLastError();
}

cudaError_t get_phi3(const lbm3_solver *s, void *out, int out_prec, cudaStream_t st)
{
    switch (s->d.prec) {
    case LBM_F64: return get_phi3_p<LBM_F64>(s, out, out_prec, st);
    case LBM_F32: return get_phi3_p<LBM_F32>(s, out, out_prec, st);
    case LBM_BF16S: return get_phi3_p<LBM_BF16S>(s, out, out_prec, st);
    }
    return cudaErrorInvalidValue;
}

int ready3(lbm3_handle h)
{
    if (!h) return fail(LBM_EINVAL, "null handle");
    if (!h->coeffs_set) return fail(LBM_EINVAL, "lbm3_set_coeffs has not been called");
    return LBM_OK;
}

}  // namespace
}  // namespace lbm

using namespace lbm;

extern "C" {

int lbm3_workspace_size(const lbm3_desc *desc, size_t *bytes)
{
    if (int rc = check_desc3(desc)) return rc;
    if (!bytes) return fail(LBM_EINVAL, "null size pointer");
    *bytes = layout3(desc).total;
    return LBM_OK;
}

int lbm3_create(lbm3_handle *h, const lbm3_desc *desc, void *dev_workspace, size_t bytes)
{
    if (!h) return fail(LBM_EINVAL, "null handle pointer");
    *h = nullptr;
    if (int rc = check_desc3(desc)) return rc;
    const Layout3 L = layout3(desc);
    if (!dev_workspace || ((uintptr_t)dev_workspace & 255) != 0)
        return fail(LBM_EINVAL, "workspace null or not 256-byte aligned");
    if (bytes < L.total) return fail(LBM_EINVAL, "workspace smaller than lbm3_workspace_size");
    lbm3_solver *s = new (std::nothrow) lbm3_solver();
    if (!s) return fail(LBM_EINVAL, "out of host memory");
    char *ws = (char *)dev_workspace;
    s->d = *desc;
    s->pitch = L.pitch;
    s->plane = L.plane;
    s->esize = L.esize;
    s->pop[0] = ws;
    s->pop[1] = ws + L.pop_bytes + L.h_bytes;
    if (L.h_bytes) {
        s->hpl[0] = (float *)(ws + L.pop_bytes);
        s->hpl[1] = (float *)(ws + 2 * L.pop_bytes + L.h_bytes);
    }
    s->staging = (double *)(ws + L.off_stage);
    s->partials = (double *)(ws + L.off_part);
    s->err = (int *)(ws + L.off_err);
    s->state_bytes = L.pop_bytes + L.h_bytes;
    *h = s;
    return LBM_OK;
}

int lbm3_destroy(lbm3_handle h)
{
    delete h;
    return LBM_OK;
}

int lbm3_set_coeffs(lbm3_handle h, const lbm3_coeffs *c)
{
    if (!h) return fail(LBM_EINVAL, "null handle");
    if (!c) return fail(LBM_EINVAL, "null lbm3_coeffs");
    if (c->conv != 0 && c->conv != 1) return fail(LBM_EINVAL, "conv must be 0 or 1");
    if (c->diff < 0 || c->diff > 2) return fail(LBM_EINVAL, "diff must be 0, 1 or 2");
    if (!(c->se > 0.0 && c->se < 2.0)) return fail(LBM_EINVAL, "s_e must lie in (0, 2)");
    if (!(c->s0 >= 0.0 && c->s0 < 2.0)) return fail(LBM_EINVAL, "s0 must lie in [0, 2)");
    for (int i = 0; i < 3; ++i)
        if (!isfinite(c->u[i])) return fail(LBM_EINVAL, "non-finite coefficient");
    if (!isfinite(c->r0) || !isfinite(c->r1) || !(c->r1 > -2.0 && c->r1 < 2.0))
        return fail(LBM_EINVAL, "source coefficients must be finite with |r1| < 2");
    double A[6];
    if (!relax_block3(c->K, A)) return fail(LBM_EINVAL, "K is not symmetric positive definite");
    h->c = *c;
    // G = A - s_e I
    h->G[0] = A[0] - c->se; h->G[1] = A[1]; h->G[2] = A[2];
    h->G[3] = A[3] - c->se; h->G[4] = A[4]; h->G[5] = A[5] - c->se;
    if (h->d.prec == LBM_F64) h->pd = compute_params3<double>(h);
    else h->pf = compute_params3<float>(h);
    h->coeffs_set = 1;
    return LBM_OK;
}

int lbm3_set_phi(lbm3_handle h, const void *dev_phi, int prec, void *stream)
{
    if (int rc = ready3(h)) return rc;
    if (!dev_phi) return fail(LBM_EINVAL, "null phi");
    if (prec != LBM_F64 && prec != LBM_F32) return fail(LBM_EINVAL, "phi must be LBM_F64 or LBM_F32");
    if (int rc = cuda_check(cudaMemsetAsync(h->err, 0, sizeof(int), (cudaStream_t)stream), "lbm3_set_phi")) return rc;
    if (int rc = cuda_check(launch3(h, dev_phi, prec, (cudaStream_t)stream), "lbm3_set_phi")) return rc;
    if (sweep3_wanted(h))
        if (int rc = cuda_check(launch_sweep3(h, true, (cudaStream_t)stream), "lbm3_set_phi (kernel attributes)")) return rc;
    h->phi_set = 1;
    return LBM_OK;
}

int lbm3_step(lbm3_handle h, int nsteps, void *stream)
{
    if (int rc = ready3(h)) return rc;
    if (!h->phi_set) return fail(LBM_EINVAL, "lbm3_set_phi has not been called");
    if (nsteps < 0) return fail(LBM_EINVAL, "negative step count");
    // an even number of two-step sweeps, so that the launches of a call stay even or odd
    // in number as its steps (a captured call ends on the buffer it started from)
    int launches[2];
    if (int rc = lbm3_step_route(h, nsteps, launches)) return rc;
    if (launches[0])
        if (int rc = cuda_check(launch_sweep3(h, true, (cudaStream_t)stream), "lbm3_step (kernel attributes)")) return rc;
    for (int i = 0; i < launches[0]; ++i) {
        if (int rc = cuda_check(launch_sweep3(h, false, (cudaStream_t)stream), "lbm3_step (two steps per sweep)")) return rc;
        h->cur ^= 1;
    }
    for (int i = 0; i < launches[1]; ++i) {
        if (int rc = cuda_check(launch3(h, nullptr, 0, (cudaStream_t)stream), "lbm3_step")) return rc;
        h->cur ^= 1;
    }
    return LBM_OK;
}

int lbm3_step_route(lbm3_handle h, int nsteps, int launches[2])
{
    if (!h) return fail(LBM_EINVAL, "null handle");
    if (!launches) return fail(LBM_EINVAL, "null launch counts");
    if (nsteps < 0) return fail(LBM_EINVAL, "negative step count");
    launches[0] = sweep3_wanted(h) ? nsteps / 4 * 2 : 0;
    launches[1] = nsteps - 2 * launches[0];
    return LBM_OK;
}

int lbm3_state_bytes(lbm3_handle h, size_t *bytes)
{
    if (!h) return fail(LBM_EINVAL, "null lbm3 handle");
    if (!bytes) return fail(LBM_EINVAL, "null size pointer");
    *bytes = h->state_bytes;
    return LBM_OK;
}

int lbm3_save(lbm3_handle h, void *dev_dst, void *stream)
{
    if (!h) return fail(LBM_EINVAL, "null lbm3 handle");
    if (!h->phi_set) return fail(LBM_EINVAL, "lbm3_set_phi has not been called");
    if (!dev_dst) return fail(LBM_EINVAL, "null destination");
    return cuda_check(cudaMemcpyAsync(dev_dst, h->pop[h->cur], h->state_bytes, cudaMemcpyDeviceToDevice,
                                      (cudaStream_t)stream), "lbm3_save");
}

int lbm3_load(lbm3_handle h, const void *dev_src, void *stream)
{
    if (!h) return fail(LBM_EINVAL, "null lbm3 handle");
    if (!dev_src) return fail(LBM_EINVAL, "null source");
    if (int rc = cuda_check(cudaMemcpyAsync(h->pop[h->cur], dev_src, h->state_bytes, cudaMemcpyDeviceToDevice,
                                            (cudaStream_t)stream), "lbm3_load"))
        return rc;
    if (h->coeffs_set && sweep3_wanted(h))
        if (int rc = cuda_check(launch_sweep3(h, true, (cudaStream_t)stream), "lbm3_load (kernel attributes)")) return rc;
    h->phi_set = 1;
    return LBM_OK;
}

int lbm3_get_phi(lbm3_handle h, void *dev_out, int prec, void *stream)
{
    if (int rc = ready3(h)) return rc;
    if (!h->phi_set) return fail(LBM_EINVAL, "lbm3_set_phi has not been called");
    if (!dev_out) return fail(LBM_EINVAL, "null output");
    if (prec != LBM_F64 && prec != LBM_F32) return fail(LBM_EINVAL, "output must be LBM_F64 or LBM_F32");
    return cuda_check(get_phi3(h, dev_out, prec, (cudaStream_t)stream), "lbm3_get_phi");
}

int lbm3_reduce(lbm3_handle h, const double *dev_ref, double *dev_out, void *stream)
{
    if (int rc = ready3(h)) return rc;
    if (!h->phi_set) return fail(LBM_EINVAL, "lbm3_set_phi has not been called");
    if (!dev_out) return fail(LBM_EINVAL, "null output");
    cudaStream_t st = (cudaStream_t)stream;
    if (int rc = cuda_check(get_phi3(h, h->staging, LBM_F64, st), "lbm3_reduce")) return rc;
    const long long n = (long long)h->d.nx * h->d.ny * h->d.nz;
    return cuda_check(launch_reduce_field(h->staging, n, dev_ref, h->partials, dev_out, st), "lbm3_reduce");
}

int lbm3_debug_flags(lbm3_handle h, int *flags, void *stream)
{
    if (!h) return fail(LBM_EINVAL, "null handle");
    if (!flags) return fail(LBM_EINVAL, "null flags pointer");
    cudaStream_t st = (cudaStream_t)stream;
    if (int rc = cuda_check(cudaMemcpyAsync(flags, h->err, sizeof(int), cudaMemcpyDeviceToHost, st), "lbm3_debug_flags"))
        return rc;
    return cuda_check(cudaStreamSynchronize(st), "lbm3_debug_flags sync");
}

}  // extern "C"
