// lbm3_relax.cuh -- the D3Q19 collision of the FP32 and FP64 kernels, every operation with its
// rounding written out (as relax() of lbm_relax.cuh, and by its two rules: a product
// that meets a sum is a fused multiply-add), so that the one-step kernel and the
// two-step sweeps return the same bits. It is the projector form of collide3() with
// the constants of every polynomial in phi folded on the host.
#pragma once

#include <type_traits>

#include "lbm3_device.cuh"

namespace lbm {

template <class C, int CONV, int DIFF, bool SRC>
__device__ __forceinline__ void relax3(const Coll3<C> &k, C f[19])
{
    C s[9], d[9];
#pragma unroll
    for (int m = 0; m < 9; ++m) {
        s[m] = vadd(f[2 * m + 1], f[2 * m + 2]);
        d[m] = vsub(f[2 * m + 1], f[2 * m + 2]);
    }
    const C rho = vadd(vadd(vadd(vadd(s[0], s[1]), vadd(s[2], s[3])), vadd(vadd(s[4], s[5]), vadd(s[6], s[7]))),
                       vadd(s[8], f[0]));
    const C jx = vadd(vadd(d[0], d[3]), vadd(d[4], vsub(d[5], d[6])));
    const C jy = vadd(vadd(d[1], d[3]), vadd(vsub(d[7], d[4]), d[8]));
    const C jz = vadd(vadd(d[2], d[5]), vadd(d[6], vsub(d[7], d[8])));
    C phi = rho;
    if constexpr (SRC) phi = vmad(rho, k.inv_den, k.phi0);               // Eq. 35
    C phi2 = phi, phi3 = phi;
    if constexpr (CONV == 1 || DIFF != 0) phi2 = vmul(phi, phi);
    if constexpr (CONV == 1 || DIFF == 2) phi3 = vmul(phi2, phi);
    const C beta = CONV == 1 ? phi2 : phi, cphi = CONV == 1 ? phi3 : phi;
    C vx = vmad(k.nb[0], beta, jx), vy = vmad(k.nb[1], beta, jy), vz = vmad(k.nb[2], beta, jz);
    C t, X;
    if constexpr (SRC && CONV == 0) {
        vx = vadd(vx, k.pc[0]);
        vy = vadd(vy, k.pc[1]);
        vz = vadd(vz, k.pc[2]);
        t = vmad(k.tb, phi, k.hr0);
        // R itself, not folded into xs: xs + hse r1 rounded once was an error of the rate that
        // every step repeated (FP64, 67 x 24 x 77, r1 = -5e-4, 33 steps: 2.4e-15 against
        // 64-bit references, 3.7e-16 so; 1,666 us and 1,729)
        X = vmad(k.hse, vmad(k.r1, phi, k.r0), vmul(k.xs, phi));
    } else {
        t = vmul(k.tb, beta);
        X = vmul(k.xs, phi);
    }
    if constexpr (CONV == 1) X = vmad(k.xc, phi3, X);
    if constexpr (DIFF == 1) X = vmad(k.xi, phi2, X);
    if constexpr (DIFF == 2) X = vmad(k.xi, phi3, X);
    if constexpr (SRC && CONV == 1) {
        const C R = vmad(k.r1, phi, k.r0), S = vmul(R, phi);
        vx = vmad(k.ph[0], S, vx);
        vy = vmad(k.ph[1], S, vy);
        vz = vmad(k.ph[2], S, vz);
        t = vmad(k.hse, S, t);
        X = vmad(k.hse, R, X);
    }
    const C gx = vmad(k.nG[0], vx, vmad(k.nG[1], vy, vmul(k.nG[2], vz)));   // -G
    const C gy = vmad(k.nG[1], vx, vmad(k.nG[3], vy, vmul(k.nG[4], vz)));
    const C gz = vmad(k.nG[2], vx, vmad(k.nG[4], vy, vmul(k.nG[5], vz)));
    const C Ux = vmad(k.u6[0], t, gx), Uy = vmad(k.u6[1], t, gy), Uz = vmad(k.u6[2], t, gz);
    const C Vx = vmad(k.u12[0], t, gx), Vy = vmad(k.u12[1], t, gy), Vz = vmad(k.u12[2], t, gz);
    C b18 = vmul(X, k.i18), b36 = vmul(X, k.i36);
    if constexpr (DIFF == 1) { b18 = vmad(k.qi, phi2, b18); b36 = vmad(k.qi, phi2, b36); }
    if constexpr (DIFF == 2) { b18 = vmad(k.qi, phi3, b18); b36 = vmad(k.qi, phi3, b36); }
    f[0] = vmad(k.i3, X, vmul(k.omse, f[0]));
    auto pair = [&](int i, C e, C o) {
        f[i] = vmad(k.omse, f[i], vadd(e, o));
        f[i + 1] = vmad(k.omse, f[i + 1], vsub(e, o));
    };
    pair(1, vmad(k.ea[0], cphi, b18), Ux);
    pair(3, vmad(k.ea[1], cphi, b18), Uy);
    pair(5, vmad(k.ea[2], cphi, b18), Uz);
    pair(7, vmad(k.ep[0], cphi, b36), vadd(Vx, Vy));
    pair(9, vmad(k.em[0], cphi, b36), vsub(Vx, Vy));
    pair(11, vmad(k.ep[1], cphi, b36), vadd(Vx, Vz));
    pair(13, vmad(k.em[1], cphi, b36), vsub(Vz, Vx));
    pair(15, vmad(k.ep[2], cphi, b36), vadd(Vy, Vz));
    pair(17, vmad(k.em[2], cphi, b36), vsub(Vy, Vz));
}

// ---- two steps per sweep --------------------------------------------------------
// A block owns a 30 x 14 column of nodes and walks along z. Iteration i computes the
// state after the first step on the plane Z0 - 1 + i of its 32 x 16 region (tile and a
// one-node halo; one pair of x-adjacent nodes per thread) into shared memory, then the
// second step on the plane before it, whose sources on the three planes around it are
// all there. A plane is kept as long as it is pulled from: the five populations with
// c_z = 1 for three planes, the nine with c_z = 0 for two, the five with c_z = -1 for
// one. Every population crosses HBM once per two steps (76 B per update in FP32); the
// halo and the two planes beyond a chunk's 16 cost 37 % of the first step's collisions (512 x
// 18 for 420 x 16), 19 % of all. Periodic lattices.
//
// What bounds it: two blocks of eight warps per SM (128 registers: the next plane's
// pulls fly during the second step) wait at the two barriers of an iteration and for
// the pulls. 256^3, 40 steps: 15.50 -> 11.39 ms (43.3k -> 58.9k MLUPS; the one-step kernel
// is at the copy bandwidth). With wall code compiled in, and the planes it needs kept
// (six more per column), 324 us per step against 285; 128^3 then 53 to 57 against 53.5 of
// the one-step kernel, 64^3 11.4 against 9.0: from 2^22 nodes on. Regions of 32 x 12
// (three blocks per SM) spill: 470 us; of 32 x 8 486.
constexpr int kS3X = 30, kS3RX = 32;
template <int TY> struct S3 {
    static constexpr int kRN = kS3RX * (TY + 2), kThreads = kRN / 2, kSmem = 38 * kRN * (int)sizeof(float);
};

// Planes with c_x = 0 keep the even and the odd columns of a row apart, odd rows the
// other way round: a pull's two columns, from two pairs, then meet no bank conflict.
__device__ __forceinline__ int s3_split(int row, int e) { return row * kS3RX + (((e ^ row) & 1) << 4) + (e >> 1); }

struct Sweep3Args {
    Coll3<F2> k;
    const float *src;
    float *dst;
    long long plane;
    int pitch, nx, ny, nz, H;       // H: planes per block
    int *err;
};

// place of direction k's plane in shared memory: c_z = 1 three slots, c_z = 0 two, c_z = -1 one
__host__ __device__ constexpr int s3_place(int k)
{
    int n = 0;
    for (int j = 0; j < k; ++j) n += c3z(j) == c3z(k);
    return n;
}
__host__ __device__ constexpr int s3_plane(int k)
{
    return c3z(k) > 0 ? 3 * s3_place(k) : (c3z(k) == 0 ? 15 + 2 * s3_place(k) : 33 + s3_place(k));
}

template <int K = 0, class F> __device__ __forceinline__ void each_k3(F f)
{
    f(std::integral_constant<int, K>());
    if constexpr (K < 18) each_k3<K + 1>(f);
}

// PAIRS: the block's pairs of columns are whole in memory (no odd period splits them).
template <int CONV, int DIFF, bool SRC, int TY, bool PAIRS>
__device__ __forceinline__ void sweep3(const Sweep3Args &a, float *sm, int X0, int Y0, int Z0, int Z1)
{
    constexpr int kRN = S3<TY>::kRN;
    const int q = threadIdx.x & 15, row = threadIdx.x >> 4;
    const int x = X0 - 1 + 2 * q, y = Y0 - 1 + row;           // first step: nodes x, x + 1
    auto wrap = [](int v, int n) { return (v % n + n) % n; };
    // columns x - 1 .. x + 2 and rows y - 1 .. y + 1 of the pulls, wrapped, as byte
    // offsets within a slab: a pull's address is a uniform pointer plus one
    unsigned col[4], rows[3];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        int c = wrap(x - 1 + j, a.nx);
        LBM_CHK(c, a.nx, a.err, kErrX);
        col[j] = (unsigned)c * 4u;
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        int r = wrap(y - 1 + j, a.ny);
        LBM_CHK(r, a.ny, a.err, kErrY);
        rows[j] = (unsigned)r * (unsigned)a.pitch * 4u;
    }
    const long long slab = (long long)a.pitch * a.ny;
    F2 g[19];
    auto load = [&](int z) {
        const int zw = z < 0 ? z + a.nz : (z >= a.nz ? z - a.nz : z);
        long long zo[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            int p = zw - 1 + j;
            p = p < 0 ? a.nz - 1 : (p >= a.nz ? 0 : p);
            LBM_CHK(p, a.nz, a.err, kErrIndex);
            zo[j] = p * slab;
        }
        each_k3([&](auto K) {
            const char *s = reinterpret_cast<const char *>(a.src + K * a.plane + zo[1 - c3z(K)]);
            const unsigned i0 = rows[1 - c3y(K)] + col[1 - c3x(K)], i1 = rows[1 - c3y(K)] + col[2 - c3x(K)];
            if (PAIRS && c3x(K) != 0) g[K] = F2(__ldg(reinterpret_cast<const float2 *>(s + i0)));
            else g[K] = F2(__ldg(reinterpret_cast<const float *>(s + i0)), __ldg(reinterpret_cast<const float *>(s + i1)));
        });
    };
    int s3 = 0;                                               // slots of this iteration's plane: s3 of three, i & 1 of two
    const int c = row * kS3RX + 2 * q, ce = s3_split(row, 0) + q, co = s3_split(row, 1) + q;
    // second step: pair (X, X + 1) of the output tile; threads without one run it on another's
    // place and keep nothing (in convergent code the constants come from uniform registers)
    const bool second = q < kS3X / 2 && row < TY;
    const int q2 = min(q, kS3X / 2 - 1), row2 = min(row, TY - 1);
    const int X = X0 + 2 * q2, Y = Y0 + row2, c2 = (row2 + 1) * kS3RX + 2 * q2 + 1;
    int e2[3], o2[3];                                         // the split planes' places in rows row2 .. row2 + 2
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        o2[j] = s3_split(row2 + j, 1) + q2;
        e2[j] = s3_split(row2 + j, 0) + q2 + 1;
    }
    load(Z0 - 1);
    for (int i = 0; i < Z1 - Z0 + 2; ++i) {
        const int z = Z0 - 1 + i, s2 = i & 1;
        if (z <= Z1) {
            relax3<F2, CONV, DIFF, SRC>(a.k, g);
            each_k3([&](auto K) {
                const int p = s3_plane(K) + (c3z(K) > 0 ? s3 : (c3z(K) == 0 ? s2 : 0));
                if (c3x(K) == 0) {
                    sm[p * kRN + ce] = g[K].v.x;
                    sm[p * kRN + co] = g[K].v.y;
                } else {
                    *reinterpret_cast<float2 *>(sm + p * kRN + c) = g[K].v;
                }
            });
        }
        __syncthreads();
        if (z + 1 <= Z1) load(z + 1);         // flies during the second step
        const int z2 = z - 1;
        if (z2 >= Z0 && z2 < Z1) {
            const int m3 = s3 == 2 ? 0 : s3 + 1;              // the slot of the plane before z2 (two iterations ago)
            F2 f[19];
            each_k3([&](auto K) {
                const int p = s3_plane(K) + (c3z(K) > 0 ? m3 : (c3z(K) == 0 ? s2 ^ 1 : 0));
                if (c3x(K) == 0) f[K] = F2(sm[p * kRN + o2[1 - c3y(K)]], sm[p * kRN + e2[1 - c3y(K)]]);
                else f[K] = F2(*reinterpret_cast<const float2 *>(sm + p * kRN + c2 - c3y(K) * kS3RX - c3x(K)));
            });
            relax3<F2, CONV, DIFF, SRC>(a.k, f);
            if (second && X < a.nx && Y < a.ny) {
                int xx = X, yy = Y, zz = z2;
                LBM_CHK(xx, a.nx, a.err, kErrX);
                LBM_CHK(yy, a.ny, a.err, kErrY);
                LBM_CHK(zz, a.nz, a.err, kErrIndex);
                // a pair that starts at the last column of an odd row ends in the row's padding
                const unsigned o = ((unsigned)yy * (unsigned)a.pitch + (unsigned)xx) * 4u;
                each_k3([&](auto K) {
                    __stcs(reinterpret_cast<float2 *>(reinterpret_cast<char *>(a.dst + K * a.plane + zz * slab) + o), f[K].v);
                });
            }
        }
        __syncthreads();
        s3 = s3 == 2 ? 0 : s3 + 1;
    }
}

template <int CONV, int DIFF, bool SRC, int TY, int MINB>
__global__ void __launch_bounds__(S3<TY>::kThreads, MINB)
k_sweep3(const __grid_constant__ Sweep3Args a)
{
    extern __shared__ __align__(16) float sm_s3[];
    const int X0 = blockIdx.x * kS3X, Y0 = blockIdx.y * TY, Z0 = blockIdx.z * a.H, Z1 = min(Z0 + a.H, a.nz);
    const bool pairs = !(a.nx & 1) || (X0 >= 2 && X0 + kS3X + 2 <= a.nx);
    if (pairs) sweep3<CONV, DIFF, SRC, TY, true>(a, sm_s3, X0, Y0, Z0, Z1);
    else sweep3<CONV, DIFF, SRC, TY, false>(a, sm_s3, X0, Y0, Z0, Z1);
}

}  // namespace lbm
