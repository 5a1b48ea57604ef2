// lbm_relax.cuh -- the collision of the FP64 and FP32 kernels of Scheme B
// (Eq. 15-18, 34-35) with its constants prepared on the host.
//
// Every operation is written with its rounding (one rounding per add, multiply
// or fused multiply-add), in scalar and in packed form alike, so every kernel
// that calls relax() on the same populations returns the same bits: one node per
// thread, two nodes per packed FP32x2 instruction, one step or several per sweep.
//
// Two rules keep that so: every product that meets a sum is written as a fused
// multiply-add (ptxas fuses a packed multiply and add even where both name
// their rounding, at places that differ from kernel to kernel), and products
// standing alone are only multiplied on or enter as the addend of one.
//
// What bounds it: FP64 kernels run at the FP64 pipe's rate, so the operation
// count is their time; the FP32 kernels issue one packed instruction for two
// nodes. The equilibrium moments are polynomials in phi, whose coefficients the
// host folds (e_eq = ke1 phi + h, eps_eq = kp1 phi - h, h the quadratic or cubic
// part), and all rates carry M0's row norms: 68 operations for the linear family
// and 73 for the 4096^2 workload's (no flux, cubic diffusion, source), where
// forming every moment from B, C and D one after another takes 100 and 86.
//
// What keeps the error of long runs at the rounding of the stored populations: the
// equilibrium moments meet the moments as a whole (FP64, bound by its pipe: their linear
// part, the largest, is taken off last, one operation fewer), and the source enters every
// population from one value of R/9. With the linear part first, and R/9 added to f[0]
// on its own, the roundings of a step leaned one way and added up. FP32 against FP64,
// relative L2: Burgers 256^2, K = 0.32, 3000 steps 3.1e-7 then, now 8.3e-8 (collide()
// 9.8e-8); cubic diffusion with decay 128^2, 2000 steps 2.2e-7 and 8.7e-8 (9.0e-8).
#pragma once

#include <type_traits>

#include "lbm_device.cuh"

namespace lbm {

__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vmad(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double vsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double vmad(double a, double b, double c) { return __fma_rn(a, b, c); }
#define LBM_F2_BINARY(NAME, OP)                                                              \
    __device__ __forceinline__ F2 NAME(F2 a, F2 b)                                           \
    {                                                                                        \
        F2 r;                                                                                \
        asm(OP " %0, %1, %2;" : "=l"(reinterpret_cast<unsigned long long &>(r.v))            \
            : "l"(reinterpret_cast<const unsigned long long &>(a.v)),                        \
              "l"(reinterpret_cast<const unsigned long long &>(b.v)));                       \
        return r;                                                                            \
    }
LBM_F2_BINARY(vadd, "add.rn.f32x2")
LBM_F2_BINARY(vsub, "sub.rn.f32x2")
LBM_F2_BINARY(vmul, "mul.rn.f32x2")
#undef LBM_F2_BINARY
__device__ __forceinline__ F2 vmad(F2 a, F2 b, F2 c)
{
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(reinterpret_cast<unsigned long long &>(r.v))
        : "l"(reinterpret_cast<const unsigned long long &>(a.v)), "l"(reinterpret_cast<const unsigned long long &>(b.v)),
          "l"(reinterpret_cast<const unsigned long long &>(c.v)));
    return r;
}

// The relaxation of one node's populations in place; phi = Eq. 35. NODE_K: A3,
// A35, A5 are the node's block, else the constant one of k. SRC: 0 no source,
// 1 a source, 2 decided by `src` at run time. Moments of Eq. 15, the change dm
// of every moment divided by its row norm, f += M0^-1 dm.
template <class C, int CONV, int DIFF, bool NODE_K, int SRC = 2>
__device__ __forceinline__ void relax(const Coll<C> &k, bool src, C f[9], C A3, C A35, C A5, C &phi_out)
{
    constexpr bool FLUX = has_flux<CONV>();
    const bool S_ON = SRC == 2 ? src : SRC == 1;
    const C a = vadd(f[1], f[3]), b = vadd(f[2], f[4]), c = vadd(f[5], f[7]), d = vadd(f[6], f[8]);
    const C da = vsub(f[1], f[3]), db = vsub(f[2], f[4]), dc = vsub(f[5], f[7]), dd = vsub(f[6], f[8]);
    const C axis = vadd(a, b), dg = vadd(c, d);
    const C rho = vadd(vadd(f[0], axis), dg);
    const C ne = vmad(k.mtwo, dg, vmad(k.four, f[0], axis));       // -e
    const C eps = vmad(k.mtwo, axis, vmad(k.four, f[0], dg));
    const C X = vsub(dc, dd), Y = vadd(dc, dd);
    C jx = vadd(da, X), jy = vadd(db, Y);
    C qx = vmad(k.mtwo, da, X), qy = vmad(k.mtwo, db, Y);
    C pxx = vsub(a, b), pxy = vsub(c, d);

    C phi = rho;
    if (S_ON) phi = vmad(rho, k.inv_den, k.phi0);
    phi_out = phi;

    // departures from the equilibrium moments (Eq. 16): te = -(e - e_eq),
    // tp = eps - eps_eq, and those of q, p and j when there is a flux
    C te, tp, phi2 = phi, phi3 = phi;
    if constexpr (CONV == 1 || DIFF != 0) phi2 = vmul(phi, phi);
    if constexpr (CONV == 1 || DIFF == 2) phi3 = vmul(phi2, phi);
    if constexpr (sizeof(C) == 8 && !std::is_same<C, F2>::value) {
        te = ne;
        tp = eps;
        if constexpr (DIFF == 1) {
            te = vmad(phi, phi, te);
            tp = vmad(phi, phi, tp);
        }
        if constexpr (CONV == 1 || DIFF == 2) {
            te = vmad(k.ke3, phi3, te);
            tp = vmad(k.ke3, phi3, tp);
        }
        te = vmad(k.ke1, phi, te);
        tp = vmad(k.nkp1, phi, tp);
    } else if constexpr (CONV == 1 || DIFF != 0) {
        C h;
        if constexpr (DIFF != 1) h = vmul(k.ke3, phi3);
        else if constexpr (CONV == 1) h = vmad(k.ke3, phi3, phi2);
        else h = phi2;
        te = vadd(ne, vmad(k.ke1, phi, h));
        tp = vadd(eps, vmad(k.nkp1, phi, h));
    } else {
        te = vmad(k.ke1, phi, ne);
        tp = vmad(k.nkp1, phi, eps);
    }
    if constexpr (FLUX) {
        const C beta = CONV == 1 ? phi2 : phi, cphi = CONV == 1 ? phi3 : phi;
        qx = vmad(k.bx, beta, qx);
        qy = vmad(k.by, beta, qy);
        jx = vmad(k.nbx, beta, jx);
        jy = vmad(k.nby, beta, jy);
        pxx = vmad(k.nkxx, cphi, pxx);
        pxy = vmad(k.nkxy, cphi, pxy);
    }
    C na3 = k.na3, na35 = k.na35, na5 = k.na5;
    if constexpr (NODE_K) {
        na3 = vmul(A3, k.nsixth);
        na35 = vmul(A35, k.nsixth);
        na5 = vmul(A5, k.nsixth);
    }
    C jxn = vmad(na3, jx, vmul(na35, jy));                         // dj/6
    C jyn = vmad(na35, jx, vmul(na5, jy));
    C pp = vmul(k.nse2, tp), nee = vmul(k.nse1, te);               // deps/36, -de/36
    C base_a, base_d;                                              // even changes of the axes, of the diagonals
    C X1, X2, Y1, Y2;                                              // odd changes of the x axis, of the diagonals; y
    // (one branch holds all that a source adds: with a second one for the odd changes the
    // compiler ran its four FP64 operations without a source too, 5 % of a step)
    auto odd = [&]() {
        X1 = vmad(k.sq4, qx, jxn);
        X2 = vmad(k.nsq4, qx, jxn);
        Y1 = vmad(k.sq6, qy, jyn);
        Y2 = vmad(k.nsq6, qy, jyn);
    };
    if (S_ON) {
        // (I - S/2) M0 R_vec of Eq. 34 with Bt = B' (Scheme B), M0 R_vec =
        // (R, -2R, R, B'_x R, -B'_x R, B'_y R, -B'_y R, 0, 0); R here is R/9, the source's
        // factors carry the 9
        const C R = vmad(k.r1, phi, k.r0);
        nee = vmad(k.nhe1, R, nee);
        pp = vmad(k.he2, R, pp);
        f[0] = vadd(f[0], vmad(k.four, vadd(pp, nee), R));
        base_a = vmad(k.mtwo, pp, vadd(R, nee));
        base_d = vmad(k.mtwo, nee, vadd(R, pp));
        if constexpr (FLUX) {
            const C S = CONV == 1 ? vmul(R, phi) : R;
            if constexpr (NODE_K) {
                const C sx = vmul(k.ux9, S), sy = vmul(k.uy9, S);
                const C c3 = vmad(k.half, na3, k.sixth), c35 = vmul(k.half, na35), c5 = vmad(k.half, na5, k.sixth);
                jxn = vmad(c3, sx, vmad(c35, sy, jxn));
                jyn = vmad(c35, sx, vmad(c5, sy, jyn));
            } else {
                jxn = vmad(k.jsx, S, jxn);
                jyn = vmad(k.jsy, S, jyn);
            }
            odd();
            X1 = vmad(k.hqx2, S, X1);
            X2 = vmad(k.hqx, S, X2);
            Y1 = vmad(k.hqy2, S, Y1);
            Y2 = vmad(k.hqy, S, Y2);
        } else {
            odd();
        }
    } else {
        f[0] = vmad(k.four, vmad(k.nse1, te, pp), f[0]);
        base_a = vmad(k.mtwo, pp, nee);
        base_d = vmad(k.mtwo, nee, pp);
        odd();
    }
    const C t1 = vmad(k.nsp7, pxx, base_a), t2 = vmad(k.sp7, pxx, base_a);
    const C t3 = vmad(k.nsp8, pxy, base_d), t4 = vmad(k.sp8, pxy, base_d);
    f[1] = vadd(f[1], vadd(t1, X1));
    f[3] = vadd(f[3], vsub(t1, X1));
    f[2] = vadd(f[2], vadd(t2, Y1));
    f[4] = vadd(f[4], vsub(t2, Y1));
    const C PP = vadd(X2, Y2), MM = vsub(X2, Y2);
    f[5] = vadd(f[5], vadd(t3, PP));
    f[7] = vadd(f[7], vsub(t3, PP));
    f[6] = vadd(f[6], vsub(t4, MM));
    f[8] = vadd(f[8], vadd(t4, MM));
}

// The collision of the storage type: BF16-shifted storage keeps collide() of
// lbm_device.cuh (its rounding to bf16 turns a last-bit change of the arithmetic
// into one of 2^-9 of the deviation), FP64 and FP32 run relax().
template <int PREC, class C, int CONV, int DIFF, bool NODE_K>
__device__ __forceinline__ void collide_stored(const Params<C> &p, C f[9], C A3, C A35, C A5, C &phi)
{
    if constexpr (PREC == LBM_BF16S) collide<C, CONV, DIFF, NODE_K>(p, f, A3, A35, A5, phi);
    else relax<C, CONV, DIFF, NODE_K>(p.k, p.has_src != 0, f, A3, A35, A5, phi);
}

// The anti-bounce-back term of direction k at a node whose link leaves through
// an x wall (ox), a y wall (oy) or both: the sides follow from the signs of c_k.
// The host's table serves the families of relax(); the others, which the general
// kernels run, and BF16-shifted storage form the term here.
template <int PREC, class C, int CONV, int DIFF>
__device__ __forceinline__ C wall_value(const Params<C> &p, int k, bool ox, bool oy)
{
    if constexpr (PREC == LBM_BF16S || CONV >= 2 || DIFF >= 3) {
        const C wx = cx(k) > 0 ? p.phi_wall[0] : p.phi_wall[1];
        const C wy = cy(k) > 0 ? p.phi_wall[2] : p.phi_wall[3];
        const C phiw = (ox && oy) ? C(0.5) * (wx + wy) : (ox ? wx : wy);
        return wall_term<C, CONV, DIFF>(p, k, phiw);
    } else {
        return p.wt[k - 1][(ox ? 1 : 0) + (oy ? 2 : 0) - 1];
    }
}

}  // namespace lbm
