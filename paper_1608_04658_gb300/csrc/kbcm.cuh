// KBC collision of one node (F1, D1) or two nodes at once (F2, packed FP32x2)
// from its moments: the form that FP64 storage, the exact stabilizer, launches
// without marks and large boxes take (see launch_bulk_t).  Same mathematics as kbc_collide
// (arXiv 1608.04658, Sec. 2, Eqs. kineticEq, kbc_relax, feq_min, gamma_min and
// the analytic stabilizer); the one-node and the two-node FP32 forms give the
// same bits for a node.
#pragma once

#include "kbcv.cuh"

namespace lbm {

// one node in double
struct D1 {
    using V = double;
    using R = double;
    static __device__ __forceinline__ V c(double s) { return s; }
    static __device__ __forceinline__ V bc(double s) { return s; }
    static __device__ __forceinline__ V add(V a, V b) { return __dadd_rn(a, b); }
    static __device__ __forceinline__ V sub(V a, V b) { return __dsub_rn(a, b); }
    static __device__ __forceinline__ V mul(V a, V b) { return __dmul_rn(a, b); }
    static __device__ __forceinline__ V fma(V a, V b, V d) { return __fma_rn(a, b, d); }
    static __device__ __forceinline__ V fnma(V a, V b, V d) { return __fma_rn(-a, b, d); }
    static __device__ __forceinline__ V neg(V a) { return -a; }
    static __device__ __forceinline__ V rcp(V a) { return rcp_fast(a); }
    static __device__ __forceinline__ V sqrt(V a) { return sqrt_fast(a); }
    static __device__ __forceinline__ double lane(V a, int) { return a; }
    static __device__ __forceinline__ V make(double a, double) { return a; }
};
// the scalar operations of a lane
template <typename R> struct O1;
template <> struct O1<float> : F1 {};
template <> struct O1<double> : D1 {};

// 1-D equilibrium factors of one axis.  The product form's factor w(c) Phi(c)
// is the entropic equilibrium of the three velocities -1, 0, 1, so its
// zeroth and first moments are 1 and u: with Phi(0) = 2 - S = 1 - sigma,
//   Phi(+-1) = 1 + 2 sigma +- 3u,   e(c) = Phi(c) - 1 without a division,
// and Phi(1) Phi(-1) = Phi(0)^2 (Phi(c) = Phi(0) B^c) gives the reciprocals.
template <typename O>
struct AxisV {
    using V = typename O::V;
    V t, sig;  // 3u and sigma = S - 1 = 3u^2/(S + 1)
    AxisV() = default;
    __device__ __forceinline__ explicit AxisV(V u)
    {
        t = O::mul(O::c(3.0), u);
        const V q = O::mul(t, u);
        sig = O::mul(q, O::rcp(O::add(O::sqrt(O::add(q, O::c(1.0))), O::c(1.0))));
    }
    __device__ __forceinline__ V e(int c) const { return c == 0 ? O::neg(sig) : O::fma(O::c(2.0), sig, c > 0 ? t : O::neg(t)); }
    __device__ __forceinline__ V phi(int c) const { return O::add(O::c(1.0), e(c)); }
    // [1/(w Phi)](c) / [1/(w Phi)](0) = 4 Phi(-c) / Phi(0), c = +-1: the weight of
    // direction c in the entropic products relative to the centre's
    __device__ __forceinline__ V r4(int c) const { return O::mul(phi(-c), O::mul(O::c(4.0), O::rcp(phi(0)))); }
};

// the shear values of a node (faces, signed quarter off-diagonal moments)
template <typename V>
struct Shear {
    V sx, sy, sz, qxy, qxz, qyz;
    __device__ __forceinline__ V at(int i) const { return shear_v<V>(i, sx, sy, sz, qxy, qxz, qyz); }
};

// Whether a node's stabilizer is defined (gamma_floor, where f is an equilibrium
// to rounding it is 2), for a product hh = <dh|dh> taken with 1/f^eq relative to
// the rest direction's, 27/(8 rho): hh goes with rho^2, the floor is one of
// <dh|dh> itself, which goes with rho.  The second bound keeps 1/hh finite.
__device__ __forceinline__ bool has_stabilizer(float hh, float rho)
{
    return hh > gamma_floor<float>() * (float)(8.0 / 27.0) * rho && hh > 1.2e-38f;
}
__device__ __forceinline__ bool has_stabilizer(double hh, double rho)
{
    return hh > gamma_floor<double>() * (8.0 / 27.0) * rho && hh > 2.3e-308;
}

// Root of Eq. (gamma_min) per lane (of those in has) from the analytic value gam
// (see exact_gamma): with x_i = f'_i(gam)/f^eq_i - 1 and t_i = b dh_i/f'_i(gam),
//   r(gam + s) = sum dh_i log(1 + x_i) - s sum dh_i t_i - s^2/2 sum dh_i t_i^2 - ...,
// all three sums in one pass (log(1 + x) and 1/(1 + x) by their Taylor series to
// x^6 and x^3, |x| <= 1/16: truncated below FP32's rounding, the second only
// steers the step).  The step solves the quadratic; what it leaves out, s (s
// t)^2/3 and smaller, is below the tolerance for all but nodes far from
// equilibrium: their bits are returned, and the caller updates them again with
// exact_gamma's safeguarded iteration (kbc_collide).  (A pass with log1pf in each of two iterations a node took 1.02 ms on the 256x192x128
// box, five times the time of its memory traffic.)
template <typename O>
__device__ __forceinline__ int exact_stabilizer(const typename O::V (&d)[Q], const Shear<typename O::V> &S,
                                                 typename O::V rho, const AxisV<O> &X, const AxisV<O> &Y,
                                                 const AxisV<O> &Z, int has, typename O::R beta,
                                                 typename O::R (&gam)[sizeof(typename O::V) / sizeof(typename O::R)])
{
    using V = typename O::V;
    using R = typename O::R;
    constexpr int NL = sizeof(V) / sizeof(R);
    const V k0 = O::rcp(O::mul(O::mul(rho, O::c(8.0 / 27.0)), O::mul(X.phi(0), O::mul(Y.phi(0), Z.phi(0)))));
    const V Ry[2] = {Y.r4(-1), Y.r4(1)}, Rz[2] = {Z.r4(-1), Z.r4(1)};
    R c1v[NL];
#pragma unroll
    for (int k = 0; k < NL; ++k) c1v[k] = R(1) - beta * gam[k];
    const V c1 = O::make(c1v[0], c1v[NL - 1]), c3 = O::bc(R(2) * beta - R(1)), b = O::bc(beta);
    V r0 = O::c(0.0), r1 = O::c(0.0), r2 = O::c(0.0);
    R xm[NL], tm[NL];
#pragma unroll
    for (int k = 0; k < NL; ++k) xm[k] = tm[k] = R(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const V Rx = a == 1 ? k0 : O::mul(k0, X.r4(a - 1));
#pragma unroll
        for (int l = 0; l < 3; ++l) {
            const V Rxy = l == 1 ? Rx : O::mul(Rx, Ry[l / 2]);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int i = 9 * a + 3 * l + c, nz = nonzero_of(i);
                const V ifeq = c == 1 ? Rxy : O::mul(Rxy, Rz[c / 2]);
                V dh = d[i], x;
                if (nz == 1 || nz == 2) {
                    const V ds = shear_sign(i) > 0 ? S.at(i) : O::neg(S.at(i));
                    dh = O::sub(d[i], ds);
                    x = O::mul(ifeq, O::fma(c1, dh, O::neg(O::mul(c3, ds))));
                } else {
                    x = O::mul(ifeq, O::mul(c1, dh));
                }
                V lg = O::fma(x, O::c(-1.0 / 6.0), O::c(1.0 / 5.0));
                lg = O::fma(x, lg, O::c(-1.0 / 4.0));
                lg = O::fma(x, lg, O::c(1.0 / 3.0));
                lg = O::fma(x, lg, O::c(-1.0 / 2.0));
                lg = O::mul(x, O::fma(x, lg, O::c(1.0)));
                const V inv = O::fnma(x, O::fnma(x, O::sub(O::c(1.0), x), O::c(1.0)), O::c(1.0));
                const V t = O::mul(O::mul(O::mul(b, dh), ifeq), inv), dt = O::mul(dh, t);
                r0 = O::fma(dh, lg, r0);
                r1 = O::add(r1, dt);
                r2 = O::fma(dt, t, r2);
#pragma unroll
                for (int k = 0; k < NL; ++k) {
                    xm[k] = fmax(xm[k], fabs(O::lane(x, k)));
                    tm[k] = fmax(tm[k], fabs(O::lane(t, k)));
                }
            }
        }
    }
    int again = 0;
#pragma unroll
    for (int k = 0; k < NL; ++k) {
        if (!(has >> k & 1)) continue;
        const R f0 = O::lane(r0, k), f1 = O::lane(r1, k), f2 = O::lane(r2, k), i1 = rcp_fast(f1);
        const R s1 = f0 * i1;
        const R s = s1 - R(0.5) * f2 * s1 * s1 * rcp_fast(f1 + f2 * s1);
        const R st = fabs(s) * tm[k];
        if (f1 > R(0) && xm[k] <= R(0.0625) && st <= R(0.0625) &&
            fabs(s) * st * st <= R(1e-6) * fmax(R(1), fabs(gam[k]))) {
            gam[k] += s;
        } else {
            again |= 1 << k;
        }
    }
    return again;
}

// In-place collision of the 27 shifted populations of one or two nodes, the
// same mathematics as kbc_collide_v with fewer operations (about 430 against
// 580 a node in FP32):
//   - all moments up to second order of g from one pass over the x-lines; the
//     second moments of d = g - g^eq are those less the product form's closed
//     expressions, so that the shear part is known before d is formed and d and
//     the entropic scalar products take one pass;
//   - equilibrium factors without a division (AxisV), 1/f^eq only relative to
//     the rest direction's, since the stabilizer is a ratio;
//   - rho W (E + drho/rho) with drho folded into the z factors.
// The x factors are formed again for the last pass: + zero, a run-time 0, keeps
// the compiler from holding the 27 equilibria in registers between the passes,
// which spills.  Against 64 bits its error is smaller than kbc_collide_v's
// (32^3 Taylor-Green box, 20 steps: 3.1e-7 against 4.4e-7).
// EXACT: the stabilizer that solves Eq. (gamma_min) when gamma_mode asks for it.
// Returns a bit per node (bit 0 the first, bit 1 the second) set when its
// density is finite and positive, and with EXACT above these a bit per node
// whose result is void: it needs kbc_collide's iteration.
template <typename O, bool EXACT>
__device__ __forceinline__ int kbc_collide_m(typename O::V (&g)[Q], typename O::R beta, typename O::R inv_beta,
                                             typename O::R rho0, int gamma_mode, typename O::R zero)
{
    using R = typename O::R;
    using V = typename O::V;
    constexpr int NL = sizeof(V) / sizeof(R);
    // all moments up to second order from the x-lines, a row of three (one
    // c_y) at a time
    V drho, jx, jy, jz, pxx, pyy, pzz, pxy, pxz, pyz;
    {
        V R[3], Rd[3], b[3], as[3], bd[3], x[3];
#pragma unroll
        for (int r = 0; r < 3; ++r) {
            V s[3], d[3], L[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int l = 3 * r + c;
                s[c] = O::add(g[18 + l], g[l]);
                d[c] = O::sub(g[18 + l], g[l]);
                L[c] = O::add(s[c], g[9 + l]);
            }
            as[r] = O::add(L[2], L[0]);
            b[r] = O::sub(L[2], L[0]);
            R[r] = O::add(as[r], L[1]);
            bd[r] = O::sub(d[2], d[0]);
            Rd[r] = O::add(O::add(d[2], d[0]), d[1]);
            x[r] = O::add(O::add(s[2], s[0]), s[1]);
        }
        pyy = O::add(R[2], R[0]);
        drho = O::add(pyy, R[1]);
        jy = O::sub(R[2], R[0]);
        jz = O::add(O::add(b[2], b[0]), b[1]);
        pzz = O::add(O::add(as[2], as[0]), as[1]);
        pyz = O::sub(b[2], b[0]);
        jx = O::add(O::add(Rd[2], Rd[0]), Rd[1]);
        pxy = O::sub(Rd[2], Rd[0]);
        pxz = O::add(O::add(bd[2], bd[0]), bd[1]);
        pxx = O::add(O::add(x[2], x[0]), x[1]);
    }
    const V rho = O::add(O::bc(rho0), drho);
    int ok = 0;
#pragma unroll
    for (int k = 0; k < NL; ++k) {
        const R r = O::lane(rho, k);
        ok |= (r > R(0) && r < R(1e30)) << k;
    }
    const V inv_rho = O::rcp(rho);
    const V ux = O::mul(jx, inv_rho), uy = O::mul(jy, inv_rho), uz = O::mul(jz, inv_rho);
    const AxisV<O> X(ux), Y(uy), Z(uz);
    // second moments of d = g - g^eq: those of g less the product form's,
    // P^eq_aa = rho (1/3 + 2 sigma_a / 3) (the third cancels in the
    // differences) and P^eq_ab = j_a u_b; then the shear values
    V sx, sy, sz, qxy, qxz, qyz;
    {
        const V r23 = O::mul(rho, O::c(2.0 / 3.0));
        const V nxz = O::fnma(r23, O::sub(X.sig, Z.sig), O::sub(pxx, pzz));
        const V nyz = O::fnma(r23, O::sub(Y.sig, Z.sig), O::sub(pyy, pzz));
        const V sixth = O::c(1.0 / 6.0), quarter = O::c(0.25);
        sx = O::mul(O::sub(O::add(nxz, nxz), nyz), sixth);
        sy = O::mul(O::sub(O::add(nyz, nyz), nxz), sixth);
        sz = O::neg(O::add(sx, sy));
        qxy = O::mul(quarter, O::fnma(jx, uy, pxy));
        qxz = O::mul(quarter, O::fnma(jx, uz, pxz));
        qyz = O::mul(quarter, O::fnma(jy, uz, pyz));
    }
    // g^eq_i = W_i (exy Phi_z + ez), exy = rho (e_y Phi_x + e_x), ez = rho e_z + drho
    V ey[3], ez[3], pz[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        ey[c] = Y.e(c - 1);
        ez[c] = O::fma(rho, Z.e(c - 1), drho);
        pz[c] = Z.phi(c - 1);
    }
    const auto W = [](int i) {
        const int nz = nonzero_of(i);
        return O::c(nz == 0 ? 8.0 / 27.0 : nz == 1 ? 2.0 / 27.0 : nz == 2 ? 1.0 / 54.0 : 1.0 / 216.0);
    };
    // d in place, and the entropic scalar products <ds|dh>, <dh|dh>, line by
    // line.  Only their ratio is used, so 1/f^eq_i is taken relative to that of
    // the rest direction: a product of 4 B^-+1 over the moving axes.
    V sh = O::c(0.0), hh = O::c(0.0);
    {
        const V Ry[2] = {Y.r4(-1), Y.r4(1)}, Rz[2] = {Z.r4(-1), Z.r4(1)};
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const V ex = O::mul(rho, X.e(a - 1)), px = O::mul(rho, X.phi(a - 1));
            const V Rx = a == 1 ? O::c(1.0) : X.r4(a - 1);
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const V exy = O::fma(ey[b], px, ex);
                V hl = O::c(0.0), sl = O::c(0.0);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    const int c = k == 0 ? 1 : k == 1 ? 0 : 2;  // the centre first
                    const int i = 9 * a + 3 * b + c, nz = nonzero_of(i);
                    const V d = O::fnma(W(i), O::fma(exy, pz[c], ez[c]), g[i]);
                    g[i] = d;
                    if (nz == 1 || nz == 2) {
                        const V sv = shear_v<V>(i, sx, sy, sz, qxy, qxz, qyz);
                        const V ds = shear_sign(i) > 0 ? sv : O::neg(sv);
                        const V dh = O::sub(d, ds), t = c == 1 ? dh : O::mul(dh, Rz[c / 2]);
                        hl = k == 0 ? O::mul(dh, t) : O::fma(dh, t, hl);
                        // (the rest direction and the corners carry no shear)
                        sl = k == 0 || (k == 1 && a == 1 && b == 1) ? O::mul(ds, t) : O::fma(ds, t, sl);
                    } else {
                        const V t = c == 1 ? d : O::mul(d, Rz[c / 2]);
                        hl = k == 0 ? O::mul(d, t) : O::fma(d, t, hl);
                    }
                }
                if (a == 1 && b == 1) {
                    hh = O::add(hh, hl);
                    sh = O::add(sh, sl);
                } else {
                    const V Rxy = b == 1 ? Rx : a == 1 ? Ry[b / 2] : O::mul(Rx, Ry[b / 2]);
                    hh = a + b == 0 ? O::mul(Rxy, hl) : O::fma(Rxy, hl, hh);
                    sh = a + b == 0 ? O::mul(Rxy, sl) : O::fma(Rxy, sl, sh);
                }
            }
        }
    }
    // stabilizer per node
    R gam[NL], c1v[NL], c2v[NL];
    int has = 0;  // (for the exact stabilizer, in place of the products)
#pragma unroll
    for (int k = 0; k < NL; ++k) {
        const R shk = O::lane(sh, k), hhk = O::lane(hh, k);
        gam[k] = R(2);
        if (EXACT) has |= has_stabilizer(hhk, O::lane(rho, k)) << k;
        if (gamma_mode != LBM_GAMMA_LBGK && (EXACT ? (has >> k & 1) != 0 : has_stabilizer(hhk, O::lane(rho, k))))
            gam[k] = O1<R>::sub(inv_beta, O1<R>::mul(O1<R>::mul(O1<R>::sub(R(2), inv_beta), shk), rcp_fast(hhk)));
    }
    if constexpr (EXACT) {
        if (gamma_mode == LBM_GAMMA_EXACT) {
            const Shear<V> S{sx, sy, sz, qxy, qxz, qyz};
            ok |= exact_stabilizer<O>(g, S, rho, X, Y, Z, has, beta, gam) << NL;
        }
    }
#pragma unroll
    for (int k = 0; k < NL; ++k) {
        c1v[k] = O1<R>::sub(R(1), O1<R>::mul(beta, gam[k]));
        c2v[k] = O1<R>::mul(beta, O1<R>::sub(gam[k], R(2)));
    }
    const V c1 = O::make(c1v[0], c1v[NL - 1]);
    const V c2 = O::make(c2v[0], c2v[NL - 1]);
    sx = O::mul(c2, sx);
    sy = O::mul(c2, sy);
    sz = O::mul(c2, sz);
    qxy = O::mul(c2, qxy);
    qxz = O::mul(c2, qxz);
    qyz = O::mul(c2, qyz);
    // g' = g^eq + c1 d + c2 ds
    AxisV<O> X2;
    X2.t = O::add(X.t, O::bc(zero));
    X2.sig = O::add(X.sig, O::bc(zero));
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const V ex = O::mul(rho, X2.e(a - 1)), px = O::mul(rho, X2.phi(a - 1));
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const V exy = O::fma(ey[b], px, ex);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int i = 9 * a + 3 * b + c, nz = nonzero_of(i);
                const V E = O::fma(exy, pz[c], ez[c]);
                V v;
                if (nz == 1 || nz == 2) {
                    const V sv = shear_v<V>(i, sx, sy, sz, qxy, qxz, qyz);
                    v = O::fma(W(i), E, shear_sign(i) > 0 ? sv : O::neg(sv));
                } else {
                    v = O::mul(W(i), E);
                }
                g[i] = O::fma(c1, g[i], v);
            }
        }
    }
    return ok;
}

}  // namespace lbm
