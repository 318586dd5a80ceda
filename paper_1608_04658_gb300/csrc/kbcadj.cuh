// Transpose of the KBC collision of one node (F1, D1) or two nodes at once (F2,
// packed FP32x2), for the bulk adjoint (arXiv 1608.04658, Sec. 2, Eq.
// kbc_relax with the analytic stabilizer).  The one-node and the two-node FP32
// forms give the same bits for a node.
#pragma once

#include "kbcm.cuh"

namespace lbm {

// lam holds dJ/df' on entry and dJ/df on exit; g are the shifted pre-collision
// populations (overwritten by d = g - g^eq).  f' = f - b (2 ds + g dh), backward:
//   ds_bar = -2b lam + a_bar dh/feq,  dh_bar = -b g lam + a_bar ds/feq + 2 b_bar dh/feq,
//   g_bar = -b <lam, dh>,  a = <ds|dh>, b = <dh|dh>, g = 1/b - (2 - 1/b) a/b,
//   df_bar = dh_bar + S^T (ds_bar - dh_bar),   feq_bar = -df_bar - (a_bar ds dh + b_bar dh^2)/feq^2,
//   then f^eq(rho, u) and u = j/rho back to f.
// As in kbc_collide_m the moments of d are those of g less the product form's,
// and 1/f^eq is taken relative to the rest direction's (every product of a_bar
// or b_bar with it is a ratio).  d ln Phi(c)/du = D0 + c dlnB per axis, so the
// velocity's adjoint needs four sums over the directions of t = feq_bar feq, as
// the density's: sum t and sum c t.
// Against 64 bits from the same state (48^3 box, FP32, lambda_T random): 3.5e-6
// after eight steps where per-direction derivatives and absolute 1/f^eq gave
// 4.2e-6, 6.4e-7 and 6.0e-7 after one.
// zero: a run-time 0 (see kbc_collide_m).
template <typename O>
__device__ __forceinline__ void kbc_vjp_v(typename O::V (&g)[Q], typename O::V (&lam)[Q], typename O::R beta,
                                          typename O::R inv_beta, typename O::R rho0, int gamma_mode, typename O::R zero)
{
    using R = typename O::R;
    using V = typename O::V;
    constexpr int NL = sizeof(V) / sizeof(R);
    V drho, jx, jy, jz, pxx, pyy, pzz, pxy, pxz, pyz;
    {
        V Rs[3], Rd[3], b[3], as[3], bd[3], x[3];
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
            Rs[r] = O::add(as[r], L[1]);
            bd[r] = O::sub(d[2], d[0]);
            Rd[r] = O::add(O::add(d[2], d[0]), d[1]);
            x[r] = O::add(O::add(s[2], s[0]), s[1]);
        }
        pyy = O::add(Rs[2], Rs[0]);
        drho = O::add(pyy, Rs[1]);
        jy = O::sub(Rs[2], Rs[0]);
        jz = O::add(O::add(b[2], b[0]), b[1]);
        pzz = O::add(O::add(as[2], as[0]), as[1]);
        pyz = O::sub(b[2], b[0]);
        jx = O::add(O::add(Rd[2], Rd[0]), Rd[1]);
        pxy = O::sub(Rd[2], Rd[0]);
        pxz = O::add(O::add(bd[2], bd[0]), bd[1]);
        pxx = O::add(O::add(x[2], x[0]), x[1]);
    }
    const V rho = O::add(O::bc(rho0), drho);
    const V irho = O::rcp(rho);
    const V ux = O::mul(jx, irho), uy = O::mul(jy, irho), uz = O::mul(jz, irho);
    const AxisV<O> X(ux), Y(uy), Z(uz);
    V sx, sy, sz, qxy, qxz, qyz;
    const V sixth = O::c(1.0 / 6.0), quarter = O::c(0.25);
    {
        const V r23 = O::mul(rho, O::c(2.0 / 3.0));
        const V nxz = O::fnma(r23, O::sub(X.sig, Z.sig), O::sub(pxx, pzz));
        const V nyz = O::fnma(r23, O::sub(Y.sig, Z.sig), O::sub(pyy, pzz));
        sx = O::mul(O::sub(O::add(nxz, nxz), nyz), sixth);
        sy = O::mul(O::sub(O::add(nyz, nyz), nxz), sixth);
        sz = O::neg(O::add(sx, sy));
        qxy = O::mul(quarter, O::fnma(jx, uy, pxy));
        qxz = O::mul(quarter, O::fnma(jx, uz, pxz));
        qyz = O::mul(quarter, O::fnma(jy, uz, pyz));
    }
    const auto W = [](int i) {
        const int nz = nonzero_of(i);
        return O::c(nz == 0 ? 8.0 / 27.0 : nz == 1 ? 2.0 / 27.0 : nz == 2 ? 1.0 / 54.0 : 1.0 / 216.0);
    };
    const auto shear = [&](int i) {
        const V sv = shear_v<V>(i, sx, sy, sz, qxy, qxz, qyz);
        return shear_sign(i) > 0 ? sv : O::neg(sv);
    };
    const V Ry[2] = {Y.r4(-1), Y.r4(1)}, Rz[2] = {Z.r4(-1), Z.r4(1)};
    // d in place; a, b and <lam, dh>
    V sh = O::c(0.0), hh = O::c(0.0), lh = O::c(0.0);
    {
        V ey[3], ez[3], pz[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            ey[c] = Y.e(c - 1);
            ez[c] = O::fma(rho, Z.e(c - 1), drho);
            pz[c] = Z.phi(c - 1);
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const V ex = O::mul(rho, X.e(a - 1)), px = O::mul(rho, X.phi(a - 1));
            const V Rx = a == 1 ? O::c(1.0) : X.r4(a - 1);
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const V exy = O::fma(ey[b], px, ex);
                const V Rxy = b == 1 ? Rx : a == 1 ? Ry[b / 2] : O::mul(Rx, Ry[b / 2]);
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    const int i = 9 * a + 3 * b + c, nz = nonzero_of(i);
                    const V d = O::fnma(W(i), O::fma(exy, pz[c], ez[c]), g[i]);
                    const V r = c == 1 ? Rxy : O::mul(Rxy, Rz[c / 2]);
                    g[i] = d;
                    if (nz == 1 || nz == 2) {
                        const V ds = shear(i), dh = O::sub(d, ds), t = O::mul(dh, r);
                        sh = O::fma(ds, t, sh);
                        hh = O::fma(dh, t, hh);
                        lh = O::fma(lam[i], dh, lh);
                    } else {
                        hh = O::fma(d, O::mul(d, r), hh);
                        lh = O::fma(lam[i], d, lh);
                    }
                }
            }
        }
    }
    // the stabilizer and the adjoints of a and b; where f is an equilibrium to
    // rounding the stabilizer is 2 and constant
    R abv[NL], bbv[NL], chv[NL];
    const R kk = O1<R>::sub(R(2), inv_beta);
#pragma unroll
    for (int k = 0; k < NL; ++k) {
        const R shk = O::lane(sh, k), hhk = O::lane(hh, k);
        const bool analytic = gamma_mode == LBM_GAMMA_ANALYTIC && has_stabilizer(hhk, O::lane(rho, k));
        const R ihh = analytic ? rcp_fast(hhk) : R(0);
        const R ratio = O1<R>::mul(shk, ihh);
        const R gam = analytic ? O1<R>::sub(inv_beta, O1<R>::mul(kk, ratio)) : R(2);
        // (kk gb)(sh/hh)/hh: the square hh^2 would underflow in FP32 near rest
        const R kgb = O1<R>::mul(kk, O1<R>::mul(-beta, O::lane(lh, k)));
        abv[k] = O1<R>::mul(-kgb, ihh);
        bbv[k] = O1<R>::mul(O1<R>::mul(kgb, ratio), ihh);
        chv[k] = O1<R>::mul(-beta, gam);
    }
    const V ab = O::make(abv[0], abv[NL - 1]), bb = O::make(bbv[0], bbv[NL - 1]), ch = O::make(chv[0], chv[NL - 1]);
    const V bb2 = O::add(bb, bb), csh = O::sub(O::bc(R(-2) * beta), ch), ab2 = O::sub(ab, bb2);
    // shear sums of ds_bar - dh_bar = (cl_s - cl_h) lam + (ab (dh - ds) - 2 bb dh)/feq
    V S6[6] = {O::c(0.0), O::c(0.0), O::c(0.0), O::c(0.0), O::c(0.0), O::c(0.0)};
    AxisV<O> X2;
    X2.t = O::add(X.t, O::bc(zero));
    X2.sig = O::add(X.sig, O::bc(zero));
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const V Rx = a == 1 ? O::c(1.0) : X2.r4(a - 1);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const V Rxy = b == 1 ? Rx : a == 1 ? Ry[b / 2] : O::mul(Rx, Ry[b / 2]);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int i = 9 * a + 3 * b + c, nz = nonzero_of(i);
                if (nz != 1 && nz != 2) continue;
                const V r = c == 1 ? Rxy : O::mul(Rxy, Rz[c / 2]);
                const V ds = shear(i), dh = O::sub(g[i], ds);
                const V t = O::fma(O::fnma(ab, ds, O::mul(ab2, dh)), r, O::mul(csh, lam[i]));
                const int m = nz == 1 ? (a != 1 ? 0 : b != 1 ? 1 : 2) : (c == 1 ? 3 : b == 1 ? 4 : 5);
                S6[m] = shear_sign(i) > 0 ? O::add(S6[m], t) : O::sub(S6[m], t);
            }
        }
    }
    const V nxzb = O::mul(O::sub(O::sub(O::add(S6[0], S6[0]), S6[1]), S6[2]), sixth);
    const V nyzb = O::mul(O::sub(O::sub(O::add(S6[1], S6[1]), S6[0]), S6[2]), sixth);
    const V pzzb = O::neg(O::add(nxzb, nyzb));
    const V pxyb = O::mul(quarter, S6[3]), pxzb = O::mul(quarter, S6[4]), pyzb = O::mul(quarter, S6[5]);
    // df_bar into lam, and the sums of t = feq_bar feq
    V t0 = O::c(0.0), tx = O::c(0.0), ty = O::c(0.0), tz = O::c(0.0);
    AxisV<O> X3;
    X3.t = O::add(X2.t, O::bc(zero));
    X3.sig = O::add(X2.sig, O::bc(zero));
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const V px = O::mul(rho, X3.phi(a - 1));
        const V Rx = a == 1 ? O::c(1.0) : X3.r4(a - 1);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const V pxy2 = O::mul(px, Y.phi(b - 1));
            const V Rxy = b == 1 ? Rx : a == 1 ? Ry[b / 2] : O::mul(Rx, Ry[b / 2]);
            V Sxy = a != 1 ? nxzb : nyzb;
            if (a != 1 && b != 1) Sxy = (a - 1) * (b - 1) > 0 ? O::add(O::add(nxzb, nyzb), pxyb) : O::sub(O::add(nxzb, nyzb), pxyb);
            V tl[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int i = 9 * a + 3 * b + c, nz = nonzero_of(i);
                const V r = c == 1 ? Rxy : O::mul(Rxy, Rz[c / 2]);
                // rest and corners carry no shear part (ds = 0, dh = d)
                const bool sh_i = nz == 1 || nz == 2;
                const V ds = sh_i ? shear(i) : O::c(0.0);
                const V dh = sh_i ? O::sub(g[i], ds) : g[i];
                const V e = sh_i ? O::fma(ab, ds, O::mul(bb, dh)) : O::mul(bb, dh);  // ab ds + bb dh
                V dfb = O::fma(O::fma(bb, dh, e), r, O::mul(ch, lam[i]));
                if (a != 1 || b != 1) dfb = O::add(dfb, Sxy);
                if (c != 1) dfb = O::add(dfb, pzzb);
                if (a != 1 && c != 1) dfb = (a - 1) * (c - 1) > 0 ? O::add(dfb, pxzb) : O::sub(dfb, pxzb);
                if (b != 1 && c != 1) dfb = (b - 1) * (c - 1) > 0 ? O::add(dfb, pyzb) : O::sub(dfb, pyzb);
                const V feq = O::mul(W(i), O::mul(pxy2, Z.phi(c - 1)));
                tl[c] = O::fma(O::mul(e, dh), r, O::mul(dfb, feq));  // -t
                lam[i] = O::add(lam[i], dfb);
            }
            const V s = O::add(O::add(tl[0], tl[2]), tl[1]);
            t0 = O::add(t0, s);
            tz = O::add(tz, O::sub(tl[2], tl[0]));
            if (a != 1) tx = a == 2 ? O::add(tx, s) : O::sub(tx, s);
            if (b != 1) ty = b == 2 ? O::add(ty, s) : O::sub(ty, s);
        }
    }
    // ub_a = D0_a sum t + dlnB_a sum c_a t with, s = sigma' = 3u/S and Phi(0) = 1 - sigma,
    //   D0 = -s/Phi(0),  dlnB = (d/du)(ln Phi(1) - ln Phi(-1))/2
    //                         = ((2s + 3) Phi(-1) - (2s - 3) Phi(1)) / (2 Phi(0)^2)
    const auto axis = [&](const AxisV<O> &A, V J) {
        const V s = O::mul(A.t, O::rcp(O::add(A.sig, O::c(1.0))));
        const V i0 = O::rcp(A.phi(0)), two_s = O::add(s, s);
        const V up = O::mul(O::add(two_s, O::c(3.0)), A.phi(-1)), dn = O::mul(O::sub(two_s, O::c(3.0)), A.phi(1));
        const V dlnB = O::mul(O::mul(O::c(0.5), O::sub(up, dn)), O::mul(i0, i0));
        return O::fma(dlnB, J, O::mul(O::neg(O::mul(s, i0)), t0));
    };
    // (the sums above are of -t)
    const V ni = O::neg(irho);
    const V bx = O::mul(axis(X3, tx), ni), by = O::mul(axis(Y, ty), ni), bz = O::mul(axis(Z, tz), ni);
    const V rb = O::fnma(bz, uz, O::fnma(by, uy, O::fnma(bx, ux, O::mul(t0, ni))));
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const V va = a == 1 ? rb : a == 2 ? O::add(rb, bx) : O::sub(rb, bx);
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            const V vb = b == 1 ? va : b == 2 ? O::add(va, by) : O::sub(va, by);
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const int i = 9 * a + 3 * b + c;
                lam[i] = O::add(lam[i], c == 1 ? vb : c == 2 ? O::add(vb, bz) : O::sub(vb, bz));
            }
        }
    }
}

}  // namespace lbm
