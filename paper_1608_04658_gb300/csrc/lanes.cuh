// Warp-per-node building blocks of the boundary and refill kernels and of
// their adjoints (arXiv 1608.04658, Secs. 2 and 3): lane i < 27 owns
// direction i; sums over directions are shuffle trees whose lane-0 result is
// broadcast, so every lane sees the same density, velocity and stabilizer.
#pragma once

#include "geom.cuh"
#include "kbc.cuh"

namespace lbm {

constexpr int BWARPS = 4;
constexpr unsigned FULL = 0xffffffffu;

template <typename R>
__device__ __forceinline__ R wsum(R v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(FULL, v, o);
    return __shfl_sync(FULL, v, 0);
}

// Sums of N values over the warp, broadcast to every lane.  At each of the
// first steps of the butterfly a lane hands on half of its values and keeps
// the other half, so that N values take about N + 3 exchanges and N
// broadcasts where one tree each takes 6 N (6 values: 8 + 6 against 36).  The
// partners of every addition are those of wsum's tree, so each sum has its bits.
// wsum_scatter6 leaves value k in lane wsum_owner6(k) and the three after it.
template <typename R>
__device__ __forceinline__ R wexchange(R keep_lo, R keep_hi, int lane, int o)
{
    const bool hi = lane & o;
    const R keep = hi ? keep_hi : keep_lo, send = hi ? keep_lo : keep_hi;
    return keep + __shfl_xor_sync(FULL, send, o);
}
template <typename R>
__device__ __forceinline__ R wsum_scatter6(const R v[6], int lane)
{
    const R a0 = wexchange(v[0], v[3], lane, 16), a1 = wexchange(v[1], v[4], lane, 16),
            a2 = wexchange(v[2], v[5], lane, 16);
    const R b0 = wexchange(a0, a2, lane, 8), b1 = wexchange(a1, R(0), lane, 8);
    R c = wexchange(b0, b1, lane, 4);
    c += __shfl_xor_sync(FULL, c, 2);
    return c + __shfl_xor_sync(FULL, c, 1);
}
// the first lane that holds value k of wsum_scatter6
__host__ __device__ constexpr int wsum_owner6(int k) { return (k >= 3 ? 16 : 0) + (k % 3 == 2 ? 8 : 0) + (k % 3 == 1 ? 4 : 0); }
template <typename R>
__device__ __forceinline__ void wsum6(R v[6], int lane)
{
    const R c = wsum_scatter6(v, lane);
#pragma unroll
    for (int k = 0; k < 6; ++k) v[k] = __shfl_sync(FULL, c, wsum_owner6(k));
}
template <typename R>
__device__ __forceinline__ void wsum4(R v[4], int lane)
{
    const R a0 = wexchange(v[0], v[2], lane, 16), a1 = wexchange(v[1], v[3], lane, 16);
    R c = wexchange(a0, a1, lane, 8);
    c += __shfl_xor_sync(FULL, c, 4);
    c += __shfl_xor_sync(FULL, c, 2);
    c += __shfl_xor_sync(FULL, c, 1);
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = __shfl_sync(FULL, c, (k >= 2 ? 16 : 0) + (k & 1 ? 8 : 0));
}
template <typename R>
__device__ __forceinline__ void wsum2(R v[2], int lane)
{
    R c = wexchange(v[0], v[1], lane, 16);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) c += __shfl_xor_sync(FULL, c, o);
    v[0] = __shfl_sync(FULL, c, 0);
    v[1] = __shfl_sync(FULL, c, 16);
}

template <typename R>
__device__ __forceinline__ R pick(const R e[3], int c)
{
    return c < 0 ? e[0] : (c > 0 ? e[2] : e[1]);
}

// Lane-parallel KBC collision: lane i < 27 holds the shifted population g_i.
template <typename R>
__device__ R kbc_collide_lanes(R g, int i, R beta, R inv_beta, R rho0, int gamma_mode, bool &ok)
{
    const bool act = i < Q;
    const int cx = act ? cx_of(i) : 0, cy = act ? cy_of(i) : 0, cz = act ? cz_of(i) : 0;
    const R gv = act ? g : R(0);
    const int lane = threadIdx.x & 31;
    R m4[4] = {gv, R(cx) * gv, R(cy) * gv, R(cz) * gv};
    wsum4(m4, lane);
    const R drho = m4[0], jx = m4[1], jy = m4[2], jz = m4[3];
    const R rho = rho0 + drho;
    ok = rho > R(0) && rho < R(1e30);
    const R inv_rho = rcp(rho);
    R ex[3], ey[3], ez[3], rx[3], ry[3], rz[3];
    axis_eq(jx * inv_rho, ex, rx);
    axis_eq(jy * inv_rho, ey, ry);
    axis_eq(jz * inv_rho, ez, rz);
    const R exy = pick(ex, cx) + pick(ey, cy) + pick(ex, cx) * pick(ey, cy);
    const R E = exy + pick(ez, cz) + exy * pick(ez, cz);
    const R geq = act ? weight<R>(i) * (drho + rho * E) : R(0);
    const R d = gv - geq;
    R p6[6] = {R(cx * cx) * d, R(cy * cy) * d, R(cz * cz) * d, R(cx * cy) * d, R(cx * cz) * d, R(cy * cz) * d};
    wsum6(p6, lane);
    const R pxx = p6[0], pyy = p6[1], pzz = p6[2], pxy = p6[3], pxz = p6[4], pyz = p6[5];
    const R nxz = pxx - pzz, nyz = pyy - pzz;
    const R ds = act ? shear_part_raw<R>(i, nxz, nyz, pxy, pxz, pyz) : R(0);
    const R dh = d - ds;
    const R ifeq = act ? inv_rho * inv_weight<R>(i) * pick(rx, cx) * pick(ry, cy) * pick(rz, cz) : R(0);
    R s2[2] = {ds * dh * ifeq, dh * dh * ifeq};
    wsum2(s2, lane);
    const R sh = s2[0], hh = s2[1];
    R gam = R(2);
    if (gamma_mode != LBM_GAMMA_LBGK && hh > gamma_floor<R>())
        gam = inv_beta - (R(2) - inv_beta) * sh * rcp(hh);
    if (gamma_mode == LBM_GAMMA_EXACT && hh > gamma_floor<R>()) {
        // exact stabilizer (see exact_gamma) with the directions on the lanes
        const R e = act ? (dh - (R(2) * beta - R(1)) * ds) * ifeq : R(0);
        const R B = act ? beta * dh * ifeq : R(0);
        R lo = B < R(0) ? (R(1) + e) / B : -R(1e30), hi = B > R(0) ? (R(1) + e) / B : R(1e30);
        for (int o = 16; o > 0; o >>= 1) {
            lo = fmax(lo, __shfl_xor_sync(0xffffffffu, lo, o));
            hi = fmin(hi, __shfl_xor_sync(0xffffffffu, hi, o));
        }
        R g = gam;
        if (!(g > lo && g < hi))
            g = (lo > -R(1e29) && hi < R(1e29)) ? R(0.5) * (lo + hi) : (g <= lo ? lo + R(1) : hi - R(1));
        const R tol = sizeof(R) == 8 ? R(1e-14) : R(1e-6);
        for (int it = 0; it < 40; ++it) {
            const R x = e - g * B;
            const R r = wsum(act ? dh * log1p_r(x) : R(0));
            const R dr = wsum(act ? -dh * B / (R(1) + x) : R(0));
            if (r > R(0)) lo = g;
            else hi = g;
            const R step = dr < R(0) ? r / dr : R(0);
            if (fabs(step) <= tol * fmax(R(1), fabs(g))) {
                g -= step;
                break;
            }
            R gn = g - step;
            if (!(gn > lo && gn < hi)) gn = R(0.5) * (lo + hi);
            g = gn;
        }
        gam = g;
    }
    return geq + (R(1) - beta * gam) * d + beta * (gam - R(2)) * ds;
}

// Shifted Grad distribution g*_i = f*_i - W_i rho0 (Eq. grad, c_s^2 = 1/3):
//   f*_i = W_i [rho + 3 rho c.u + (9/2) Qt : (c c - I/3)],  Qt = Pi - rho/3 I.
template <typename R>
__device__ __forceinline__ R grad_shifted(int i, R rho, R rho0, const R u[3], const R Qt[6])
{
    const R cx = R(cx_of(i)), cy = R(cy_of(i)), cz = R(cz_of(i));
    const R cu = cx * u[0] + cy * u[1] + cz * u[2];
    // Qt = (xx, yy, zz, xy, xz, yz)
    const R qcc = Qt[0] * cx * cx + Qt[1] * cy * cy + Qt[2] * cz * cz
                + R(2) * (Qt[3] * cx * cy + Qt[4] * cx * cz + Qt[5] * cy * cz);
    const R tr = (Qt[0] + Qt[1] + Qt[2]) * R(1.0 / 3.0);
    return weight<R>(i) * ((rho - rho0) + R(3) * rho * cu + R(4.5) * (qcc - tr));
}

// Qt = rho u u - (rho c_s^2 / (2 beta)) (grad u + grad u^T)  (Eqs. pressure, pressure2)
template <typename R>
__device__ __forceinline__ void pressure_excess(R rho, const R u[3], const R du[3][3], R beta, R Qt[6])
{
    const R k = rho / (R(6) * beta);
    Qt[0] = rho * u[0] * u[0] - k * R(2) * du[0][0];
    Qt[1] = rho * u[1] * u[1] - k * R(2) * du[1][1];
    Qt[2] = rho * u[2] * u[2] - k * R(2) * du[2][2];
    Qt[3] = rho * u[0] * u[1] - k * (du[0][1] + du[1][0]);
    Qt[4] = rho * u[0] * u[2] - k * (du[0][2] + du[2][0]);
    Qt[5] = rho * u[1] * u[2] - k * (du[1][2] + du[2][1]);
}

// velocity gradient du[a][b] = d u_a / d x_b from the staged neighbourhood
template <typename R>
__device__ __forceinline__ void fd_gradient(const R (*su)[4], const int *sok, const R uc[3], R du[3][3])
{
    const int step[3] = {9, 3, 1};
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const int kp = 13 + step[b], km = 13 - step[b];
        const bool op = sok[kp], om = sok[km];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            R v = R(0);
            if (op && om) v = R(0.5) * (su[kp][1 + a] - su[km][1 + a]);
            else if (op) v = su[kp][1 + a] - uc[a];
            else if (om) v = uc[a] - su[km][1 + a];
            du[a][b] = v;
        }
    }
}

// Stage populations of neighbourhood nodes selected by 'need' into sf[k][i]
// and their density/velocity into su[k] (lane k).  sok[k] must be set.  The
// nodes of a batch are loaded before any is stored, so that their latencies
// overlap; one batch holds the nodes of a flat wall (itself, six neighbours,
// eight more links).  (All 27 in line, most of them skipped, was a third of the
// boundary kernel's instructions.)  ALL: all 27 at once, for a refilled node,
// which needs most of them.
template <typename S, typename R, bool ALL = false>
__device__ __forceinline__ void stage(const Lattice &L, const S *fa, int lane, int nk,
                                      uint32_t need, R (*sf)[28], R (*su)[4], const int *sok)
{
    constexpr int BATCH = 16;
    const S *p = fa + (size_t)(lane < Q ? lane : 0) * (size_t)L.N;
    if constexpr (ALL) {
        R v[Q];
#pragma unroll
        for (int k = 0; k < Q; ++k) {
            const int node = __shfl_sync(FULL, nk, k);
            v[k] = ((need >> k) & 1u) && node >= 0 && lane < Q ? Codec<S>::load(p + node) : R(0);
        }
#pragma unroll
        for (int k = 0; k < Q; ++k)
            if (lane < Q) sf[k][lane] = v[k];
    }
    for (uint32_t m = ALL ? 0u : need; m;) {
        R v[BATCH];
        uint32_t t = m;
#pragma unroll
        for (int j = 0; j < BATCH; ++j) {
            v[j] = R(0);
            if (t) {
                const int node = __shfl_sync(FULL, nk, __ffs(t) - 1);
                t &= t - 1;
                if (node >= 0 && lane < Q) v[j] = Codec<S>::load(p + node);
            }
        }
#pragma unroll
        for (int j = 0; j < BATCH; ++j)
            if (m) {
                if (lane < Q) sf[__ffs(m) - 1][lane] = v[j];
                m &= m - 1;
            }
    }
    __syncwarp();
    if (lane < Q && ((need >> lane) & 1u) && nk >= 0) {
        R f[28];
        if constexpr (sizeof(R) == 4) {
            // (rows of 28 floats: eight lanes' quarter rows lie in different banks)
#pragma unroll
            for (int c = 0; c < 7; ++c) {
                const float4 q = reinterpret_cast<const float4 *>(sf[lane])[c];
                f[4 * c] = q.x;
                f[4 * c + 1] = q.y;
                f[4 * c + 2] = q.z;
                f[4 * c + 3] = q.w;
            }
        } else {
#pragma unroll
            for (int i = 0; i < Q; ++i) f[i] = sf[lane][i];
        }
        R r = 0, j[3] = {0, 0, 0};
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const int c[3] = {cx_of(i), cy_of(i), cz_of(i)};
            r += f[i];
#pragma unroll
            for (int a = 0; a < 3; ++a)
                if (c[a]) j[a] = c[a] > 0 ? j[a] + f[i] : j[a] - f[i];
        }
        const R rho = R(L.rho0) + r;
        su[lane][0] = rho;
        su[lane][1] = j[0] / rho;
        su[lane][2] = j[1] / rho;
        su[lane][3] = j[2] / rho;
    }
    __syncwarp();
}

__device__ __forceinline__ void node_xyz(const Lattice &L, int n, int &x, int &y, int &z)
{
    const int r = n / L.nx;
    x = n - r * L.nx;
    z = r / L.ny;
    y = r - z * L.ny;
}

// offset of the neighbour along direction i away from the box faces
__device__ __forceinline__ int direction_offset(const Lattice &L, int i)
{
    return cx_of(i) + L.nx * (cy_of(i) + L.ny * cz_of(i));
}

// neighbour x + c_i (-1 outside the box) and pull source x - c_i (-1 an
// equilibrium face's value, -2 the bounce-back at a wall, which wins) of a node
// on a box face; out of line, most bodies touch none
__device__ __noinline__ static void face_sources(const Lattice &L, int x, int y, int z, int i, int &nk, int &src)
{
    const int c[3] = {cx_of(i), cy_of(i), cz_of(i)}, p0[3] = {x, y, z}, nn[3] = {L.nx, L.ny, L.nz};
    int p[3], kind = 0;
    for (int a = 0; a < 3; ++a) {
        p[a] = p0[a] - c[a];
        if (p[a] >= 0 && p[a] < nn[a]) continue;
        const int face = L.face[2 * a + (p[a] < 0 ? 0 : 1)];
        if (face == LBM_FACE_PERIODIC) p[a] = (p[a] + nn[a]) % nn[a];
        else if (face == LBM_FACE_OUTFLOW) p[a] = p[a] < 0 ? 0 : nn[a] - 1;
        else kind = max(kind, face == LBM_FACE_WALL ? 2 : 1);
    }
    src = kind ? -kind : p[0] + L.nx * (p[1] + L.ny * p[2]);
    nk = neighbour(L, x, y, z, c[0], c[1], c[2]);
}

// Lane i < 27 of a boundary node: neighbour nk and pull source src along its
// direction (face_sources), fluid marks of the neighbours into sok; returns the
// missing set, the directions whose source is solid.  Off the faces sources and
// neighbours are the same nodes, so one mark per lane gives both.  off:
// direction_offset of the lane.
__device__ __forceinline__ uint32_t node_links(const Lattice &L, const uint8_t *flags, int n, int x, int y,
                                               int z, int lane, int off, int *sok, int &nk, int &src)
{
    const bool act = lane < Q;
    nk = src = -1;
    if (x > 0 && x < L.nx - 1 && y > 0 && y < L.ny - 1 && z > 0 && z < L.nz - 1) {
        bool solid = false;
        if (act) {
            nk = n + off;
            src = n - off;
            solid = flags[nk] & FL_SOLID;
            sok[lane] = !solid;
        }
        return __brev(__ballot_sync(FULL, solid && lane != 13)) >> (32 - Q);
    }
    bool solid = false;
    if (act) {
        face_sources(L, x, y, z, lane, nk, src);
        sok[lane] = nk >= 0 && !(flags[nk] & FL_SOLID);
        solid = lane != 13 && src >= 0 && (flags[src] & FL_SOLID);
    }
    return __ballot_sync(FULL, solid);
}

}  // namespace lbm
