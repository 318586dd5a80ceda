// Moving-wall Grad boundary with KBC collision and momentum exchange, and the
// refill of uncovered nodes (arXiv 1608.04658, Sec. 3, Eqs. grad, pressure,
// pressure2, target velocity/density; Sec. 4.1 Galilean-invariant momentum
// exchange).
//
// One warp per listed node; lane i < 27 owns direction i.  The populations of
// the 3x3x3 neighbourhood that a node needs (itself, its six face neighbours
// for the finite-difference velocity gradient, and x_b + c_i for each missing
// i) are staged in shared memory as [node k][direction i]; lane k then forms
// the density and velocity of neighbourhood node k.  Sums over directions are
// shuffle trees whose lane-0 result is broadcast, so every lane sees the same
// density, velocity and stabilizer.
//
// Bound by instructions and their latency (3000 a node, a twentieth of the DRAM
// rate): the sources of an inner node from one mark a lane, 15 staged nodes for
// 27, a link search of five or six evaluations for 24 and no conversion of the
// wall's velocity per node took the 1024x512x64 airfoil's from 142 to 117 us
// (16,000 nodes); a body of a few hundred nodes waits for its instructions (a
// warp passes through once: 21 us for 300 nodes, before and after).
//
// Readings of points the paper leaves open (the oracle takes the same ones):
//   missing set D = {i : x_b - c_i solid at t+1}; wall point x_w = x_b - q_i c_i;
//   u_f,i from the previous-step state at x_b + c_i, or the wall velocity alone
//   when that node is not fluid; rho_dyn with rho0; f^bb_i = f'_{opp i}(x_b, t);
//   grad u: central difference where both face neighbours are fluid,
//   one-sided where one is, zero otherwise; Pi with rho_tgt and u_tgt; only
//   the missing populations are replaced; the node then collides with KBC.
//   Refill: mean density of the neighbours fluid at t (rho0 if none), the body
//   velocity (the swimmer's material velocity at the node's arc position),
//   gradient with the wall velocity at the centre.
#include "force.cuh"

namespace lbm {

// Minimum resident blocks per SM for the boundary and refill kernels: 7
// blocks of 128 threads cap them at 72 registers, so each of their blocks
// takes the registers of one bulk block on the SM it shares with the bulk
// launch beside it.
#ifndef LBM_LIST_MIN_BLOCKS
#define LBM_LIST_MIN_BLOCKS 7
#endif

template <typename S>
__global__ void __launch_bounds__(BWARPS * 32, LBM_LIST_MIN_BLOCKS) boundary_kernel(
    const __grid_constant__ Lattice L, const __grid_constant__ GeomParams G, DevBody *b, const int *blist,
    const int *bpos, double *bforce, const S *fa,
    S *fb, const uint8_t *flags)
{
    after_previous();
    using R = typename Codec<S>::R;
    __shared__ __align__(16) R s_f[BWARPS][Q][28];
    __shared__ R s_u[BWARPS][Q][4];
    __shared__ LinkScratch s_link[BWARPS];
    __shared__ WallMotion<R> s_wall;
    __shared__ int s_ok[BWARPS][Q];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    R (*sf)[28] = s_f[w];
    R (*su)[4] = s_u[w];
    int *sok = s_ok[w];
    // (the first node of the warp is read beside the count, not after it; the list
    // has room for every warp that passes this check)
    const int first = blockIdx.x * BWARPS + w;
    int n = first < G.cap_boundary ? blist[first] : 0;
    const int count = min(b->n_boundary, G.cap_boundary);
    const size_t N = (size_t)L.N;
    const R rho0 = (R)L.rho0;

    s_wall.load(G, b);
    const int i = lane;
    const bool act = i < Q;
    const int cx = act ? cx_of(i) : 0, cy = act ? cy_of(i) : 0, cz = act ? cz_of(i) : 0;
    const int off = direction_offset(L, act ? i : 13);

    for (int slot = first; slot < count; slot += gridDim.x * BWARPS) {
        if (slot != first) n = blist[slot];
        int x, y, z;
        node_xyz(L, n, x, y, z);
        // missing set: directions whose pull source is solid at t+1;
        // neighbourhood node k = lane: x_b + c_k
        int nk, src;
        const uint32_t mask = node_links(L, flags, n, x, y, z, lane, off, sok, nk, src);
        const bool miss = act && ((mask >> i) & 1u);
        // known pulled populations (face rules as in the bulk kernel)
        R Fi = R(0);
        if (act && !miss && src >= 0) Fi = Codec<S>::load(fa + (size_t)i * N + src);
        __syncwarp();
        const uint32_t need = (1u << 13) | (1u << 22) | (1u << 4) | (1u << 16) | (1u << 10) |
                              (1u << 14) | (1u << 12) | mask;
        stage<S, R>(L, fa, lane, nk, need, sf, su, sok);
        if (act && !miss && src < 0) Fi = src == -2 ? sf[13][26 - i] : (R)L.g_face[i];
        // target density and velocity over the missing set
        const R fbb = act ? sf[13][26 - (act ? i : 0)] : R(0);  // shifted f'_{opp i}(x_b, t)
        double q = 0;
        R uw[3] = {0, 0, 0};
        float ul[3] = {0, 0, 0};
        if (G.kind == LBM_BODY_MESH) {
            MeshHit hit{-1, 0.0, 0.0};
            double ud[3] = {0, 0, 0};
            mesh_links_warp<R>(G, b, x, y, z, mask, lane, q, ud, hit, s_link[w]);
            for (int a = 0; a < 3; ++a) {
                uw[a] = (R)ud[a];
                ul[a] = (float)(ud[a] - (double)uw[a]);
            }
        } else if (miss) {
            for (int a = 0; a < 3; ++a) {
                uw[a] = s_wall.U[a];
                ul[a] = s_wall.lo[a];
            }
            link_data<R>(L, G, b, s_wall.air, x, y, z, i, q, uw, ul);
        }
        const R qq = (R)q;
        // (the airfoil's and the swimmer's links are found in the precision of R)
        float ql = 0.f;
        if (sizeof(R) == 4 && (G.kind == LBM_BODY_SPHERE || G.kind == LBM_BODY_PLANES)) ql = (float)(q - (double)qq);
        const R gstat = miss ? fbb : Fi;
        const R dyn = miss ? R(6) * weight<R>(i) * rho0 * (R(cx) * uw[0] + R(cy) * uw[1] + R(cz) * uw[2]) : R(0);
        R ut[3] = {0, 0, 0};
        if (miss) {
            if (sok[i]) {
                for (int a = 0; a < 3; ++a) ut[a] = (qq * su[i][1 + a] + uw[a]) / (R(1) + qq);
            } else {
                for (int a = 0; a < 3; ++a) ut[a] = uw[a];
            }
        }
        const R nmiss = R(__popc(mask));
        R t[6] = {act ? gstat : R(0), dyn, ut[0], ut[1], ut[2], R(0)};
        wsum6(t, lane);
        const R rho_t = rho0 + t[0] + t[1];
        const R u_t[3] = {t[2] / nmiss, t[3] / nmiss, t[4] / nmiss};
        R du[3][3];
        const R uc[3] = {su[13][1], su[13][2], su[13][3]};
        fd_gradient<R>(su, sok, uc, du);
        R Qt[6];
        pressure_excess<R>(rho_t, u_t, du, (R)L.beta, Qt);
        R gi = Fi;
        if (miss) gi = grad_shifted<R>(i, rho_t, rho0, u_t, Qt);

        // momentum exchange on missing links: the fluid hands the body
        // (c_opp - u_w) f'_opp(x_b, t) and gets back (c_i - u_w) F_i(x_b, t+1),
        // together -c_i (f_out + f_in) + u_w (f_in - f_out); the node's sums go
        // into its band slot, which the force kernel turns into force and torque
        // a slab's links count where it owns the fluid node
        const bool own = z >= G.own_lo && z < G.own_hi;
        double *fslot = bforce + (size_t)bpos[slot] * FORCE_SLOT;
        if (__any_sync(FULL, miss && force_overflows<R>(fbb, gi, uw))) {
            const double o[3] = {body_offset(L, G, b, 0, x), body_offset(L, G, b, 1, y), body_offset(L, G, b, 2, z)};
            const double ud[3] = {(double)uw[0] + (double)ul[0], (double)uw[1] + (double)ul[1], (double)uw[2] + (double)ul[2]};
            force_plain(fslot, lane, own && miss, i, (double)fbb, (double)gi, q, ud, o, L.rho0);
        } else {
            node_force<R>(fslot, lane, own && miss, cx, cy, cz, i, fbb, gi, qq, ql, uw, ul);
        }

        bool ok;
        const R out = kbc_collide_lanes<R>(gi, i, (R)L.beta, (R)L.inv_beta, rho0, L.gamma_mode, ok);
        if (lane == 0 && !ok) atomicOr(&b->status, ST_UNSTABLE);
        if (act) Codec<S>::store(fb + (size_t)i * N + n, out);
        __syncwarp();
    }
}

template <typename S>
__global__ void __launch_bounds__(BWARPS * 32, LBM_LIST_MIN_BLOCKS) refill_kernel(
    const __grid_constant__ Lattice L, const __grid_constant__ GeomParams G, const DevBody *b, const int *ulist,
    S *fa, const uint8_t *flags)
{
    after_previous();
    using R = typename Codec<S>::R;
    __shared__ __align__(16) R s_f[BWARPS][Q][28];
    __shared__ R s_u[BWARPS][Q][4];
    __shared__ int s_ok[BWARPS][Q];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    R (*sf)[28] = s_f[w];
    R (*su)[4] = s_u[w];
    int *sok = s_ok[w];
    const int count = min(b->n_uncovered, G.cap_uncovered);
    const size_t N = (size_t)L.N;
    const R rho0 = (R)L.rho0;
    for (int slot = blockIdx.x * BWARPS + w; slot < count; slot += gridDim.x * BWARPS) {
        const int n = ulist[slot];
        int x, y, z;
        node_xyz(L, n, x, y, z);
        const bool act = lane < Q;
        int nk = -1;
        if (act && lane != 13) nk = neighbour(L, x, y, z, cx_of(lane), cy_of(lane), cz_of(lane));
        // neighbours that were fluid at t carry valid populations
        if (act) sok[lane] = nk >= 0 && !(flags[nk] & FL_SOLID_PREV);
        __syncwarp();
        uint32_t need = __ballot_sync(FULL, act && sok[lane]);
        stage<S, R, true>(L, fa, lane, nk, need, sf, su, sok);
        const R cnt = R(__popc(need));
        const R rsum = wsum((act && sok[lane]) ? su[lane][0] : R(0));
        const R rho = cnt > R(0) ? rsum / cnt : rho0;
        R u[3] = {(R)b->U[0], (R)b->U[1], (R)b->U[2]};
        if (G.kind == LBM_BODY_PLANES) {
            const double *v = (double)y < 0.5 * (G.y_lo + G.y_hi) ? G.U_lo : G.U_hi;
            u[0] = (R)v[0]; u[1] = (R)v[1]; u[2] = (R)v[2];
        } else if (G.kind == LBM_BODY_MESH) {
            // material velocity of the swimmer at the node's arc position
            double v[3];
            mesh_material_velocity_warp(G, b, (double)x, (double)y, lane, v);
            u[0] = (R)v[0]; u[1] = (R)v[1]; u[2] = (R)v[2];
        }
        R du[3][3], Qt[6];
        fd_gradient<R>(su, sok, u, du);
        pressure_excess<R>(rho, u, du, (R)L.beta, Qt);
        if (act) Codec<S>::store(fa + (size_t)lane * N + n, grad_shifted<R>(lane, rho, rho0, u, Qt));
        __syncwarp();
    }
}

// ----------------------------------------------------------------- launchers

// Grid of the list kernels (grid-stride over the list).  The boundary kernel
// runs beside the bulk kernel, and every resident block of it holds shared
// memory and registers the bulk kernel could use; LBM_LIST_BLOCKS caps the
// grid (build-time knob; two blocks per SM measured best for the sphere and
// the airfoil with the 72-register cap, FP16 sphere step 0.178 -> 0.167 ms
// against one block per SM).
#ifndef LBM_LIST_BLOCKS
#define LBM_LIST_BLOCKS 304
#endif
// The links of the swimmer (a triangle search) and of the airfoil (a root on
// the outline) make their boundary kernel the long part of the body's launch
// chain: LBM_LINK_LIST_BLOCKS gives it more blocks (608 took the 256x128x128
// swimmer's step from 0.359 to 0.256 ms and the two-level airfoil's coarse
// step from 1.13 to 1.05 ms; 1064 measured 1.07).
#ifndef LBM_LINK_LIST_BLOCKS
#define LBM_LINK_LIST_BLOCKS 608
#endif
static int list_blocks(int cap, int max_blocks = LBM_LIST_BLOCKS)
{
    int nb = (cap + BWARPS - 1) / BWARPS;
    return nb < 1 ? 1 : (nb > max_blocks ? max_blocks : nb);
}

cudaError_t launch_boundary(int storage, const Lattice &L, const GeomParams &G, Scratch &S, int cur,
                            const void *fa, void *fb, const uint8_t *flags, cudaStream_t s)
{
    return dispatch_storage(storage, [&](auto tag) {
        using T = std::remove_pointer_t<decltype(tag)>;
        const int nb = list_blocks(G.cap_boundary, G.kind == LBM_BODY_MESH || G.kind == LBM_BODY_AIRFOIL ? LBM_LINK_LIST_BLOCKS : LBM_LIST_BLOCKS);
        return launch_after(L.short_bulk, boundary_kernel<T>, nb, BWARPS * 32, s, L, G, S.body + cur, S.blist, S.bpos, S.bforce, (const T *)fa,
                            (T *)fb, flags);
    });
}

cudaError_t launch_refill(int storage, const Lattice &L, const GeomParams &G, Scratch &S, int cur, void *fa,
                          const uint8_t *flags, cudaStream_t s)
{
    return dispatch_storage(storage, [&](auto tag) {
        using T = std::remove_pointer_t<decltype(tag)>;
        return launch_after(L.short_bulk, refill_kernel<T>, list_blocks(G.cap_uncovered), BWARPS * 32, s, L, G, S.body + cur, S.ulist, (T *)fa,
                            flags);
    });
}

}  // namespace lbm
