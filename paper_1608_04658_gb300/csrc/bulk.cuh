// Bulk fused pull-stream + KBC collide (arXiv 1608.04658, Sec. 2, Eq. kineticEq
// with Eq. kbc_relax).
//
// Two nodes per thread (bulk_pair_kernel) or one (bulk_kernel), threads along x
// (the fastest axis of every population plane) so each of the 27 plane loads and
// stores of a warp is one contiguous run; the +-1 x-shift of a pull touches one
// extra 32-byte sector per warp, which the neighbouring warp reads anyway, so
// DRAM traffic stays at one read and one write per population.  Nodes marked
// SOLID or BOUNDARY are left to the boundary kernel.  With a body, one launch
// takes the nodes outside the body's sweep box (no flag read) while the body's
// geometry runs beside it, and a second the nodes of the box once their marks
// are known.
#pragma once

#include <algorithm>
#include <type_traits>

#include "pull.cuh"

namespace lbm {

// Forms of the collision: V kbc_collide_v, M kbc_collide_m, MX the same with the
// exact stabilizer, X kbc_collide with it (FP64).
enum CollideForm { FORM_V = 0, FORM_M = 1, FORM_MX = 2, FORM_X = 3 };

// Minimum resident blocks per SM requested from the register allocator for
// the one-node kernel: 7 blocks of 128 threads cap it at 72 registers (no
// spill) and give 28 warps per SM, which measured faster on GB300 than 80
// registers with 6 blocks or 64 with 8.  The exact stabilizer's terms and FP64
// storage spill at 72 registers; they get fewer blocks.
template <typename S, int FORM>
struct BulkBlocks {
    static constexpr int value = FORM >= FORM_MX || std::is_same<S, double>::value ? 4 : 7;
};

// Resident blocks (warps) per SM asked of the register allocator for the
// two-node kernel: 16, which fit in 128 registers without spilling.  Measured on
// GB300 (768x256x256 periodic box): FP32 0.839 of the copy bandwidth at 20
// against 1.03 at 16, FP16 0.66 at 18 against 0.74.  The exact stabilizer takes
// 12 (168 registers).
template <int FORM>
struct PairBlocks {
    static constexpr int value = FORM == FORM_MX ? 12 : 16;
};
// One warp a block: the last block of a row that is no multiple of 128 nodes
// long then holds no registers for warps that have nothing to do (160x97x83
// FP16: 53.4 us a step with blocks of 64 threads, 161x97x83 BF16 57 us, 47 with
// 32); rows of whole blocks take the same time.
constexpr int PAIR_THREADS = 32;

// The update of one node by kbc_collide with the exact stabilizer's safeguarded
// iteration, out of line and after everything else of its thread: the few nodes
// that exact_stabilizer hands back.
template <typename S>
__device__ __noinline__ void exact_node_update(const Lattice &L, const S *fa, S *fb,
                                               int *status, int x, int y, int z)
{
    using R = typename Codec<S>::R;
    const int n = x + L.nx * (y + L.ny * z);
    R g[Q];
    gather_global<S>(L, fa, x, y, z, n, g);
    if (!kbc_collide<R, true>(g, (R)L.beta, (R)L.inv_beta, (R)L.rho0, L.gamma_mode)) atomicOr(status, ST_UNSTABLE);
#pragma unroll
    for (int i = 0; i < Q; ++i) Codec<S>::store(fb + n + L.plane[i], g[i]);
}

template <typename S, int FORM>
__global__ void __launch_bounds__(128, (BulkBlocks<S, FORM>::value)) bulk_kernel(const __grid_constant__ Lattice L, const S *fa,
                                                   S *fb,
                                                   const uint8_t *flags,
                                                   int *status,
                                                   const int *sweep, int mode, int capx,
                                                   int capy, int z0)
{
    after_previous();
    using R = typename Codec<S>::R;
    int x, y, z;
    if (mode == BULK_BAND) {
        // one thread per position of the capacity box, x fastest
        const int k = blockIdx.x * blockDim.x + threadIdx.x;
        const int lx = k % capx, ly = (k / capx) % capy, lz = k / (capx * capy);
        if (lx >= sweep[3] || ly >= sweep[4] || lz >= sweep[5]) return;
        x = sweep_coord(sweep[0] + lx, L.nx);
        y = sweep_coord(sweep[1] + ly, L.ny);
        z = sweep_coord(sweep[2] + lz, L.nz);
    } else {
        x = blockIdx.x * blockDim.x + threadIdx.x;
        y = blockIdx.y;
        z = z0 + (int)blockIdx.z;
        if (x >= L.nx) return;
        // y and z are uniform over the block, so only rows crossing the box
        // test x
        if (mode == BULK_OUTSIDE && in_sweep(sweep, 1, y, L.ny, L.face[2] == LBM_FACE_PERIODIC) &&
            in_sweep(sweep, 2, z, L.nz, L.face[4] == LBM_FACE_PERIODIC) &&
            in_sweep(sweep, 0, x, L.nx, L.face[0] == LBM_FACE_PERIODIC))
            return;
    }
    const int nx = L.nx, ny = L.ny;
    const int n = x + nx * (y + ny * z);
    if (flags != nullptr && (flags[n] & (FL_SOLID | FL_BOUNDARY))) return;

    // all 27 pulls are issued unconditionally (wall/equilibrium sources read
    // the node itself and are replaced afterwards)
    R g[Q];
    gather_global<S>(L, fa, x, y, z, n, g);
    bool ok;
    if constexpr (FORM == FORM_X) ok = kbc_collide<R, true>(g, (R)L.beta, (R)L.inv_beta, (R)L.rho0, L.gamma_mode);
    else if constexpr (FORM == FORM_V) ok = kbc_collide_v<F1>(g, L.beta_f, L.inv_beta_f, L.rho0_f, L.gamma_mode) & 1;
    else if constexpr (std::is_same<R, double>::value)
        ok = kbc_collide_m<D1, false>(g, L.beta, L.inv_beta, L.rho0, L.gamma_mode, (double)L.zero_f) & 1;
    else {
        const int r = kbc_collide_m<F1, FORM == FORM_MX>(g, L.beta_f, L.inv_beta_f, L.rho0_f, L.gamma_mode, L.zero_f);
        if (FORM == FORM_MX && (r & 2)) {
            exact_node_update<S>(L, fa, fb, status, x, y, z);
            return;
        }
        ok = r & 1;
    }
    if (!ok) atomicOr(status, ST_UNSTABLE);
    S *q = fb + n;
#pragma unroll
    for (int i = 0; i < Q; ++i) Codec<S>::store(q + L.plane[i], g[i]);
}

// Two nodes per thread, (x0, x0 + 1) with x0 even: each pull is an aligned word
// of the pair (two for c_x = +-1), the collision runs on both nodes in packed
// FP32x2 arithmetic, each store writes the pair's word.  ODD: rows of odd
// length, whose pairs are not aligned: single elements in place of the words;
// the last thread takes the pair (nx - 2, nx - 1) and stores its second node.  Node
// selection as in bulk_kernel (ALL or OUTSIDE; the sweep box takes the one-node
// kernel), per node of the pair.  XPER: the x axis is periodic; YZPER: the y and
// z axes are.
template <typename S, int FORM, bool XPER, bool YZPER, bool ODD>
__device__ __forceinline__ void pair_update(const Lattice &L, const S *fa, S *fb,
                                            const uint8_t *flags, int *status,
                                            const int *sweep, int mode, int x0, int y, int z)
{
    int act = 3;  // bit 0: node x0 is updated here, bit 1: node x0 + 1
    if (ODD && x0 + 1 == L.nx) {
        --x0;
        act = 2;
    }
    if (mode == BULK_OUTSIDE && in_sweep(sweep, 1, y, L.ny, L.face[2] == LBM_FACE_PERIODIC) &&
        in_sweep(sweep, 2, z, L.nz, L.face[4] == LBM_FACE_PERIODIC)) {
        const bool per = L.face[0] == LBM_FACE_PERIODIC;
        act &= (in_sweep(sweep, 0, x0, L.nx, per) ? 0 : 1) | (in_sweep(sweep, 0, x0 + 1, L.nx, per) ? 0 : 2);
        if (!act) return;
    }
    const int n0 = x0 + L.nx * (y + L.ny * z);
    if (flags != nullptr) {
        // (the caller's marks may begin at any address)
        const bool bytes = ODD || (reinterpret_cast<size_t>(flags) & 1);
        const unsigned fw = bytes ? flags[n0] | flags[n0 + 1] << 8 : *reinterpret_cast<const unsigned short *>(flags + n0);
        if (fw & (FL_SOLID | FL_BOUNDARY)) act &= ~1;
        if ((fw >> 8) & (FL_SOLID | FL_BOUNDARY)) act &= ~2;
        if (!act) return;
    }
    float2 g[Q];
    gather_pair<S, XPER, YZPER, ODD>(L, fa, x0, y, z, n0, g);
    int ok;
    if constexpr (FORM == FORM_V) ok = kbc_collide_v<F2>(g, L.beta_f, L.inv_beta_f, L.rho0_f, L.gamma_mode);
    else ok = kbc_collide_m<F2, FORM == FORM_MX>(g, L.beta_f, L.inv_beta_f, L.rho0_f, L.gamma_mode, L.zero_f);
    const int again = FORM == FORM_MX ? act & (ok >> 2) : 0;
    act &= ~again;
    if (act & ~ok) atomicOr(status, ST_UNSTABLE);
    S *q = fb + n0;
    if (!ODD && act == 3) {
#pragma unroll
        for (int i = 0; i < Q; ++i) Pair<S>::store(q + L.plane[i], g[i]);
        return;
    }
    if (act & 1) {
#pragma unroll
        for (int i = 0; i < Q; ++i) Codec<S>::store(q + L.plane[i], g[i].x);
    }
    if (act & 2) {
#pragma unroll
        for (int i = 0; i < Q; ++i) Codec<S>::store(q + 1 + L.plane[i], g[i].y);
    }
    if constexpr (FORM == FORM_MX) {
        if (again & 1) exact_node_update<S>(L, fa, fb, status, x0, y, z);
        if (again & 2) exact_node_update<S>(L, fa, fb, status, x0 + 1, y, z);
    }
}

// One block per 64 nodes of a row.  A row that touches no y or z face
// other than a periodic one pulls only from inside the box along y and z, so
// it takes the y/z-periodic form of the gather whatever the box's y and z
// faces are (the choice is uniform over the block).
template <typename S, int FORM, bool XPER, bool YZPER, bool ODD>
__global__ void __launch_bounds__(PAIR_THREADS, PairBlocks<FORM>::value) bulk_pair_kernel(
    const __grid_constant__ Lattice L, const S *fa, S *fb,
    const uint8_t *flags, int *status, const int *sweep, int mode, int z0)
{
    after_previous();
    const int x0 = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
    if (x0 >= L.nx) return;
    const int y = blockIdx.y, z = z0 + (int)blockIdx.z;
    if constexpr (!YZPER) {
        const bool face_row = (L.face[2] != LBM_FACE_PERIODIC && (y == 0 || y == L.ny - 1)) ||
                              (L.face[4] != LBM_FACE_PERIODIC && (z == 0 || z == L.nz - 1));
        if (!face_row) {
            pair_update<S, FORM, XPER, true, ODD>(L, fa, fb, flags, status, sweep, mode, x0, y, z);
            return;
        }
    }
    pair_update<S, FORM, XPER, YZPER, ODD>(L, fa, fb, flags, status, sweep, mode, x0, y, z);
}

// ----------------------------------------------------------------- launchers
template <typename S, int FORM>
cudaError_t launch_bulk_form(const Lattice &L, const S *fa, S *fb, const uint8_t *flags, int *status, cudaStream_t s,
                             int mode, const int *sweep, const int *cap, int z_lo, int z_n)
{
    // early where no body's chain runs beside it or that chain is the step: the
    // sweep box's blocks, waiting in their places at the end of a long chain, cost
    // the bulk launch beside it half a percent
    const bool early = (mode == BULK_ALL && !flags) || L.short_bulk;
    // FP32 and 16-bit storage take the two-node kernel for everything but the
    // sweep box (every node gets the same bits either way).  FP32 rows of odd
    // length stay with the one-node kernel, whose whole lines suit a launch bound
    // by memory (147x21x180: 27 us a step, 30 as unaligned pairs; in 16 bits, bound
    // by arithmetic, 161x97x83 57 against 44), but for the exact stabilizer.
    if constexpr (!std::is_same<S, double>::value) {
        constexpr bool odd_pairs = sizeof(S) == 2 || FORM == FORM_MX;
        const bool odd = L.nx & 1;
        if (mode != BULK_BAND && L.nx > 1 && (odd_pairs || !odd)) {
            const bool xper = L.face[0] == LBM_FACE_PERIODIC,
                       yzper = L.face[2] == LBM_FACE_PERIODIC && L.face[4] == LBM_FACE_PERIODIC;
            auto kernel = bulk_pair_kernel<S, FORM, false, false, false>;
            if constexpr (odd_pairs)
                if (odd) kernel = bulk_pair_kernel<S, FORM, false, false, true>;
            // (the faces known at compile time where it pays: not beside the
            // exact stabilizer's arithmetic, nor beside single-element loads)
            if constexpr (FORM != FORM_MX) {
                if (!odd && xper && yzper) kernel = bulk_pair_kernel<S, FORM, true, true, false>;
                else if (!odd && xper) kernel = bulk_pair_kernel<S, FORM, true, false, false>;
                else if (!odd && yzper) kernel = bulk_pair_kernel<S, FORM, false, true, false>;
            }
            const dim3 g2(((L.nx + 1) / 2 + PAIR_THREADS - 1) / PAIR_THREADS, L.ny, z_n);
            return launch_after(early, kernel, g2, PAIR_THREADS, s, L, fa, fb, flags, status, sweep, mode, z_lo);
        }
    }
    int bx = L.nx >= 128 ? 128 : ((L.nx + 31) / 32) * 32;
    dim3 grid((L.nx + bx - 1) / bx, L.ny, z_n);
    int capx = 1, capy = 1;
    if (mode == BULK_BAND) {
        bx = 128;
        capx = cap[0];
        capy = cap[1];
        const long long vol = (long long)cap[0] * cap[1] * cap[2];
        grid = dim3((unsigned)((vol + bx - 1) / bx), 1, 1);
    }
    return launch_after(early, bulk_kernel<S, FORM>, grid, bx, s, L, fa, fb, flags, status, sweep, mode, capx, capy, z_lo);
}

// In FP32 and 16 bits a launch over every node without marks takes
// kbc_collide_m, and so does every launch on a box of this many nodes or more
// (768x256x256 FP16 1219 -> 1062 us, 1024x512x64 with faces 874 -> 767).  A
// launch beside a body's chain or with marks on a smaller box (a refinement's
// levels too, with or without a body) keeps kbc_collide_v.  Below the line it is
// one of bits and not of time: a step in us by the one and the other form is, in
// FP32 and FP16, 156 and 154, 132 and 121 (128x128x256 sphere), 168 and 173, 142
// and 132 (512x256x32 airfoil), 208 and 203, 184 and 174 (256x128x128 swimmer),
// 379 and 366, 340 and 331 (256x128x32 airfoil on two levels); the other order
// of operations moves the rounding of a store, which shows in sums of both
// signs, such as the mean thrust of an adjoint's objective.  A slab goes by the
// whole box, whose bits its own layers have to give.
constexpr long long MOMENT_FORM_NODES = 1LL << 23;

template <typename S>
cudaError_t launch_bulk_t(const Lattice &L, const S *fa, S *fb, const uint8_t *flags, int *status, cudaStream_t s,
                          int mode, const int *sweep, const int *cap, int z_lo, int z_n)
{
    const auto form = [&](auto f) {
        return launch_bulk_form<S, decltype(f)::value>(L, fa, fb, flags, status, s, mode, sweep, cap, z_lo, z_n);
    };
    constexpr bool dbl = std::is_same<S, double>::value;
    if (L.gamma_mode == LBM_GAMMA_EXACT) return form(std::integral_constant<int, dbl ? FORM_X : FORM_MX>{});
    if constexpr (!dbl)
        if (L.n_box < MOMENT_FORM_NODES && (mode != BULK_ALL || flags)) return form(std::integral_constant<int, FORM_V>{});
    return form(std::integral_constant<int, FORM_M>{});
}

}  // namespace lbm
