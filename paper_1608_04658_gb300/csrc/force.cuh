// Momentum exchange of a boundary node's links (arXiv 1608.04658, Sec. 4.1):
// the sums that the boundary kernel leaves per node and what the force kernel
// reads from them.
#pragma once

#include <cstddef>

#include "lanes.cuh"
#include "pair32.cuh"

namespace lbm {

// A boundary node's sums over its links into its slot (see ForceSlot).  FP32
// and 16-bit storage: sums of -c (f_out + f_in) + u_w (f_in - f_out) without
// W rho0, and of the torque's -q (f_in - f_out) (c x u_w), as pairs hi + lo of
// FP32 numbers (q + ql, uw + ul what a double gives), error-free but for 2^-48
// of values a hundredth of f; W rho0 as the integer sum of 216 W c.  FP64
// arithmetic here
// runs with a fifth of the lanes at work (the missing links of one node) on a
// pipe of two lanes a clock and SM: it took the larger part of this kernel's
// time (airfoil 225 us with it).  The force kernel does it for 32 nodes a warp.
template <typename R>
__device__ __forceinline__ void node_force(double *slot, int lane, bool link, int cx, int cy, int cz,
                                           int i, R fbb, R gi, R q, float ql, const R uw[3],
                                           const float ul[3]);
template <>
__device__ __forceinline__ void node_force<double>(double *slot, int lane, bool link, int cx, int cy,
                                                   int cz, int i, double fbb, double gi, double q, float,
                                                   const double uw[3], const float *)
{
    // force without W rho0, and -sum q (f_in - f_out) (c x u_w)
    double v[6] = {0, 0, 0, 0, 0, 0};
    if (link) {
        const double sum = fbb + gi, dif = gi - fbb, h = -q * dif;
        const int c[3] = {cx, cy, cz};
        for (int a = 0; a < 3; ++a) {
            v[a] = fma(uw[a], dif, c[a] == 0 ? 0.0 : (c[a] > 0 ? -sum : sum));
            const int b1 = (a + 1) % 3, b2 = (a + 2) % 3;
            v[3 + a] = h * (c[b1] * uw[b2] - c[b2] * uw[b1]);
        }
    }
    const double s = wsum_scatter6(v, lane);
#pragma unroll
    for (int k = 0; k < 6; ++k)
        if (lane == wsum_owner6(k)) reinterpret_cast<ForceSlot<double> *>(slot)->v[k] = s;
    const int w = link ? weight216(i) : 0;
    const int k0 = __reduce_add_sync(FULL, w * cx), k1 = __reduce_add_sync(FULL, w * cy),
              k2 = __reduce_add_sync(FULL, w * cz);
    if (lane == 0) reinterpret_cast<ForceSlot<double> *>(slot)->k = pack_k(k0, k1, k2);
}
template <>
__device__ __forceinline__ void node_force<float>(double *slot, int lane, bool link, int cx, int cy,
                                                  int cz, int i, float fbb, float gi, float q, float ql,
                                                  const float uw[3], const float ul[3])
{
    Pair32 F[3] = {}, H[3] = {};
    if (link) {
        const Pair32 sum = two_sum(fbb, gi), dif = two_sum(gi, -fbb);
        const int c[3] = {cx, cy, cz};
        for (int a = 0; a < 3; ++a) {
            const Pair32 p = Pair32{uw[a], ul[a]} * dif;
            F[a] = c[a] == 0 ? p : (c[a] > 0 ? p - sum : p + sum);
        }
        const Pair32 h = Pair32{-q, -ql} * dif;
        for (int a = 0; a < 3; ++a) {
            const int b1 = (a + 1) % 3, b2 = (a + 2) % 3;
            const float s1 = (float)c[b1], s2 = (float)-c[b2];
            H[a] = h * (Pair32{s1 * uw[b2], s1 * ul[b2]} + Pair32{s2 * uw[b1], s2 * ul[b1]});
        }
    }
    // sums as in wsum_scatter6: component 2 to the upper half of the warp, 1 to
    // the upper quarter of the lower half
    const auto exchange = [&](Pair32 a, Pair32 b, int o) {
        const bool up = lane & o;
        const Pair32 keep = up ? b : a, send = up ? a : b;
        return keep + Pair32{__shfl_xor_sync(FULL, send.hi, o), __shfl_xor_sync(FULL, send.lo, o)};
    };
    const Pair32 none = {0.f, 0.f};
    Pair32 Fs = exchange(exchange(F[0], F[2], 16), exchange(F[1], none, 16), 8);
    Pair32 Hs = exchange(exchange(H[0], H[2], 16), exchange(H[1], none, 16), 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
        Fs = Fs + Pair32{__shfl_xor_sync(FULL, Fs.hi, o), __shfl_xor_sync(FULL, Fs.lo, o)};
        Hs = Hs + Pair32{__shfl_xor_sync(FULL, Hs.hi, o), __shfl_xor_sync(FULL, Hs.lo, o)};
    }
    const int w = link ? weight216(i) : 0;
    const int k0 = __reduce_add_sync(FULL, w * cx), k1 = __reduce_add_sync(FULL, w * cy),
              k2 = __reduce_add_sync(FULL, w * cz);
    ForceSlot<float> *p = reinterpret_cast<ForceSlot<float> *>(slot);
    if ((lane & 7) == 0 && lane < 24) {
        const int a = lane >> 3;  // lane 0, 8, 16: components 0, 1, 2
        p->hi[a] = Fs.hi;
        p->lo[a] = Fs.lo;
        p->h[a] = Hs.hi;
        p->hl[a] = Hs.lo;
    }
    if (lane == 0) p->k = pack_k(k0, k1, k2);
}

// What a node leaves whose sums overflow, or whose state is no longer finite:
// force and torque themselves (o: the node's offset from the reference point),
// in FP64 from the full populations, link by link, so that an infinite
// population gives the infinities and NaNs of the momentum exchange and not
// those of how it is evaluated.  Out of line, no node of a stable run takes it.
constexpr int SLOT_PLAIN = 1 << 24;
__device__ __noinline__ static void force_plain(double *slot, int lane, bool link, int i, double fbb, double gi, double q,
                                                const double uw[3], const double o[3], double rho0)
{
    double v[6] = {0, 0, 0, 0, 0, 0};
    if (link) {
        const double W = weight<double>(i) * rho0, fout = fbb + W, fin = gi + W;
        const double c[3] = {(double)cx_of(i), (double)cy_of(i), (double)cz_of(i)};
        double r[3];
        for (int a = 0; a < 3; ++a) {
            v[a] = (-c[a] - uw[a]) * fout - (c[a] - uw[a]) * fin;
            r[a] = o[a] - q * c[a];
        }
        v[3] = r[1] * v[2] - r[2] * v[1];
        v[4] = r[2] * v[0] - r[0] * v[2];
        v[5] = r[0] * v[1] - r[1] * v[0];
    }
    const double s = wsum_scatter6(v, lane);
    ForceSlot<double> *p = reinterpret_cast<ForceSlot<double> *>(slot);
#pragma unroll
    for (int k = 0; k < 6; ++k)
        if (lane == wsum_owner6(k)) p->v[k] = s;
    if (lane == 0) p->k = SLOT_PLAIN;
}

// whether a link's values are outside the range in which the sums of the other
// form can neither overflow nor lose their low parts
template <typename R>
__device__ __forceinline__ bool force_overflows(R fbb, R gi, const R uw[3])
{
    const R big = sizeof(R) == 4 ? R(1e30) : R(1e290);
    return !(fabs(fbb) + fabs(gi) < big && fabs(uw[0]) + fabs(uw[1]) + fabs(uw[2]) < R(1e6));
}

// The node's force F and torque M about the reference point from its slot; o:
// its offset from there (see ForceSlot).
template <typename R>
__device__ __forceinline__ void slot_force(const double *slot, double rho0, const double o[3], double F[3], double M[3])
{
    static_assert(offsetof(ForceSlot<float>, k) == offsetof(ForceSlot<double>, k), "a plain slot is told by its k");
    const ForceSlot<R> *p = reinterpret_cast<const ForceSlot<R> *>(slot);
    const int k = p->k;
    if (k & SLOT_PLAIN) {
        const ForceSlot<double> *w = reinterpret_cast<const ForceSlot<double> *>(slot);
        for (int a = 0; a < 3; ++a) {
            F[a] = w->v[a];
            M[a] = w->v[3 + a];
        }
        return;
    }
    double h[3];
    for (int a = 0; a < 3; ++a) {
        if constexpr (sizeof(R) == 8) {
            F[a] = p->v[a];
            h[a] = p->v[3 + a];
        } else {
            F[a] = (double)p->hi[a] + (double)p->lo[a];
            h[a] = (double)p->h[a] + (double)p->hl[a];
        }
        F[a] -= (rho0 / 108.0) * unpack_k(k, a);
    }
    for (int a = 0; a < 3; ++a) {
        const int b1 = (a + 1) % 3, b2 = (a + 2) % 3;
        M[a] = o[b1] * F[b2] - o[b2] * F[b1] + h[a];
    }
}

}  // namespace lbm
