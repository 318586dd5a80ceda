// Mass, momentum and kinetic energy of one node for the global sums
// (lbm_totals, lbm_totals_noalloc).
//
// The sums are FP64 sums, but the GPU adds two FP64 lanes a clock and SM
// against 128 FP32 lanes: 27 conversions, weights and moments in double cost
// about 140 FP64 operations a node, 8.3 ms on a 256^3 FP32 box whose 1.8 GB
// cross the memory bus in 0.27 ms.  For FP32 and 16-bit storage the sums of a
// node are therefore formed as unevaluated pairs hi + lo of FP32 numbers by
// error-free transformations (the two-sum of Knuth, The Art of Computer
// Programming 2, 4.2.2, and the two-product with a fused multiply-add): each
// addition's rounding error is carried in lo, so a pair holds some 48 bits of
// the sum of the *shifted* populations.  These are a few hundredths of W rho0,
// so the pair is as exact as the FP64 sum of the full populations, whose own
// rounding of g + W rho0 it does not make.  The rest density is added once per
// thread, the pairs go into FP64 accumulators every few nodes.
#pragma once

#include "kbc.cuh"
#include "pair32.cuh"

namespace lbm {

// sums of the shifted populations over the directions, weighted by 1, c_x, c_y,
// c_z (x-lines l = 3(cy+1) + (cz+1), then the rows of the 3x3 line sums)
template <typename T, typename G>
__device__ __forceinline__ void node_sums(const G &g, T m[4])
{
    T s[9], jx{};
#pragma unroll
    for (int l = 0; l < 9; ++l) {
        const T p = g(18 + l), q = g(l);
        s[l] = (p + q) + g(9 + l);
        jx = l == 0 ? p - q : jx + (p - q);
    }
    T row[3], jz{};
#pragma unroll
    for (int r = 0; r < 3; ++r) {
        row[r] = (s[3 * r] + s[3 * r + 2]) + s[3 * r + 1];
        const T d = s[3 * r + 2] - s[3 * r];
        jz = r == 0 ? d : jz + d;
    }
    m[0] = (row[0] + row[2]) + row[1];
    m[1] = jx;
    m[2] = row[2] - row[0];
    m[3] = jz;
}

// The node's full sums in FP64 one direction at a time: a state outside the
// range of the forms below (unstable: huge, infinite or not a number), whose
// every sum shows it.
template <typename R>
__device__ __noinline__ void node_totals_plain(const R (&g)[Q], double rho0, double out[5])
{
    double r = 0, j[3] = {0, 0, 0};
    for (int i = 0; i < Q; ++i) {
        const double v = (double)g[i] + weight<double>(i) * rho0;
        r += v;
        j[0] += cx_of(i) * v;
        j[1] += cy_of(i) * v;
        j[2] += cz_of(i) * v;
    }
    out[0] = r;
    out[1] = j[0];
    out[2] = j[1];
    out[3] = j[2];
    out[4] = 0.5 * (j[0] * j[0] + j[1] * j[1] + j[2] * j[2]) / r;
}

// FP64 sums of a thread's nodes: mass excess over rho0, momentum, kinetic
// energy; add() takes a node's 27 stored populations (loaded by the caller, so
// that the loads are in flight together).
template <typename R>
struct NodeTotals {
    double acc[5] = {0, 0, 0, 0, 0};
    long long count = 0;
    __device__ __forceinline__ void add(const R (&g)[Q], double rho0)
    {
        double m[4];
        node_sums<double>([&](int i) { return (double)g[i]; }, m);
        if (!(fabs(m[0]) < 1e100)) {
            double t[5];
            node_totals_plain<double>(g, rho0, t);
            for (int k = 0; k < 5; ++k) acc[k] += t[k];
            return;
        }
        ++count;
        const double rho = rho0 + m[0];
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[k] += m[k];
        acc[4] += 0.5 * (m[1] * m[1] + m[2] * m[2] + m[3] * m[3]) / rho;
    }
    __device__ __forceinline__ void finish(double rho0) { acc[0] += (double)count * rho0; }
};

template <>
struct NodeTotals<float> {
    // FP32 pairs are emptied into the FP64 sums every FLUSH nodes: their lo
    // parts then lose at most FLUSH roundings of 2^-48 of the partial sum
    static constexpr int FLUSH = 16;
    double acc[5] = {0, 0, 0, 0, 0};
    Pair32 part[5] = {};
    // what the squares of the pairs leave out, lo^2: of one sign, so that it does
    // not average out over the nodes (3e-15 of the kinetic energy in FP32)
    float squares = 0.f;
    int held = 0;
    long long count = 0;
    __device__ __forceinline__ void flush()
    {
#pragma unroll
        for (int k = 0; k < 5; ++k) {
            acc[k] += value(part[k]);
            part[k] = Pair32{0.f, 0.f};
        }
        acc[4] += (double)squares;
        squares = 0.f;
        held = 0;
    }
    __device__ __forceinline__ void add(const float (&g)[Q], double rho0)
    {
        Pair32 m[4];
        node_sums<Pair32>([&](int i) { return Pair32{g[i], 0.f}; }, m);
        const float r0 = (float)rho0;
        const Pair32 rho = Pair32{r0, (float)(rho0 - (double)r0)} + m[0];
        const Pair32 q = (square(m[1]) + square(m[2])) + square(m[3]);
        // quotient q / rho: the FP32 one and its remainder's, the second with what
        // the reciprocal leaves of it (inv (1 + e1)): the square of the
        // reciprocal's error has one sign, 1e-15 of the sum
        const float inv = rcp_fast(rho.hi), k1 = __fmul_rn(q.hi, inv);
        const float rem = __fadd_rn(__fmaf_rn(-k1, rho.hi, q.hi), __fmaf_rn(-k1, rho.lo, q.lo));
        const float e1 = __fmaf_rn(-rho.lo, inv, __fmaf_rn(-rho.hi, inv, 1.f)), k2 = __fmul_rn(rem, inv);
        const Pair32 ke = two_sum(k1, __fmaf_rn(k2, e1, k2));
        // the range in which the pairs' products neither overflow nor lose
        // their remainders to underflow
        if (rho.hi > 1e-6f && rho.hi < 1e6f && fabsf(m[0].hi) < 1e6f && q.hi < 1e12f &&
            (q.hi > 1e-24f || q.hi == 0.f)) {
            ++count;
#pragma unroll
            for (int k = 0; k < 4; ++k) part[k] = part[k] + m[k];
            part[4] = part[4] + ke;
            squares = __fmaf_rn(__fmaf_rn(m[1].lo, m[1].lo, __fmaf_rn(m[2].lo, m[2].lo, __fmul_rn(m[3].lo, m[3].lo))), inv, squares);
            if (++held == FLUSH) flush();
        } else {
            double t[5];
            node_totals_plain<float>(g, rho0, t);
#pragma unroll
            for (int k = 0; k < 4; ++k) acc[k] += t[k];
            acc[4] += 2.0 * t[4];
        }
    }
    __device__ __forceinline__ void finish(double rho0)
    {
        flush();
        acc[0] += (double)count * rho0;
        acc[4] *= 0.5;
    }
};

}  // namespace lbm
