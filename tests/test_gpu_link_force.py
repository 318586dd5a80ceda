"""The momentum exchange of a boundary node's links (csrc/force.cuh), compiled by itself: what the force kernel reads from a
node's slot against the same sums in extended precision."""
import ctypes as C
import subprocess

import numpy as np
import pytest

from paper_1608_04658_gb300 import builder

pytestmark = pytest.mark.gpu

SRC = r"""
#include "force.cuh"
using namespace lbm;
// one warp a node, lane i its link i (27 lanes of 32); out: F and M of the node, at offset o from the reference point
template <typename R>
__global__ void nodes(int n, const unsigned *mask, const double *fbb, const double *gi, const double *q,
                      const double *uw, const double *off, double rho0, double *slots, double *out)
{
    const int node = blockIdx.x, i = threadIdx.x;
    if (node >= n) return;
    const bool act = i < Q, link = act && (mask[node] >> i & 1u);
    const int cx = act ? cx_of(i) : 0, cy = act ? cy_of(i) : 0, cz = act ? cz_of(i) : 0, k = node * 32 + i;
    R u[3];
    float ul[3];
    for (int a = 0; a < 3; ++a) {
        u[a] = (R)uw[3 * k + a];
        ul[a] = (float)(uw[3 * k + a] - (double)u[a]);
    }
    const R qq = (R)q[k];
    const double o[3] = {off[3 * node], off[3 * node + 1], off[3 * node + 2]};
    double *slot = slots + node * FORCE_SLOT;
    if (__any_sync(FULL, link && force_overflows<R>((R)fbb[k], (R)gi[k], u)))
        force_plain(slot, i, link, i, fbb[k], gi[k], q[k], uw + 3 * k, o, rho0);
    else
        node_force<R>(slot, i, link, cx, cy, cz, i, (R)fbb[k], (R)gi[k], qq, (float)(q[k] - (double)qq), u, ul);
    __syncwarp();
    if (i == 0) slot_force<R>(slots + node * FORCE_SLOT, rho0, o, out + 6 * node, out + 6 * node + 3);
}
extern "C" __attribute__((visibility("default"))) int run(int wide, int n, const unsigned *mask, const double *fbb,
    const double *gi, const double *q, const double *uw, const double *off, double rho0, double *out)
{
    unsigned *dm; double *d[7];
    const size_t m[7] = {32u * n, 32u * n, 32u * n, 96u * n, 3u * n, (size_t)FORCE_SLOT * n, 6u * n};
    if (cudaMalloc(&dm, 4 * n)) return 1;
    for (int k = 0; k < 7; ++k) if (cudaMalloc(&d[k], 8 * m[k])) return 1;
    const double *h[5] = {fbb, gi, q, uw, off};
    cudaMemcpy(dm, mask, 4 * n, cudaMemcpyHostToDevice);
    for (int k = 0; k < 5; ++k) cudaMemcpy(d[k], h[k], 8 * m[k], cudaMemcpyHostToDevice);
    if (wide) nodes<double><<<n, 32>>>(n, dm, d[0], d[1], d[2], d[3], d[4], rho0, d[5], d[6]);
    else nodes<float><<<n, 32>>>(n, dm, d[0], d[1], d[2], d[3], d[4], rho0, d[5], d[6]);
    const int e = cudaMemcpy(out, d[6], 8 * m[6], cudaMemcpyDeviceToHost);
    cudaFree(dm);
    for (int k = 0; k < 7; ++k) cudaFree(d[k]);
    return e;
}
"""

CX = np.array([(i // 9 - 1, (i // 3) % 3 - 1, i % 3 - 1) for i in range(27)])
W216 = np.array([(64, 16, 4, 1)[int(np.abs(c).sum())] for c in CX])


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("link_force")
    (d / "t.cu").write_text(SRC)
    subprocess.check_call([builder.nvcc(), *builder.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I", builder.CSRC,
                           "-I", builder.INCLUDE, str(d / "t.cu"), "-o", str(d / "t.so")])
    return C.CDLL(str(d / "t.so"))


def _run(lib, wide, mask, fbb, gi, q, uw, rho0, off=None):
    n = len(mask)
    out = np.zeros((n, 6))
    p = [np.ascontiguousarray(a) for a in (mask, fbb, gi, q, uw, np.zeros((n, 3)) if off is None else off)]
    assert lib.run(C.c_int(wide), C.c_int(n), *[a.ctypes.data_as(C.c_void_p) for a in p], C.c_double(rho0), out.ctypes.data_as(C.c_void_p)) == 0
    return out


def _links(n, wide, seed):
    """Nodes with 1 to 13 missing links, populations of a few hundredths of W rho0, fractions in (0, 1], a wall of up to 0.1;
    FP32 nodes have FP32 populations and a wall and fractions in double, as a sphere's are."""
    rng = np.random.default_rng(seed)
    mask = np.zeros(n, dtype=np.uint32)
    for k in range(n):
        for i in rng.choice([i for i in range(27) if i != 13], rng.integers(1, 14), replace=False):
            mask[k] |= np.uint32(1 << int(i))
    r = np.float64 if wide else np.float32
    fbb, gi = (rng.normal(size=(n, 32)) * 0.02 for _ in range(2))
    q, uw = 1.0 - rng.random((n, 32)), rng.uniform(-0.1, 0.1, (n, 32, 3))
    return mask, fbb.astype(r).astype(np.float64), gi.astype(r).astype(np.float64), q, uw


@pytest.mark.parametrize("wide", [1, 0])
@pytest.mark.parametrize("n", [1, 700])
def test_node_at_the_reference_point(lib, wide, n):
    """F = sum of -c (f_out + f_in) + u_w (f_in - f_out) and M = sum of -q (f_in - f_out) (c x u_w).  Pairs of FP32 numbers
    hold 48 bits: some 10 operations of 2^-47 on each term, 2^-43 of the sum of magnitudes; in FP64 2^-49."""
    rho0, L = 1.1, np.longdouble
    mask, fbb, gi, q, uw = _links(n, wide, 3 + wide)
    out = _run(lib, wide, mask, fbb, gi, q, uw, rho0)
    m = ((mask[:, None] >> np.arange(27)) & 1).astype(bool)[..., None]
    c, w = CX.astype(L), (W216.astype(L) / 216 * L(rho0))[None, :, None]
    fo, fi = (a[:, :27, None].astype(L) for a in (fbb, gi))
    u, qq = uw[:, :27].astype(L), q[:, :27, None].astype(L)
    terms = -c * (fo + fi + 2 * w) + u * (fi - fo)
    h = -qq * (fi - fo) * np.cross(np.broadcast_to(c, u.shape), u)
    ref = np.concatenate([np.where(m, terms, 0).sum(1), np.where(m, h, 0).sum(1)], 1)
    mag = np.concatenate([np.where(m, np.abs(c) * (np.abs(fo) + np.abs(fi)) + np.abs(u) * (np.abs(fi) + np.abs(fo)), 0).sum(1),
                          np.where(m, qq * (np.abs(fi) + np.abs(fo)) * 2 * np.abs(u).max(2, keepdims=True) * np.ones(3), 0).sum(1)], 1)
    rest = np.concatenate([np.where(m, 2 * w * np.abs(c), 0).sum(1), np.zeros((n, 3))], 1)  # (FP64 once: rho0 / 108 times a whole number)
    tol = (2.0 ** -49 if wide else 2.0 ** -43) * mag + 2.0 ** -51 * rest
    assert np.all(np.abs(out - ref) <= tol), np.abs((out - ref) / mag).max(0)


@pytest.mark.parametrize("wide", [1, 0])
@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan, 2e38, -3e38])
def test_a_broken_population(lib, wide, value):
    """A node with one population that is not finite, or so large that sums of two overflow FP32: force and torque are those
    of the links' momentum exchange, (-c - u_w) f_out - (c - u_w) f_in and its moment, in double: the same infinities, the
    same NaNs, finite sums to FP64 rounding (13 links, 2^-48 of the largest)."""
    rho0, n = 1.1, 64
    mask, fbb, gi, q, uw = _links(n, wide, 9)
    if not wide:
        uw = uw.astype(np.float32).astype(np.float64)
    rng = np.random.default_rng(11)
    off = rng.uniform(-20.0, 20.0, (n, 3))
    for k in range(n):
        i = rng.choice([i for i in range(27) if mask[k] >> np.uint32(i) & np.uint32(1)])
        (fbb if k % 2 else gi)[k, i] = np.float32(value)
    uw[: n // 4] = 0.0  # (a wall at rest)
    out = _run(lib, wide, mask, fbb, gi, q, uw, rho0, off)
    with np.errstate(all="ignore"):
        for k in range(n):
            F, M, big = np.zeros(3), np.zeros(3), 0.0
            for i in range(27):
                if mask[k] >> np.uint32(i) & np.uint32(1):
                    c, W = CX[i].astype(np.float64), W216[i] / 216 * rho0
                    d = (-c - uw[k, i]) * (fbb[k, i] + W) - (c - uw[k, i]) * (gi[k, i] + W)
                    r = off[k] - q[k, i] * c
                    F, M = F + d, M + np.cross(r, d)
                    big = max(big, 64.0 * np.nanmax(np.where(np.isfinite(d), np.abs(d), 0.0)))
            ref = np.concatenate([F, M])
            assert np.array_equal(np.isnan(out[k]), np.isnan(ref)), (k, out[k], ref)
            ok = ~np.isnan(ref)
            fin = np.isfinite(ref)
            assert np.array_equal(out[k][ok & ~fin], ref[ok & ~fin])
            assert np.all(np.abs(out[k][fin] - ref[fin]) <= 2.0 ** -48 * 13 * big)
