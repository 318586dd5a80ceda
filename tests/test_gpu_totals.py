"""Global sums (lbm_totals, lbm_totals_noalloc) against a plain FP64 sum of the stored populations."""
import ctypes as C

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

CX = np.array([(i // 9 - 1, (i // 3) % 3 - 1, i % 3 - 1) for i in range(27)], dtype=np.float64)


def _reference(lat):
    """Sums over the fluid nodes in extended precision, and the sums of the magnitudes that were added."""
    f = lat.populations().reshape(27, -1).astype(np.longdouble)
    fluid = (lat.flags.cpu().numpy().reshape(-1) & 1) == 0
    f = f[:, fluid]
    r, j = f.sum(0), CX.T.astype(np.longdouble) @ f
    ke = 0.5 * (j ** 2).sum(0) / r
    return (np.array([r.sum(), *j.sum(1), ke.sum()], dtype=np.float64),
            np.array([r.sum(), *[np.abs(f).sum()] * 3, (np.abs(f).sum(0) * np.abs(j).sum(0) / r).sum()], dtype=np.float64))


def _noalloc(lat, flags):
    import torch

    import paper_1608_04658_gb300 as lbm
    fn = lbm.lib().lbm_totals_noalloc
    fn.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p, C.c_void_p]
    out = torch.zeros(5, dtype=torch.float64, device=lat.device)
    assert fn(C.addressof(lat.params), lat.f.data_ptr(), lat.flags.data_ptr() if flags else None, out.data_ptr(),
              C.c_void_p(lat.stream.cuda_stream)) == 0
    return out.cpu().numpy()


# one node; a few nodes; more nodes than one flush of a thread's partial sums (16 * 608 * 256), with a body
@pytest.mark.parametrize("shape,body", [((1, 1, 1), False), ((7, 5, 3), False), ((33, 17, 21), True), ((160, 130, 130), True)])
@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16", "bf16"])
def test_totals_match_fp64_sums(storage, shape, body):
    import paper_1608_04658_gb300 as lbm
    rho, u, xi = synth.parity_fields(shape, 5)
    lat = lbm.Lattice(shape, 0.02, storage=storage, rho0=1.1)
    if body:
        lat.set_geometry(lbm.sphere((shape[0] / 2 + 0.1, shape[1] / 2, shape[2] / 2), 3.3))
    lat.init_state(1.1 * rho, u, xi, 1e-2)
    ref, mag = _reference(lat)
    # 27 additions a node and one per node in FP64 or in pairs of 48 bits, the latter on the deviations from rest
    # (a fiftieth of the populations); the sums over the nodes are FP64 (2^-53 each, tree of threads and blocks)
    tol = (64 * 2.0 ** -53 + 32 * 2.0 ** -48 / 50 + np.prod(shape) / 1e5 * 2.0 ** -53) * mag
    assert np.all(np.abs(lat.totals() - ref) <= tol)
    assert np.all(np.abs(_noalloc(lat, body) - ref) <= tol)


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_totals_of_a_broken_state(storage, bad):
    import paper_1608_04658_gb300 as lbm
    shape = (12, 6, 5)
    rho, u, xi = synth.parity_fields(shape, 6)
    lat = lbm.Lattice(shape, 0.02, storage=storage)
    lat.init_state(rho, u, xi, 1e-2)
    lat.f[13, 2, 3, 4] = bad  # the rest population: no finite component, so that no sum may stay finite
    for t in (lat.totals(), _noalloc(lat, False)):
        assert not np.isfinite(t).any()
        assert t[0] == bad or (np.isnan(t[0]) and np.isnan(bad))


def test_totals_of_large_populations():
    """Finite FP32 values whose FP32 sums overflow are summed in FP64."""
    import paper_1608_04658_gb300 as lbm
    lat = lbm.Lattice((4, 4, 4), 0.02, storage="fp32")
    lat.init_state(np.ones((4, 4, 4)), np.zeros((4, 4, 4, 3)))
    lat.f[:, 1, 1, 1] = 3e38
    ref, mag = _reference(lat)
    t = lat.totals()
    assert np.all(np.abs(t - ref)[:4] <= 1e-14 * mag[0])


@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
def test_kinetic_energy_has_no_bias(storage):
    """The signed error of the kinetic energy over twelve boxes: what the division of the pairs leaves out has one sign and
    does not average out over the nodes, the roundings of the sums do.  These: some 270 block sums added one after the
    other, 2^-53 of the running sum each, a walk of sqrt(270 / 3) of them, 1e-15 a box, 3e-16 of the mean of twelve; the
    bound is twice that."""
    import paper_1608_04658_gb300 as lbm
    shape, err = (48, 40, 36), []
    for seed in range(12):
        rho, u, xi = synth.parity_fields(shape, 100 + seed)
        lat = lbm.Lattice(shape, 0.02, storage=storage)
        lat.init_state(rho, u, xi, 1e-2)
        W = np.array([(64, 16, 4, 1)[int(np.abs(c).sum())] for c in CX], dtype=np.longdouble) / 216
        f = lat.f.double().cpu().numpy().reshape(27, -1).astype(np.longdouble) + W[:, None]
        ke = (0.5 * ((CX.T.astype(np.longdouble) @ f) ** 2).sum(0) / f.sum(0)).sum()
        err.append(float((np.longdouble(lat.totals()[4]) - ke) / ke))
        lat.close()
    assert abs(np.mean(err)) <= 6e-16, err
