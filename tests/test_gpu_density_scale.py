"""The step does not depend on the unit of density: reference densities far from 1, in which populations, and even more
their products, are very small or very large FP32 numbers."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

SCALES = [1e-14, 1e-7, 1e7, 1e14]


def _lat(storage, rho0, gamma, body, shape=(34, 18, 16)):
    import paper_1608_04658_gb300 as lbm
    rho, u, xi = synth.parity_fields(shape, 23)
    lat = lbm.Lattice(shape, 0.02, storage=storage, rho0=rho0, gamma_mode=gamma)
    if body:
        lat.set_geometry(lbm.sphere((16.3, 8.6, 7.7), 3.3, U=(0.02, -0.01, 0.015)))
        lat.f_b.zero_()  # solid nodes hold no defined state
    lat.init_state(rho * rho0, u, xi, 1e-2 * rho0)
    return lat


@pytest.mark.parametrize("rho0", SCALES)
@pytest.mark.parametrize("storage", ["fp64", "fp32", "bf16"])
@pytest.mark.parametrize("gamma", [0, 1])
@pytest.mark.parametrize("body", [False, True])
def test_step(storage, rho0, gamma, body):
    """Populations over rho0 against those of rho0 = 1 (a power of ten is no power of two, so roundings differ): two steps,
    some 2^-24 (FP32) or 2^-8 of the shifted value (BF16) a step, of values below 0.3."""
    tol = {"fp64": 1e-13, "fp32": 2e-6, "bf16": 4e-3}[storage]
    out = []
    for r in (1.0, rho0):
        lat = _lat(storage, r, gamma, body)
        lat.step(2)
        out.append(lat.f.double() / r)
    assert float((out[0] - out[1]).abs().max()) <= tol


@pytest.mark.parametrize("rho0", SCALES)
@pytest.mark.parametrize("storage", ["fp64", "fp32"])
@pytest.mark.parametrize("nx", [34, 33])
def test_gradient(storage, rho0, nx):
    """lambda_0 = d(lambda_T . f)/df has no unit: the same for every rho0, to the rounding of the adjoint's arithmetic (1e-4
    of the largest entry, as between FP32 and FP64 in test_gpu_adjoint_forms.py)."""
    shape, out = (nx, 18, 16), []
    lamT = torch.tensor(np.random.default_rng(3).normal(size=(27,) + shape[::-1]))
    for r in (1.0, rho0):
        lat = _lat(storage, r, 0, False, shape)
        out.append(lat.adjoint(2, lambda_T=lamT.to(lat.device), want_lambda0=True)["lambda_0"].double())
    assert float((out[0] - out[1]).abs().max()) <= (1e-10 if storage == "fp64" else 1e-4) * float(out[0].abs().max())
