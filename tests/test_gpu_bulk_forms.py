"""The bulk update's forms at the sizes where each begins and ends: rows of one to three nodes and of one node more or
less than a warp's pairs, in every storage form and with each stabilizer, against the FP64 oracle; the forms of the
collision that 16-bit storage takes below and above the size at which it changes."""
import numpy as np
import pytest

import oracle
import synth
from parity_util import rel_err

pytestmark = pytest.mark.gpu

FACES = {"periodic": (0,) * 6, "walls": (1, 1, 1, 1, 0, 0), "tunnel": (2, 3, 2, 2, 0, 0), "mixed": (1, 2, 2, 3, 1, 2)}
TOL = {"fp64": 1e-12, "fp32": 2e-6, "fp16": 2e-3, "bf16": 8e-3}  # two steps; half an ulp of the shifted value a store


@pytest.mark.parametrize("nx", [1, 2, 3, 63, 64, 65, 66, 127, 129])
@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16", "bf16"])
@pytest.mark.parametrize("faces", list(FACES))
def test_row_lengths(nx, storage, faces):
    import paper_1608_04658_gb300 as lbm
    shape = (nx, 5, 4)
    rho, u, xi = synth.parity_fields(shape, 71)
    for gamma in (0, 1, 2):
        lat = lbm.Lattice(shape, 0.02, storage=storage, faces=FACES[faces], u_face=(0.03, 0.01, -0.02), gamma_mode=gamma)
        lat.init_state(rho, u, xi, 1e-2)
        orc = oracle.Oracle(shape, nu=0.02, faces=FACES[faces], u_face=(0.03, 0.01, -0.02), gamma_mode=gamma)
        orc.init_state(rho, u, xi, 1e-2)
        lat.step(2)
        orc.step(2)
        assert rel_err(lat.populations(), orc.get_f()) < TOL[storage], gamma


@pytest.mark.parametrize("storage,tol", [("fp32", 1e-4), ("fp16", 2e-2)])
def test_exact_stabilizer_far_from_equilibrium(storage, tol):
    """Noise of a third of the weights: post-collision populations from a few hundredths of equilibrium to twice it, so
    that nodes take the safeguarded iteration beside others that the one-pass root serves.  Bounds: ten FP32 roundings
    of W against populations of 0.02 W; half an FP16 ulp of 0.3 W against 0.02 W, twice."""
    import paper_1608_04658_gb300 as lbm
    shape = (66, 6, 5)
    rho, u, xi = synth.parity_fields(shape, 73)
    amp = np.linspace(0.0, 0.3, shape[0])
    xi = xi * amp
    lat = lbm.Lattice(shape, 0.02, storage=storage, gamma_mode=1)
    orc = oracle.Oracle(shape, nu=0.02, gamma_mode=1)
    lat.init_state(rho, u, xi, 1.0)
    orc.init_state(rho, u, xi, 1.0)
    orc.set_f(lat.populations())
    lat.step(1)
    orc.step(1)
    assert rel_err(lat.populations(), orc.get_f()) < tol


@pytest.mark.parametrize("nz", [255, 257])
def test_16bit_forms_on_either_side_of_their_line(nz):
    """A 256x128xnz box is below (2^23 nodes) or above; with a body the lattice takes one form or the other and has to
    agree with FP64 storage to the storage's own rounding either way."""
    import torch

    import paper_1608_04658_gb300 as lbm
    out = {}
    for storage in ("fp64", "fp16"):
        lat = lbm.Lattice((256, 128, nz), 0.01, storage=storage)
        lat.set_geometry(lbm.sphere((128.3, 64.2, 100.1), 9.0, U=(0.02, 0.0, 0.0)))
        gen = torch.Generator(device="cuda").manual_seed(5)
        u = 0.03 * (2 * torch.rand((nz, 128, 256, 3), generator=gen, device="cuda") - 1)
        lat.init_state(torch.ones((nz, 128, 256), device="cuda"), u)
        lat.step(1)
        fluid = (lat.flags & 1) == 0
        out[storage] = (lat.f.double(), fluid)
    a, fluid = out["fp64"]
    b, _ = out["fp16"]
    d = (a - b)[:, fluid]
    # one rounding on set-up, one on the store: 2^-11 of values spread over the weights, of both signs
    assert float(d.norm() / a[:, fluid].norm()) < 2 * 2.0 ** -11
