"""The bulk adjoint's one-node and two-node forms at the row lengths where each begins and ends, in every storage form,
against the FP64 form (which the tape of the oracle checks) from the same state."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu

FACES = {"periodic": (0,) * 6, "walls": (1, 1, 1, 1, 0, 0), "tunnel": (2, 3, 2, 2, 0, 0), "mixed": (1, 2, 2, 3, 1, 2)}


@pytest.mark.parametrize("nx", [1, 2, 3, 4, 62, 64, 65, 66, 130])
@pytest.mark.parametrize("storage", ["fp32", "fp16", "bf16"])
@pytest.mark.parametrize("faces", list(FACES))
def test_row_lengths(nx, storage, faces):
    """One step, so that no rounding of a store enters: the FP32 arithmetic of the adjoint alone, whose stabilizer
    divides sums of d = g - g^eq, 1e-2 of W here, known to 2^-24 of g, 0.05 W and more: some 1e-6, a hundred of it for
    the worst of 27 N entries."""
    import paper_1608_04658_gb300 as lbm
    shape = (nx, 5, 4)
    rho, u, xi = synth.parity_fields(shape, 71)
    lamT = np.random.default_rng(5).normal(size=(27,) + shape[::-1]).astype(np.float32)
    for gamma in (0, 2):
        out = []
        f = None
        for st in (storage, "fp64"):
            lat = lbm.Lattice(shape, 0.02, storage=st, faces=FACES[faces], u_face=(0.03, 0.01, -0.02), gamma_mode=gamma)
            lat.init_state(rho, u, xi, 1e-2)
            if f is None:
                f = lat.populations()
            else:
                lat.set_populations(f)
            # (an array that begins 4 bytes off an 8-byte boundary: the caller's own)
            t = torch.empty(lamT.size + 1, dtype=torch.float32, device=lat.device)[1:].view(lamT.shape)
            t.copy_(torch.tensor(lamT))
            out.append(lat.adjoint(1, lambda_T=t, want_lambda0=True)["lambda_0"].double().cpu().numpy())
        assert np.abs(out[0] - out[1]).max() <= 1e-4 * np.abs(out[1]).max(), gamma


@pytest.mark.parametrize("nx", [34, 35])
def test_several_steps_with_a_body_near_the_faces(nx):
    """The pairs that a band's edge, a solid node or a refilled node cuts: a moving sphere, FP32 against FP64 over
    three steps (states that differ by 2^-24 of W a step, beside the bound above)."""
    import paper_1608_04658_gb300 as lbm
    shape = (nx, 20, 18)
    rho, u, xi = synth.parity_fields(shape, 73)
    rng = np.random.default_rng(7)
    lamT = rng.normal(size=(27,) + shape[::-1])
    for order in ("split", "sequential"):
        out = []
        for st in ("fp32", "fp64"):
            lat = lbm.Lattice(shape, 0.02, storage=st, faces=(0, 0, 1, 1, 0, 0))
            lat.set_geometry(lbm.sphere((16.3, 9.6, 8.7), 4.3, U=(0.2, -0.1, 0.15)))
            lat.set_launch_order(order)
            lat.init_state(rho, 0.2 * u, xi, 1e-2)
            r = lat.adjoint(3, (0.3, -1.0, 0.2), lambda_T=torch.tensor(lamT, device=lat.device), want_lambda0=True)
            out.append(r["lambda_0"].double().cpu().numpy())
        assert np.abs(out[0] - out[1]).max() <= 1e-3 * np.abs(out[1]).max(), order
