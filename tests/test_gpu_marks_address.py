"""The caller's node marks are bytes and may begin at an odd address."""
import ctypes as C

import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def _lat(storage, gamma, odd, order):
    import paper_1608_04658_gb300 as lbm
    shape = (34, 20, 18)
    rho, u, xi = synth.parity_fields(shape, 61)
    lat = lbm.Lattice(shape, 0.02, storage=storage, gamma_mode=gamma)
    if odd:
        lbm.lib().lbm_destroy(lat._ctx)
        lat.flags = torch.zeros(lat.N + 1, dtype=torch.uint8, device=lat.device)[1:].view(lat.flags.shape)
        lat._ctx = C.c_void_p()
        assert lat.flags.data_ptr() % 2 == 1
        assert lbm.lib().lbm_create(C.byref(lat.params), lat.f_a.data_ptr(), lat.f_b.data_ptr(), lat.flags.data_ptr(),
                                    C.c_void_p(lat.stream.cuda_stream), C.byref(lat._ctx)) == 0
    lat.f_b.zero_()
    lat.set_geometry(lbm.sphere((16.3, 9.6, 8.7), 4.3, U=(0.02, -0.01, 0.015)))
    lat.set_launch_order(order)
    lat.init_state(rho, 0.2 * u, xi, 1e-2)
    lat.step(2)
    return lat


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("gamma", [0, 1])
@pytest.mark.parametrize("order", ["split", "sequential"])
def test_same_bits(storage, gamma, order):
    a, b = _lat(storage, gamma, False, order), _lat(storage, gamma, True, order)
    assert torch.equal(a.flags, b.flags) and torch.equal(a.f, b.f)
