"""What a gradient call takes from the state before it and leaves behind: the free yaw's initial spin whatever the number
of segments, the body after odd and even horizons, the body after a call that fails, and the memory that it asks for."""
import numpy as np
import pytest
import torch

import synth

pytestmark = pytest.mark.gpu


def _allocator(lat):
    """Blocks that hold NaNs (0xFF bytes) where nothing has been written; returns the sizes asked for."""
    live, sizes = {}, []

    def alloc(n, stream):
        t = torch.full((n,), 0xFF, dtype=torch.uint8, device=lat.device)
        torch.cuda.synchronize()
        live[t.data_ptr()] = t
        sizes.append(n)
        return t.data_ptr()

    lat.use_allocator(alloc, lambda p, stream: live.pop(p))
    return sizes


def _swimmer(free, shape=(48, 24, 24)):
    """A turning swimmer in the centre-of-mass frame."""
    import paper_1608_04658_gb300 as lbm
    rest, tris = synth.swimmer_mesh(24.0, 48, 16)
    rho, u, xi = synth.parity_fields(shape, 47)
    lat = lbm.Lattice(shape, 0.02, storage="fp64")
    sizes = _allocator(lat)
    lat.set_geometry(lbm.swimmer((24.137, 12.371, 12.293), rest, tris, 24.0, 0.125, 24.0, 96.0, free=free, mass=synth.swimmer_volume(24.0),
                                 U=(-0.01, 0.004, 0.0), psi=0.1, omega=0.003))
    lat.init_state(rho, 0.2 * u, xi, 1e-3)
    return lat, sizes


@pytest.mark.parametrize("free", [4, 7])
@pytest.mark.parametrize("horizon", [1, 2, 5, 12])
def test_spin_gradient_does_not_depend_on_the_segments(free, horizon):
    """K = horizon is one segment, K = 1 as many as there are steps; with the default of ceil(sqrt(horizon)) horizons 1 and
    2 are one segment too.  Equal but for the order of the double atomics into the band slots (1e-12, as for the held
    swimmer)."""
    res = []
    for K in (horizon, 1, 4, 0):
        lat, _ = _swimmer(free)
        res.append(lat.adjoint(horizon, (-1.0, 0.0, 0.0), want_lambda0=True, checkpoint_every=K))
        lat.close()
    assert np.all(np.isfinite(res[0]["dJ_dtheta"])) and np.abs(res[0]["dJ_dtheta"]).max() > 0
    for r in res[1:]:
        assert r["J"] == res[0]["J"]
        assert np.allclose(r["dJ_dtheta"], res[0]["dJ_dtheta"], rtol=1e-12, atol=1e-14 * np.abs(res[0]["dJ_dtheta"]).max())


def _sphere(storage, shape=(24, 20, 22)):
    import paper_1608_04658_gb300 as lbm
    rho, u, xi = synth.parity_fields(shape, 4)
    lat = lbm.Lattice(shape, 0.02, storage=storage, faces=(1, 1, 1, 1, 0, 0))
    lat.set_geometry(lbm.sphere((11.37, 9.61, 10.83), 4.3, U=(0.02, -0.01, 0.03), free=True, g=(0, 0, -1e-4)))
    lat.init_state(rho, 0.3 * u, xi, 1e-3)
    return lat


def _same_body(a, b):
    return all(np.array_equal(np.asarray(a[k]), np.asarray(b[k])) for k in a if k != "n_band")


@pytest.mark.parametrize("storage", ["fp64", "fp32", "fp16"])
@pytest.mark.parametrize("horizon,K", [(1, 0), (2, 0), (3, 0), (3, 1), (3, 3), (4, 0), (7, 2)])
def test_context_goes_on_as_after_the_steps(storage, horizon, K):
    """The body, the populations and the steps that follow are those of lbm_step, bit for bit."""
    lat, ref = _sphere(storage), _sphere(storage)
    for l in (lat, ref):
        l.set_launch_order("split")
    lat.adjoint(horizon, (1.0, 0.0, 0.5), checkpoint_every=K)
    ref.step(horizon)
    for _ in range(3):
        assert _same_body(lat.body(), ref.body())
        fluid = (ref.flags & 1) == 0
        assert torch.equal(lat.flags, ref.flags) and torch.equal(lat.f[:, fluid], ref.f[:, fluid])
        lat.step(1)
        ref.step(1)


def test_failed_forward_run_leaves_the_body_alone():
    """More rows than a grid has (65,535): the forward run's first bulk launch is refused, before anything of the body has
    been saved to be restored."""
    import paper_1608_04658_gb300 as lbm
    shape = (12, 65540, 12)
    lat = lbm.Lattice(shape, 0.02, storage="fp16")
    _allocator(lat)
    lat.set_geometry(lbm.sphere((5.7, 30000.3, 6.1), 3.3, U=(0.02, -0.01, 0.03), free=True))
    lat.init_state(torch.ones(shape[::-1], device=lat.device), torch.zeros((*shape[::-1], 3), device=lat.device))
    before = lat.body()
    with pytest.raises(lbm.LbmError):
        lat.adjoint(3, (1.0, 0.0, 0.0))
    assert _same_body(lat.body(), before)


@pytest.mark.parametrize("storage,es,rs", [("fp64", 8, 8), ("fp32", 4, 4), ("fp16", 2, 4)])
@pytest.mark.parametrize("horizon,K", [(1, 1), (7, 3), (9, 9)])
def test_memory_asked_for(storage, es, rs, horizon, K):
    """What include/lbm.h says of a box without a body: ceil(horizon/K) + K - 1 states in the storage type, two in the
    adjoint's, (ceil(horizon/K) + K + 4) N bytes of marks (and a few kilobytes)."""
    import paper_1608_04658_gb300 as lbm
    shape = (40, 32, 24)
    N, nseg = 40 * 32 * 24, -(-horizon // K)
    lat = lbm.Lattice(shape, 0.02, storage=storage)
    sizes = _allocator(lat)
    lat.init_state(*synth.uniform_fields(shape))
    lat.adjoint(horizon, lambda_T=torch.ones((27,) + shape[::-1], device=lat.device), checkpoint_every=K)
    bound = (nseg + K - 1) * 27 * N * es + 2 * 27 * N * rs + (nseg + K + 4) * N + 65536
    assert 0.9 * bound < sum(sizes) <= bound
