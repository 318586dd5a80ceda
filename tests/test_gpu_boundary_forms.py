"""The boundary kernel's single-precision link search and its two ways to a node's sources (off the box faces, on them)
against the FP64 kernels from the same state."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

FACES = {"periodic": (0,) * 6, "walls": (1, 1, 1, 1, 0, 0), "tunnel": (2, 3, 2, 2, 0, 0), "mixed": (1, 2, 2, 3, 1, 2)}


def _compare(shape, faces, geometry, u0, tol):
    """One step, FP32 against FP64 from the FP32 lattice's initial populations; FP32 roundings of f (2^-24 of values up
    to 1) and of a link fraction (tol) of a wall momentum of 0.1 W."""
    import paper_1608_04658_gb300 as lbm
    rho, u, xi = synth.parity_fields(shape, 29)
    f, out = None, []
    for storage in ("fp32", "fp64"):
        lat = lbm.Lattice(shape, 0.02, storage=storage, faces=faces, u_face=u0)
        lat.f_b.zero_()  # solid nodes hold no defined state
        lat.set_geometry(geometry)
        lat.init_state(rho, 0.2 * u + np.array(u0), xi, 1e-3)
        if f is None:
            f = lat.populations()
        else:
            lat.set_populations(f)
        lat.step(1)
        b = lat.body()
        out.append((lat.populations(), np.array(b["F"]), (b["n_boundary"], b["n_uncovered"], b["n_links"]), b["status"]
                    if "status" in b else 0))
    assert out[0][2] == out[1][2] and out[0][2][0] > 0
    assert np.abs(out[0][0] - out[1][0]).max() <= tol
    assert np.abs(out[0][1] - out[1][1]).max() <= tol * out[0][2][2]


@pytest.mark.parametrize("faces", list(FACES))
@pytest.mark.parametrize("X", [(4.3, 9.6, 8.8), (19.6, 3.2, 12.9), (11.8, 15.7, 2.1)])
def test_sphere_at_the_box_faces(faces, X):
    import paper_1608_04658_gb300 as lbm
    U = (0.04, -0.03, 0.05)
    _compare((24, 19, 17), FACES[faces], lbm.sphere(X, 4.2, U=U), (0.03, 0.0, 0.0), 2e-6)


@pytest.mark.parametrize("chord", [17.3, 32.0, 60.7])
@pytest.mark.parametrize("angle", [-25.0, 0.0, 4.0, 90.0])
def test_airfoil_link_search(chord, angle):
    """Nose, trailing edge and both sides at four angles; a link's fraction is known to 2^-24 of the chord over the
    slope of the outline's margin along the link, a few 1e-5 but where the link grazes the outline."""
    import paper_1608_04658_gb300 as lbm
    wl = synth.plunging_airfoil()
    ca, sa = np.cos(np.radians(angle)), np.sin(np.radians(angle))
    shape = (90, 90, 5)
    le = (45.37 - 0.5 * chord * ca, 44.81 + 0.5 * chord * sa)
    geo = lbm.airfoil(le, chord, float(ca), float(sa), 1.6, 0.05, wl["camber_m"], wl["camber_p"], wl["thick"], 3.0)
    _compare(shape, FACES["tunnel"], geo, (0.05, 0.0, 0.0), 2e-5)
