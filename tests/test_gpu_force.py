"""The force and torque of a step (boundary kernel's per-node sums, force kernel) against a plain FP64 evaluation of the
momentum exchange over the links, for a body whose wall moves and whose links have every fraction."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


# a sphere of a few links, one of several hundred boundary nodes, one across the periodic edge; airfoil and swimmer
# against the oracle are in test_gpu_parity.py
@pytest.mark.parametrize("shape,X,R", [((12, 13, 14), (6.1, 6.3, 6.2), 1.3), ((40, 36, 44), (19.7, 18.2, 21.9), 11.4),
                                       ((33, 20, 22), (32.6, 10.2, 0.4), 5.2)])
@pytest.mark.parametrize("storage,tol", [("fp64", 1e-11), ("fp32", 2e-5), ("fp16", 2e-2), ("bf16", 2e-1)])
def test_force_and_torque_match_the_oracle(shape, X, R, storage, tol):
    import paper_1608_04658_gb300 as lbm
    U = (0.03, -0.05, 0.02)
    rho, u, xi = synth.parity_fields(shape, 17)
    lat = lbm.Lattice(shape, 0.02, storage=storage, rho0=1.2)
    lat.set_geometry(lbm.sphere(X, R, U=U))
    lat.init_state(1.2 * rho, u, xi, 1e-2)
    orc = oracle.Oracle(shape, nu=0.02, rho0=1.2, body=oracle.sphere_body(X, R, U=U))
    orc.init_state(1.2 * rho, u, xi, 1e-2)
    for _ in range(2):
        lat.step(1)
        orc.step(1)
        F, M = lat.forces()
        Fo, Mo = np.array(orc.body.F), np.array(orc.body.M)
        # rounding of the populations (half an ulp of storage of values below 0.05, some 1e-3 of the wall's
        # momentum flux) against the force's own size, a factor of ten for the sums of both signs
        assert np.abs(F - Fo).max() <= tol * max(np.abs(Fo).max(), 1e-2)
        assert np.abs(M - Mo).max() <= tol * R * max(np.abs(Mo).max() / R, np.abs(Fo).max(), 1e-2)
