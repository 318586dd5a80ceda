"""A launch that the CUDA runtime refuses is reported by the call that asked for it, and by no later one."""
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_refused_step_leaves_no_error_behind():
    """More rows than a grid has (65,535): the step is refused; what follows, on this lattice or another, is not."""
    import paper_1608_04658_gb300 as lbm
    tall = lbm.Lattice((2, 65536, 2), 0.02, storage="fp32")
    rho, u = synth.uniform_fields(tall.shape)
    tall.init_state(rho, u)
    with pytest.raises(lbm.LbmError):
        tall.step(1)
    tall.init_state(rho, u)
    with pytest.raises(lbm.LbmError):
        tall.step(1)
    small = lbm.Lattice((8, 8, 8), 0.02, storage="fp32")
    small.init_state(*synth.uniform_fields(small.shape))
    small.step(1)
