"""Parameter terms of the reverse sweep, several steps to a launch: the gradient does not depend on how
the checkpoints cut the steps into launches."""
import numpy as np
import pytest

import hmc_synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    from conftest import build_libhmc
    build_libhmc()
    import paper_1009_0457_gb300 as G
    return G


# The states and lambdas are the same bits whatever the cut, a cell's terms too; only sums change their
# order.  FP32: TwoSum pairs, so what is left is one rounding (2^-24) of a node's summed lambda; FP64:
# 2^-53 times the square root of 17 x 1836 summands.
@pytest.mark.parametrize("precision,tol", [(0, 1e-12), (1, 1e-6)])
@pytest.mark.parametrize("steps", [1, 8, 9, 17])
def test_gradient_is_independent_of_the_checkpoints(G, precision, tol, steps):
    shape, Q = (12, 18, 68), 6
    eul, sp = S.euler_uniform_so3(Q, 7), S.voronoi_spins(shape, 9, Q, 8)
    ref = None
    for ck in (1, 7, 8, 9, 16, 17, 40):
        g = G.HMC(shape, Q, c11=246.5, c12=147.3, c44=124.7, bc=G.HMC_BC_STRAIN6,
                  strain6=(1e-3, -3e-4, -4e-4, 2e-4, -1e-4, 1e-4), mpm_steps_per_mcs=0, precision=precision)
        g.set_orientations(eul, sp)
        g.adjoint_forward(steps, ck)
        grad = [np.array(g.adjoint_backward(1.0, None)) for _ in range(2)]
        g.close()
        assert np.array_equal(grad[0], grad[1])   # a second reverse sweep finds what the first one found
        if ref is None:
            ref = grad[0]
        for part in (slice(0, 3), slice(3, 9)):
            assert np.abs(grad[0][part] - ref[part]).max() <= tol * np.abs(ref[part]).max()
