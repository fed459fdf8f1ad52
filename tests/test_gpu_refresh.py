"""Level 0 of the V-cycle takes the current pressure block at every Newton
iteration, also when the coarse values are kept for a timestep (amg_refresh
1) and level 0 runs inside the cluster cycle."""
import numpy as np
import pytest

import dp_inputs as di
import oracle as O
from test_gpu_parity import gpu, interior, small

pytestmark = pytest.mark.gpu


def second_solve(s, prob):
    """(iterations, relative residual) of a timestep's second Newton solve, at
    an iterate far from the first one's."""
    s.assemble(prob.dt)
    rc, _ = s.solve_step()
    assert rc == 0
    p, sw, bhp = interior(prob, 21)
    s.set_iterate(p, np.clip(sw + 0.2 * (np.arange(len(sw)) % 3), 0.2, 0.8), bhp)
    s.assemble(prob.dt * 20.0)
    rc, st = s.solve_step()
    assert rc == 0
    return st.linear_iters, st.lin_relres


# the whole cycle in the cluster: Gauss-Seidel on every level, or on the
# finest only
@pytest.mark.parametrize("make", [di.tiny, lambda: small(17, 16, 15)])
@pytest.mark.parametrize("gs_levels", [30, 1])
@pytest.mark.parametrize("precision", [0, 1])
def test_cluster_level_0_is_current(make, gs_levels, precision):
    """The second solve against the oracle's and against the cycle of one
    launch a phase: as many iterations and the same residual, to the 1e-6 of
    the FP64 preconditioner comparisons, or the 1e-2 that five to ten
    iterations leave of an FP32 preconditioner's 24 bits."""
    prob = make()
    kw = dict(eta_fixed=1e-4, amg_refresh=1, amg_gs_levels=gs_levels)
    c = second_solve(gpu().Sim(prob, gpu().options("parity", precision=precision, **kw)), prob)
    g = second_solve(gpu().Sim(prob, gpu().options("parity", precision=precision, cluster_rows=-1,
                                                   **kw)), prob)
    o = second_solve(O.OracleSim(prob, O.options("parity", **kw)), prob)
    tol = 1e-2 if precision else 1e-6
    for other in (g, o):
        assert c[0] == other[0], (c, g, o)
        assert abs(c[1] - other[1]) <= tol * other[1] + 1e-11, (c, g, o)
