"""The V-cycle's coarse kernels against the oracle at the sizes where they
change shape."""
import numpy as np
import pytest

import dp_inputs as di
import oracle as O
from test_gpu_parity import gpu, interior, small

pytestmark = pytest.mark.gpu


def relres(prob, its, state=None, **kw):
    """Relative residual after `its` FGMRES iterations from zero, both sides."""
    out = []
    for s in (gpu().Sim(prob, gpu().options("parity", eta_fixed=1e-14, gmres_maxit=its, **kw)),
              O.OracleSim(prob, O.options("parity", eta_fixed=1e-14, gmres_maxit=its,
                                          **{k: v for k, v in kw.items() if k != "cluster_rows"}))):
        if state is not None:
            s.set_iterate(*state)
        s.assemble(prob.dt)
        _, st = s.solve_step()
        out.append(st.lin_relres)
    return out


# n = 2 nx (+ 1 with the well): one warp row, the 32-row register steps of the
# inverse's columns, even and odd leading dimensions, the largest size of the
# shared-memory factorisation (160) and one beyond it (its predecessor runs)
@pytest.mark.parametrize("nx,wells", [(1, "none"), (1, "bhp"), (15, "bhp"), (16, "none"),
                                      (16, "bhp"), (32, "none"), (32, "bhp"), (48, "bhp"),
                                      (64, "none"), (64, "bhp"), (79, "bhp"), (80, "none"),
                                      (80, "bhp"), (101, "bhp")])
def test_dense_coarsest_level(nx, wells):
    """A hierarchy of one level is the dense solve itself: after two iterations
    from a random state (rows change places) both sides have the same residual,
    to the 1e-6 of the preconditioner comparisons of test_gpu_parity plus the
    rounding floor of a solve."""
    prob = small(nx, 1, 1, wells=wells)
    g, o = relres(prob, 2, interior(prob, nx), amg_coarse_max=256)
    assert abs(g - o) <= 1e-6 * o + 1e-12
