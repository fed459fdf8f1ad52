"""Small realisations (up to 8192 rows), whose preconditioner, coarse cycle and
Arnoldi step run as cluster launches: several of them at once on streams of
their own, and the update of a solve, not its residual alone."""
import threading

import numpy as np
import pytest

import dp_inputs as di
from test_gpu_parity import gpu, interior, small, update_close

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,precision", [("parity", 0), ("report", 1)])
def test_several_streams_equal_alone(mode, precision):
    """Eight realisations of 2 to 8192 rows, each advanced twice by its own
    host thread on its own stream: the states each has alone, bit for bit."""
    d = gpu()
    probs = [small(1, 1, 1, wells="bhp"), di.tiny(), small(7, 5, 3), small(6, 5, 40),
             small(17, 16, 15), small(64, 64, 1, wells="none"), di.tiny(3), small(17, 16, 15, seed=4)]

    def advance(sims):
        out = [None] * len(sims)

        def one(k):
            rcs = [sims[k].advance(probs[k].dt)[0] for _ in range(2)]
            out[k] = rcs, sims[k].get_state()
        return out, one

    alone = []
    for k, p in enumerate(probs):
        s = d.Sim(p, d.options(mode, precision=precision))
        rcs = [s.advance(p.dt)[0] for _ in range(2)]
        alone.append((rcs, s.get_state()))
        s.close()
    streams = [d.OwnedStream() for _ in probs]
    sims = [d.Sim(p, d.options(mode, precision=precision), stream=s.torch)
            for p, s in zip(probs, streams)]
    out, one = advance(sims)
    threads = [threading.Thread(target=one, args=(k,)) for k in range(len(sims))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for a, b in zip(alone, out):
        assert a[0] == b[0] == [0, 0]
        for x, y in zip(a[1], b[1]):
            np.testing.assert_array_equal(x, y)
    for s in sims:
        s.close()
    for s in streams:
        s.close()


@pytest.mark.parametrize("grid,wells", [((1, 1, 1), "bhp"), ((7, 5, 3), "two"), ((64, 64, 1), "none"),
                                        ((17, 16, 15), "two")])
@pytest.mark.parametrize("kw", [{}, dict(gmres_restart=3, reorth=1e-10), dict(schur=1),
                                dict(precision=1, reorth=2.0)])
def test_update_of_a_solve(grid, wells, kw):
    """The update of a solve to 1e-11 with the cluster launches against the one
    with a launch a phase, to the parity tolerance."""
    prob = small(*grid, wells=wells)
    state = interior(prob, 3)
    y = []
    for rows in (0, -1):
        s = gpu().Sim(prob, gpu().options("parity", eta_fixed=1e-11, cluster_rows=rows, **kw))
        s.set_iterate(*state)
        s.assemble(prob.dt)
        rc, _ = s.solve_step()
        assert rc == 0
        y.append(s.update())
        s.close()
    update_close(y[0], y[1], prob.n_cells)
