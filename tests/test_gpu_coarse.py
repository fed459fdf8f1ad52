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


# where the cluster cycle's vectors live (FP64, shared budget 224 KB): everything
# replicated (levels of 3268 rows down); x replicated, the right-hand sides and
# residuals in global memory (about 15000 rows down, its colours in several
# trips); a level whose x does not fit (29828 rows) is left to its own launches;
# l1-Jacobi below the finest in the cluster
@pytest.mark.parametrize("grid,gs_levels,cluster_rows",
                         [((100, 100, 10), 30, 4000), ((80, 80, 8), 30, 0),
                          ((100, 100, 10), 30, 40000), ((80, 80, 8), 1, 20000)])
def test_cluster_cycle_vectors(grid, gs_levels, cluster_rows):
    g, o = relres(di.layered(*grid), 3, amg_gs_levels=gs_levels, cluster_rows=cluster_rows)
    assert abs(g - o) <= 1e-6 * o


@pytest.mark.parametrize("coarse_max", [2, 40, 2000])
def test_cluster_cycle_from_level_0(coarse_max):
    """The whole cycle in the cluster (602 rows), down to a coarsest level that
    is smoothed, dense, or level 0 itself."""
    prob = di.tiny()
    g, o = relres(prob, 3, interior(prob, 5), amg_coarse_max=coarse_max)
    assert abs(g - o) <= 1e-6 * o + 1e-12


def test_small_realisations_dependent_launches_change_no_result():
    """Every kernel of an Arnoldi step as a programmatic dependent (DPSIM_PDL
    63, the default) or that class off (31): the same state, bit for bit, in a
    child process each."""
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    code = ("import sys; sys.path.insert(0, sys.argv[1])\n"
            "import dp_inputs as di, numpy as np\n"
            "from paper_1808_04338_gb300 import dpsim\n"
            "h = []\n"
            "for prob, mode, kw in ((di.tiny(), 'parity', {}), (di.layered(31, 29, 6), 'parity', {}),\n"
            "                       (di.layered(47, 45, 5), 'report', dict(precision=1)),\n"
            "                       (di.layered(47, 45, 5), 'report', dict(precision=2, schur=1))):\n"
            "    s = dpsim.Sim(prob, dpsim.options(mode, **kw))\n"
            "    rc, st = s.advance(prob.dt)\n"
            "    assert rc == 0\n"
            "    h += [a.tobytes().hex() for a in s.get_state()] + [st.linear_iters]\n"
            "import hashlib; print(hashlib.sha256(repr(h).encode()).hexdigest())\n")
    out = [subprocess.run([sys.executable, "-c", code, root], capture_output=True, text=True,
                          env=dict(os.environ, DPSIM_PDL=m), check=True).stdout for m in ("63", "31")]
    assert out[0] == out[1] and len(out[0].strip()) == 64


@pytest.mark.parametrize("gravity", [0.0, 9.80665])
@pytest.mark.parametrize("capillary", [False, True])
@pytest.mark.parametrize("swc_fraction", [0.0, 0.5, 1.0])
def test_assembly_with_resting_phases_bit_exact(gravity, capillary, swc_fraction):
    """J and R bit for bit, signs of zeros included, where a phase is at its
    residual saturation (its flux terms are left out) in none, half or all of
    the cells, for both flow directions; three kinds of wells, one of them
    with more perforations than a warp has lanes."""
    from test_gpu_parity import with_pc
    prob = small(6, 5, 40, wells="none", g=gravity)
    prob.wells = [di.Well(di.WELL_RATE_INJ, 0, 0, 0, 39, 100.0 * di.BBL_DAY),
                  di.Well(di.WELL_BHP, 5, 4, 3, 3, 2500.0 * di.PSI),
                  di.Well(di.WELL_OIL_RATE, 2, 2, 1, 38, 1.0, limit=15.0 * di.PSI)]
    prob.bhp0 = np.array([3100.0, 2500.0, 2700.0]) * di.PSI
    if capillary:
        with_pc(prob)
    rng = np.random.default_rng(11)
    nc = prob.n_cells
    p = prob.p0 + rng.uniform(-3e5, 3e5, nc)
    p[::7] = prob.p0[::7]                      # equal pressures too
    sw = rng.uniform(0.25, 0.75, nc)
    rest = rng.random(nc) < swc_fraction
    sw[rest] = np.where(rng.random(rest.sum()) < 0.5, prob.swc, 1.0 - prob.sor)
    out = []
    for s in (gpu().Sim(prob, gpu().options("parity")), O.OracleSim(prob, O.options("parity"))):
        s.set_iterate(p, sw, prob.bhp0)
        s.assemble(prob.dt)
        out.append(s.jacobian())
    for g, o in zip(out[0][2:], out[1][2:]):
        assert np.array_equal(g.view(np.uint64), o.view(np.uint64))


def few(prob, its, kw, state):
    """(iterations, relative residual, update) of one solve of at most `its` iterations."""
    s = gpu().Sim(prob, gpu().options("parity", eta_fixed=1e-13, gmres_maxit=its, **kw))
    s.set_iterate(*state)
    s.assemble(prob.dt)
    _, st = s.solve_step()
    return st.linear_iters, st.lin_relres


# the cluster launches of a small realisation against one launch a phase
# (cluster_rows < 0): a location, no wells, a well of short rows and of long
# rows (more than 24 blocks), the last size that takes them (8192 rows) and
# the next, restarts, one and two Gram-Schmidt passes, precisions, the
# eliminated system
@pytest.mark.parametrize("grid,wells", [((1, 1, 1), "bhp"), ((9, 1, 1), "none"), ((7, 5, 3), "two"),
                                        ((6, 5, 40), "two"), ((64, 64, 1), "none"),
                                        ((64, 64, 1), "bhp"), ((17, 16, 15), "two")])
@pytest.mark.parametrize("kw", [{}, dict(gmres_restart=3, reorth=1e-10), dict(schur=1),
                                dict(precision=1, amg_gs_levels=1), dict(precision=1, schur=1),
                                dict(precision=1, reorth=2.0, amg_coarse_max=16)])
def test_small_preconditioner_and_arnoldi_step(grid, wells, kw):
    prob = small(*grid, wells=wells)
    state = interior(prob, 3)
    its, r = few(prob, 5, kw, state)
    its0, r0 = few(prob, 5, dict(kw, cluster_rows=-1), state)
    assert its == its0
    # FP64: rounding; FP32 preconditioner: its 24 bits, through five iterations
    # (a residual at the floor of the system's conditioning agrees in size only)
    tol = 1e-6 if not kw.get("precision") else 1e-2
    assert abs(r - r0) <= tol * r0 + 1e-11
