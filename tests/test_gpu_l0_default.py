"""The kernel of level 0's colour sweeps that a realisation starts with: the
pipelined one on the default stream and in a server of one worker, a thread
per row on a stream of its own, where other streams may share the GPU.  No call changes it but
sim_set_l0_kernel and sim_autotune, and the results do not depend on it."""
import numpy as np
import pytest

import dp_inputs as di

pytestmark = pytest.mark.gpu


def gpu():
    from paper_1808_04338_gb300 import dpsim
    return dpsim


def pipelined(sim, dt):
    """Launches of level 0's pipelined kernels in one timestep."""
    sim.time_kernel("_tma")
    sim.kernel_timing(reset=True)
    rc, _ = sim.advance(dt)
    _, n = sim.kernel_timing(reset=True)
    sim.time_kernel(None)
    assert rc == 0
    return n


def test_default_by_stream_and_kept_by_advance_many():
    d = gpu()
    prob = di.layered(45, 43, 8)          # 30960 rows: level 0 outside the cluster cycle
    streams = [d.OwnedStream() for _ in range(2)]
    sims = [d.Sim(prob, d.options("report", precision=1)) for _ in range(2)]
    sims += [d.Sim(prob, d.options("report", precision=1), stream=s.torch) for s in streams]
    first = [pipelined(s, prob.dt) for s in sims]
    assert first[0] > 0 and first[1] > 0 and first[2] == first[3] == 0
    states = [s.get_state() for s in sims]
    rc, _, _ = d.advance_many(sims, [prob.dt] * len(sims), threads=4)
    assert rc == 0
    assert [pipelined(s, prob.dt) > 0 for s in sims] == [True, True, False, False]
    states += [s.get_state() for s in sims]
    for k, st in enumerate(states):
        for a, b in zip(st, states[k // 4 * 4]):
            np.testing.assert_array_equal(a, b)
    for s in sims:
        s.close()
    for s in streams:
        s.close()
