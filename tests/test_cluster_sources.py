"""Stores to another CTA's shared memory, checked in the CUDA sources.

A CTA of a cluster may touch another's shared memory only once that CTA is
known to have started: a kernel that does has arrived at and waited for a
cluster barrier before its first such access."""
import re

from test_pdl_sources import body_of, sources, stores

REMOTE = re.compile(r"map_shared_rank\s*\(|\bmapa\.")
BARRIER = re.compile(r"\bcl\.sync\(\)|\b(?:cl|small)_wait\(\)|barrier_wait\s*\(")


def functions(text):
    return re.findall(r"__global__[^;{]*?\b(k_\w+)\s*\(", text)


def unsynchronised(text):
    """Kernels of `text` whose first access to another CTA's shared memory
    comes before every cluster barrier of their body."""
    bad = []
    for k in sorted(set(functions(text))):
        body = body_of(text, k, "__global__") or ""
        m = REMOTE.search(body)
        if m and not BARRIER.search(body[:m.start()]):
            bad.append(k)
    return bad


def test_remote_shared_memory_after_a_cluster_barrier():
    text = sources()
    assert "k_orth_small" in functions(text) and "map_shared_rank" in text
    assert unsynchronised(text) == []
    # the phases of the coarse cycle wait before they store
    for f, store in (("gs_sweep_cl", ".put("), ("jacobi_pre_cl", ".put("), ("dense_mv_cl", ".put("),
                     ("csr_phase", "done(")):
        body = body_of(text, f, "__device__")
        assert 0 <= body.index("cl_wait()") < body.index(store), f


def test_the_check_catches_a_missing_barrier():
    src = """
__global__ void k_early(float *x) {
  __shared__ float p[8];
  *cl.map_shared_rank(&p[0], 1) = x[0];
  cl.sync();
}
__global__ void k_fine(float *x) {
  __shared__ float p[8];
  small_arrive();
  small_wait();
  *cl.map_shared_rank(&p[0], 1) = x[0];
  cl.sync();
}
"""
    assert unsynchronised(src) == ["k_early"]


def own_entry_stores(text):
    """Stores to a replicated vector whose value reads that vector in the same
    statement: the lanes of a row's group each store to some of the copies, so
    a lane may read an entry that another lane has already replaced."""
    return [m.group(0) for m in re.finditer(r"\b(\w+)\.put\s*\([^;]*?\b\1\.get\s*\([^;]*;", text)]


def test_replicated_entries_are_read_before_any_lane_stores():
    text = sources()
    assert own_entry_stores(text) == []
    # a row's own entry is read before the reduction, and the lanes meet between
    for f, read, store in (("csr_phase", "own(m.q)", "done("), ("gs_sweep_cl", "xi = x.get(i)", ".put(")):
        body = body_of(text, f, "__device__")
        assert body.index(read) < body.index("group_reduce") < body.index("__syncwarp()") < \
            body.index(store), f
    assert own_entry_stores("auto add = [&](int i) { x.put(i, x.get(i) + s, gl, pG, C); };")
    assert not own_entry_stores("t.put(i, b.get(i) - s, gl, G, C); x.put(i, o + s, gl, G, C);")


def test_cluster_kernels_launched_as_dependents_wait_before_they_store():
    """The kernels launched through cudaLaunchKernelEx as programmatic
    dependents, which the check of DP_LAUNCH_PDL's kernels does not see: they
    reach griddep_wait before any store, and let their own dependents in only
    after it."""
    text = sources()
    for k in ("k_coarse_cycle", "k_cpr_small", "k_orth_small"):
        body = body_of(text, k, "__global__")
        wait = body.index("griddep_wait()")
        assert wait < body.index("griddep_launch_dependents()"), k
        assert stores(body[:wait]) == [], k
