"""What a call leaves behind when it does not succeed."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def tmg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_02800_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("m", [60_000, 1_300_000])
def test_timed_out_count_writes_no_rows(tmg, m):
    """An enumeration whose count pass runs out of a bounded wait (one-block and long offset scans): the status, the
    row buffer as it was, and an exact next call."""
    g = synth.powerlaw_graph(m // 15, m, 313, span=9.46 * m / 8)
    gg = tmg.Graph.from_synth(g)
    mo = synth.cycle(3, 3600)
    q = gg.compile(mo)
    cap = 4096
    out = torch.full((cap, 3), -9, dtype=torch.int32, device="cuda")
    q.inject_fault(1)
    with pytest.raises(tmg.TMError) as e:
        q.enumerate(out)
    assert e.value.status == tmg.E_TIMEOUT
    assert bool((out == -9).all())
    rows, total = oracle.Graph.from_synth(g).enumerate(mo, cap=cap)
    assert q.enumerate(out) == (cap, total, True) and total > cap
    assert np.array_equal(out.cpu().numpy(), rows)


def test_smallest_budget_of_a_served_enumeration(tmg):
    """A budget that holds a request's rows and its chunk counts at 64 roots a chunk admits it, also on a graph small
    enough for smaller chunks; one byte less does not."""
    m, cap = 77_000, 1000
    g = synth.powerlaw_graph(5000, m, 313, span=9e6)
    gg = tmg.Graph.from_synth(g)
    mo = synth.cycle(3, 3600)
    q = gg.compile(mo)
    rows, total = oracle.Graph.from_synth(g).enumerate(mo, cap=cap)
    nch = -(-m // 64)
    need = cap * 3 * 4 + (nch + 2) * 8 + nch * 4 + 256         # rows, counts and list, scan scratch
    srv = gg.serve(mem_budget_bytes=need - 1)
    with pytest.raises(tmg.TMError) as e:
        srv.submit(q, True, cap)
    assert e.value.status == tmg.E_ADMISSION
    srv.stop()
    srv = gg.serve(mem_budget_bytes=need)
    for _ in range(2):
        tk = srv.submit(q, True, cap)
        r = srv.wait(tk, 60_000)
        assert (r.total, r.n_written) == (total, len(rows))
        assert np.array_equal(srv.matches(r).cpu().numpy(), rows)
        srv.release(tk)
    srv.stop()


def test_failed_edge_permutation_leaves_its_array(tmg):
    """A permutation asked for while a blocking stream is being captured, which the legacy stream it runs on must not
    join: the CUDA error's status, the array as it was, and a right next call."""
    import ctypes
    rt = ctypes.CDLL("libcudart.so.13")
    n, m = 1000, 40_000                # above the few that are widened on the host
    rng = np.random.default_rng(2)
    t = rng.integers(0, 5000, m).astype(np.int64)
    gg = tmg.Graph.load(n, rng.integers(0, n, m).astype(np.int32), rng.integers(0, n, m).astype(np.int32), t)
    gg.edge_perm()
    torch.cuda.synchronize()
    st, graph = ctypes.c_void_p(), ctypes.c_void_p()
    assert rt.cudaStreamCreate(ctypes.byref(st)) == 0
    assert rt.cudaStreamBeginCapture(st, 2) == 0                   # cudaStreamCaptureModeRelaxed
    keep = 0x7777_7777_7777_7777
    out = np.full(m, keep, np.int64)
    status = tmg.lib().tm_graph_edge_perm(gg._h, out.ctypes.data)
    rt.cudaStreamEndCapture(st, ctypes.byref(graph))
    if graph.value:
        rt.cudaGraphDestroy(graph)
    rt.cudaStreamDestroy(st)
    rt.cudaGetLastError()
    assert status == tmg.E_CUDA
    assert (out == keep).all()
    assert np.array_equal(gg.edge_perm(), np.argsort(t, kind="stable"))


def test_failed_calls_leave_host_outputs(tmg):
    """Work counters after a timed-out wait, and the kernel times of a batch that runs out of memory."""
    import ctypes
    g = synth.powerlaw_graph(2_000, 30_000, 5, span=3e5)
    gg = tmg.Graph.from_synth(g)
    q = gg.compile(synth.cycle(3, 3600))
    w = tmg._Work()
    ctypes.memset(ctypes.byref(w), 0x55, ctypes.sizeof(w))
    q.inject_fault(1)
    assert tmg.lib().tm_query_work(gg._h, q._h, None, ctypes.byref(w)) == tmg.E_TIMEOUT
    assert bytes(w) == b"\x55" * ctypes.sizeof(w)
    assert q.work()["matches"] == q.count()
    ms = (ctypes.c_double * 2)(7.0, 7.0)
    q2 = gg.compile(synth.cycle(4, 3600))
    hs, caps = (ctypes.c_void_p * 2)(q._h.value, q2._h.value), (ctypes.c_uint64 * 2)(0, 0)
    nw, tot = (ctypes.c_uint64 * 2)(9, 9), (ctypes.c_uint64 * 2)(9, 9)
    bufs = (ctypes.c_void_p * 2)()
    args = (gg._h, hs, 2, None, bufs, caps, nw, tot, ms)
    tmg.inject_alloc_failure(0)
    assert tmg.lib().tm_enumerate_batch(*args) == tmg.E_OOM
    tmg.inject_alloc_failure(-1)
    assert list(ms) == [7.0, 7.0] and list(nw) == [9, 9] and list(tot) == [9, 9]
    assert tmg.lib().tm_enumerate_batch(*args) == tmg.E_TRUNCATED
    assert list(tot) == [q.count(), q2.count()] and list(nw) == [0, 0] and 0 < ms[0] < 1e3 and ms[1] == 0
