"""What the library does with device memory: who may still be using what it frees, and what it
gives back.  Failures are made on the host by the library's allocation hook.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

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


def path(k, delta):
    return synth.Motif([(i, i + 1) for i in range(k)], delta)


def test_failed_batch_leaves_nothing_running(tmg):
    """A batch enumeration whose n-th allocation fails, for every n: when the call returns, none of its work is
    still on the stream (its caller frees the queries next), and later calls are exact."""
    g = synth.powerlaw_graph(100_000, 1_000_000, 77, span=9_460_800.0)
    mos = [path(4, 54_000), path(3, 7_200)]
    gg = tmg.Graph.from_synth(g)
    want = [gg.compile(mo).count() for mo in mos]
    gg.free()
    torch.cuda.synchronize()
    caps = [1000, 1000]
    failures = 0
    for after in range(64):
        gg = tmg.Graph.from_synth(g)              # a fresh graph has no batch buffers yet
        qs = [gg.compile(mo) for mo in mos]
        outs = [torch.full((c, mo.k), -9, dtype=torch.int32, device="cuda") for c, mo in zip(caps, mos)]
        torch.cuda.synchronize()
        tmg.inject_alloc_failure(after)
        try:
            got = gg.enumerate_batch(qs, outs)
        except tmg.TMError as e:
            assert torch.cuda.current_stream().query(), after
            tmg.inject_alloc_failure(-1)
            failures += 1
            assert e.status == tmg.E_OOM
            assert all(bool((o == -9).all()) for o in outs), after
            for q in qs:
                q.free()
            assert gg.compile(mos[1]).count() == want[1]
            gg.free()
            continue
        tmg.inject_alloc_failure(-1)
        assert got[1] == want
        gg.free()
        break
    # two queries' chunk buffers, then the count's and the fill's batch buffers
    assert 12 <= failures < 64


@pytest.mark.parametrize("on_device", [False, True])
def test_load_fails_at_every_allocation(tmg, on_device):
    """A load whose n-th allocation fails, for every n up to the one that succeeds: the status, nothing left on the
    stream, and an exact graph at the end."""
    m, n = 600_001, 5_000
    rng = np.random.default_rng(5)
    cols = [rng.integers(0, n, m).astype(np.int32), rng.integers(0, n, m).astype(np.int32),
            rng.integers(0, 1 << 40, m).astype(np.int64), rng.integers(0, 3, m).astype(np.uint8),
            rng.integers(0, 2, n).astype(np.uint8)]
    args = [torch.from_numpy(c).cuda() for c in cols] if on_device else cols
    for after in range(64):
        torch.cuda.synchronize()
        tmg.inject_alloc_failure(after)
        try:
            gg = tmg.Graph.load(n, *args)
        except tmg.TMError as e:
            assert torch.cuda.current_stream().query(), after
            assert e.status == tmg.E_OOM
            continue
        finally:
            tmg.inject_alloc_failure(-1)
        break
    assert (11 if on_device else 15) <= after < 64        # every buffer of the build was refused once
    assert np.array_equal(gg.edge_perm(), np.argsort(cols[2], kind="stable"))


def free_mb():
    return torch.cuda.mem_get_info()[0] >> 20


def load(tmg, m, seed=1):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    ends = [torch.randint(0, 100_000, (m,), device="cuda", generator=gen, dtype=torch.int32) for _ in range(2)]
    t = torch.randint(0, 1 << 30, (m,), device="cuda", generator=gen)
    torch.cuda.synchronize()
    return lambda: tmg.Graph.load(100_000, *ends, t)


def test_freed_memory_is_kept_and_given_back(tmg):
    """What the library's pool keeps after frees: something for the next load, whatever servers ran before and
    whatever graph is resident, at most 4 GiB, at once and without a synchronisation by the caller; and the
    device's default pool is left alone."""
    import ctypes
    rt = ctypes.CDLL("libcudart.so.13")
    pool, thr = ctypes.c_void_p(), ctypes.c_uint64(12_345)
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert rt.cudaMemPoolSetAttribute(pool, 4, ctypes.byref(thr)) == 0        # cudaMemPoolAttrReleaseThreshold
    small, big = load(tmg, 2_000_000), load(tmg, 40_000_000)

    def kept(fn):
        """MB held after fn() and a synchronisation that fn's graphs held, too."""
        g = fn()
        torch.cuda.synchronize()
        held = free_mb()
        g.free()
        torch.cuda.synchronize()
        return g.device_bytes >> 20, free_mb() - held

    mb, returned = kept(small)
    assert mb > 200 and returned <= 2
    g = small()
    srv = g.serve(mem_budget_bytes=1 << 20)
    srv.stop()
    g.free()
    mb, returned = kept(small)
    assert returned <= 2, "a server's small budget must not stay behind"
    g = big()
    assert g.device_bytes > 5 << 30
    mb, returned = kept(small)
    assert returned <= 2, "a large resident graph must not use up what is kept"
    torch.cuda.synchronize()
    before = free_mb()
    need = g.device_bytes >> 20
    g.free()
    after = free_mb()
    assert after - before >= need - 4096 - 320, "memory above the limit goes back when the graph is freed"
    g = big()
    srv = g.serve(mem_budget_bytes=12 << 30)
    srv.stop()
    g.free()
    assert free_mb() >= after - 320, "a server's large budget must not stay behind"
    thr.value = 0
    assert rt.cudaMemPoolGetAttribute(pool, 4, ctypes.byref(thr)) == 0 and thr.value == 12_345
    thr.value = 0
    rt.cudaMemPoolSetAttribute(pool, 4, ctypes.byref(thr))


def test_process_ends_with_everything_alive(tmp_path):
    """A program that ends without freeing its graph, queries, batch buffers and server ends in order."""
    code = """
import torch, synth, paper_2310_02800_gb300 as tmg
for c in (tmg.Graph, tmg.Query):
    c.free = lambda self: None
tmg.Server.stop = lambda self: None
g = synth.powerlaw_graph(2000, 20_000, 3, span=2e5)
keep = []
for _ in range(3):
    gg = tmg.Graph.from_synth(g)
    qs = [gg.compile(synth.cycle(k, 3600)) for k in (3, 4)]
    keep.append((gg, qs, gg.count_batch(qs), [q.count() for q in qs]))
    assert keep[-1][2] == keep[-1][3]
print("done", flush=True)
"""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, (r.returncode, r.stdout, r.stderr)


@pytest.mark.parametrize("m", [1, 5_000, 32_767, 32_768, 32_769, 60_000])
def test_permutation_of_few_edges(tmg, m):
    """Around the size from which ids are widened on the device: the permutation, and one that finds no device memory."""
    rng = np.random.default_rng(m)
    t = rng.integers(0, 1 + m // 3, m).astype(np.int64)
    gg = tmg.Graph.load(100, rng.integers(0, 100, m).astype(np.int32), rng.integers(0, 100, m).astype(np.int32), t)
    want = np.argsort(t, kind="stable")
    assert np.array_equal(gg.edge_perm(), want)
    tmg.inject_alloc_failure(0)
    assert np.array_equal(gg.edge_perm(), want)
    tmg.inject_alloc_failure(-1)
    assert np.array_equal(gg.edge_perm(), want)
