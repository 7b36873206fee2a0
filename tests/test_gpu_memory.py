"""What the library does with device memory: who may still be using what it frees, and what it
gives back.  Failures are made on the host by the library's allocation hook.
"""
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
