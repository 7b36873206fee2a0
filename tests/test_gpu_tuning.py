"""Tuned queries on small graphs, where the default chunk size follows the input."""
import statistics

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


def kernel_us(q, n=80):
    q.profile(True)
    got = []
    for _ in range(n):
        q.count()
        got.append(q.last_ms()[0] * 1e3)
    return statistics.median(got)


def within(fn, bound):
    """Whether one of three timings is within the bound (one alone may be disturbed)."""
    return any(fn() < bound for _ in range(3))


@pytest.mark.parametrize("m", [20_000, 77_000])
def test_tuning_keeps_what_the_default_gives(tmg, m):
    """4-edge out-stars, whose small chunks make them 1.5 to 3 times as fast here: the tuner times the default and
    keeps it unless another setting is faster, and setting back what was read changes nothing (a quarter
    allowed for the clock)."""
    g = synth.powerlaw_graph(m // 10, m, 5, span=9.46 * m)
    gg = tmg.Graph.from_synth(g)
    mo = synth.out_star(4, 3600)
    want = oracle.Graph.from_synth(g).count(mo)
    q = gg.compile(mo)
    assert q.count() == want
    default = kernel_us(q)
    q.set_tuning(**q.tuning.as_dict())
    assert within(lambda: kernel_us(q), 1.25 * default)
    q.set_tuning(**{**q.tuning.as_dict(), "chunk_roots": 256})
    assert q.count() == want and q.tuning.chunk_roots == 256
    q = gg.compile(mo)
    q.autotune()
    assert q.count() == want
    assert within(lambda: kernel_us(q), 1.25 * default)
    assert within(lambda: kernel_us(gg.compile(mo)), 1.25 * default)          # the graph's cached choice
    # a query whose chunk size was set to something slower is tuned back
    q = gg.compile(mo)
    q.set_tuning(4, 256, 2, 512)
    q.autotune()
    assert within(lambda: kernel_us(q), 1.25 * default) and q.count() == want
