"""Sizes at which the search's work splitting can go wrong, against the CPU oracle.

Whole numbers throughout: results are equal or wrong.
"""
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


def graph(n, m, span, seed, loops=True):
    rng = np.random.default_rng(seed)
    src = rng.integers(0, n, m).astype(np.int32)
    dst = rng.integers(0, n, m).astype(np.int32)
    if not loops:
        dst = np.where(dst == src, (dst + 1) % n, dst).astype(np.int32)
    t = rng.integers(0, span, m).astype(np.int64)
    el = rng.integers(0, 3, m).astype(np.uint8)
    nl = rng.integers(0, 2, n).astype(np.uint8)
    return n, src, dst, t, el, nl


MOTIFS = [
    synth.Motif([(0, 1)], 0), synth.Motif([(0, 1)], 5, elabel=[1]),
    synth.Motif([(0, 1), (1, 2)], 60), synth.Motif([(0, 1), (2, 3)], 40),
    synth.Motif([(0, 1), (1, 0), (0, 1)], 200), synth.cycle(3, 300), synth.Motif([(0, 1), (1, 2), (2, 0)], 300, [90, 200]),
    synth.out_star(3, 90), synth.in_star(3, 90), synth.Motif([(0, 1), (1, 2), (2, 3)], 120, elabel=[2, -1, 0]),
    synth.Motif([(0, 1), (1, 2), (2, 3), (3, 0)], 400, nlabel=[1, -1, 0, -1]),
    synth.Motif([(0, 1), (1, 2), (2, 0)], 300, anti=[(1, 0, 0, 100)]),
]


@pytest.mark.parametrize("m", [1, 2, 31, 32, 33, 63, 64, 65, 127, 129, 511, 2047, 5001])
def test_root_scan_edges(tmg, m):
    """Graphs around the 64-root scan step and the smallest chunks; root ranges that start and
    end on odd edges: totals, per-root counts and every row."""
    n, src, dst, t, el, nl = graph(max(3, min(24, m)), m, max(8, m * 2), seed=m)
    og = oracle.Graph(n, src, dst, t, el, nl)
    gg = tmg.Graph.load(n, src, dst, t, el, nl)
    for mo in MOTIFS:
        q = gg.compile(mo)
        want, want_pr = og.count(mo, per_root=True)
        pr = torch.full((m,), -1, dtype=torch.int64, device="cuda")
        assert q.count(per_root=pr) == want, mo
        assert np.array_equal(pr.cpu().numpy(), want_pr.astype(np.int64)), mo
        for a, b in ((0, m), (1, m), (m // 3, m - m // 5), (m // 2, m // 2), (m - 1, m)):
            part = torch.full((b - a,), -1, dtype=torch.int64, device="cuda")
            assert q.count_roots(a, b, per_root=part) == int(want_pr[a:b].sum()), (mo, a, b)
            assert np.array_equal(part.cpu().numpy(), want_pr[a:b].astype(np.int64)), (mo, a, b)
        rows = og.enumerate(mo, cap=want + 1)[0]
        out = torch.full((want + 1, mo.k), -7, dtype=torch.int32, device="cuda")
        assert q.enumerate(out)[:2] == (want, want), mo
        assert np.array_equal(out[:want].cpu().numpy(), rows), mo


@pytest.mark.parametrize("nq", [1, 7, 64])
def test_many_queries_on_a_small_graph(tmg, nq):
    """A batch whose warps switch queries with roots still buffered: totals of every batched form."""
    n, src, dst, t, el, nl = graph(30, 3001, 6000, seed=nq)
    og = oracle.Graph(n, src, dst, t, el, nl)
    gg = tmg.Graph.load(n, src, dst, t, el, nl)
    mos = [MOTIFS[(5 * j) % len(MOTIFS)] for j in range(nq)]
    qs = [gg.compile(mo) for mo in mos]
    want = [og.count(mo, per_root=True)[0] for mo in mos]
    assert gg.count_batch(qs) == want
    tot = torch.zeros(nq, dtype=torch.int64, device="cuda")
    assert gg.count_batch_noalloc(qs, tot).tolist() == want
    outs = [torch.full((max(1, w), mo.k), -7, dtype=torch.int32, device="cuda") for w, mo in zip(want, mos)]
    nw, tots, trunc = gg.enumerate_batch(qs, outs)
    assert tots == want and nw == want and not trunc
    for mo, w, o in zip(mos, want, outs):
        assert np.array_equal(o[:w].cpu().numpy(), og.enumerate(mo, cap=w + 1)[0]), mo


CHORDS = [
    synth.chorded_four_cycle(1000), synth.chorded_four_cycle(400),
    synth.Motif([(0, 1), (1, 2), (2, 3), (2, 0)], 1000),               # the new node sends the chord
    synth.Motif([(0, 1), (2, 1), (2, 3), (0, 2)], 700),                # the new node is found in an in-list
    synth.Motif([(0, 1), (1, 2), (2, 3), (3, 1), (0, 3)], 900),        # a chord node the previous edge does not touch
    synth.Motif([(0, 1), (1, 2), (2, 3), (0, 2)], 1000, [500, 1000, 1000], elabel=[-1, 1, -1, -1]),
    synth.Motif([(0, 1), (1, 2), (2, 3), (2, 0)], 1000, anti=[(1, 0, 0, 30)]),
]


@pytest.mark.parametrize("w", [1, 7, 31, 33, 64, 65, 255, 257, 1500])
def test_chord_filter_edges(tmg, w):
    """Chorded motifs where two hubs send w edges each into one window: candidate windows and filtered lists
    around the step sizes, the longest list that is filtered and windows long enough to be donated."""
    rng = np.random.default_rng(w)
    leaves = 4 + w // 8
    n = leaves + 2

    def leaf(k):
        return rng.integers(2, n, k)

    src = np.concatenate([np.repeat([0, 1], w), leaf(leaves), leaf(leaves), np.array([0, 1, 0, 1, 0])])
    dst = np.concatenate([leaf(2 * w), leaf(leaves), rng.integers(0, 2, leaves), np.array([1, 0, 1, 0, 0])])
    m = len(src)
    t = rng.integers(0, 1000, m).astype(np.int64)
    t[-5:] = rng.integers(0, 60, 5)
    el, nl = rng.integers(0, 3, m).astype(np.uint8), np.zeros(n, np.uint8)
    src, dst = src.astype(np.int32), dst.astype(np.int32)
    og = oracle.Graph(n, src, dst, t, el, nl)
    gg = tmg.Graph.load(n, src, dst, t, el, nl)
    for mo in CHORDS:
        q = gg.compile(mo)
        want, want_pr = og.count(mo, per_root=True)
        pr = torch.full((m,), -1, dtype=torch.int64, device="cuda")
        assert q.count(per_root=pr) == want, mo
        assert np.array_equal(pr.cpu().numpy(), want_pr.astype(np.int64)), mo
        rows = og.enumerate(mo, cap=min(want, 20_000) + 1)[0][: min(want, 20_000)]
        out = torch.full((max(1, len(rows)), mo.k), -7, dtype=torch.int32, device="cuda")
        assert q.enumerate(out)[:2] == (len(rows), want), mo
        assert np.array_equal(out[: len(rows)].cpu().numpy(), rows), mo


FANS = [
    synth.out_star(3, 1000), synth.in_star(3, 1000), synth.out_star(3, 300), synth.Motif([(0, 1), (1, 2), (1, 3)], 1000),
    synth.Motif([(0, 1), (2, 0), (3, 0)], 900), synth.Motif([(0, 1), (0, 2), (0, 3)], 1000, [1000, 50]),
    synth.Motif([(0, 1), (0, 2), (0, 3)], 1000, [50, 1000]), synth.Motif([(0, 1), (0, 2), (0, 3)], 1000, elabel=[-1, -1, 1]),
    synth.out_star(4, 1000),
]


@pytest.mark.parametrize("w", [2, 31, 32, 33, 63, 64, 65, 96, 255, 256, 257, 300])
def test_fan_window_edges(tmg, w):
    """Motifs whose last two edges leave (enter) one node, counted as pairs within a window of w entries: around
    the 32-lane steps and tiles and the longest window taken, with equal times and repeated neighbours, next to
    many one- and two-entry windows."""
    rng = np.random.default_rng(100 + w)
    n = 40 + w
    hub = np.zeros(w + 1, np.int64)
    leaf = rng.integers(1, 10 + w // 4, w + 1)
    few = rng.integers(1, n, 3 * n)
    src = np.concatenate([hub, leaf, few, rng.integers(0, n, 3 * n)]).astype(np.int32)
    dst = np.concatenate([leaf, hub, rng.integers(0, n, 3 * n), few]).astype(np.int32)
    m = len(src)
    t = np.concatenate([rng.integers(0, max(3, 2 * w // 3), 2 * (w + 1)), rng.integers(0, 20_000, m - 2 * (w + 1))]).astype(np.int64)
    t[: 2 * (w + 1)] *= 900 // max(3, 2 * w // 3)
    el, nl = rng.integers(0, 3, m).astype(np.uint8), np.zeros(n, np.uint8)
    og = oracle.Graph(n, src, dst, t, el, nl)
    gg = tmg.Graph.load(n, src, dst, t, el, nl)
    for mo in FANS[: 9 if w <= 65 else 8]:
        q = gg.compile(mo)
        want, want_pr = og.count(mo, per_root=True)
        pr = torch.full((m,), -1, dtype=torch.int64, device="cuda")
        assert q.count(per_root=pr) == want, mo
        assert np.array_equal(pr.cpu().numpy(), want_pr.astype(np.int64)), mo
        assert q.count() == want, mo
        rows = og.enumerate(mo, cap=5_000)[0]
        out = torch.full((5_000, mo.k), -7, dtype=torch.int32, device="cuda")
        assert q.enumerate(out)[:2] == (len(rows), want), mo
        assert np.array_equal(out[: len(rows)].cpu().numpy(), rows), mo


@pytest.mark.parametrize("chunks", [1, 4095, 4096, 4097, 16384, 16385])
def test_row_offsets_edges(tmg, chunks):
    """Enumerations whose chunk counts end around a round of the one-block offset scan and around its
    largest buffer: every row, and buffers that hold none, one, half and all but one of them."""
    m = 8 * chunks
    n, src, dst, t, el, nl = graph(max(4, min(50, m)), m, 4 * m, seed=chunks)
    og = oracle.Graph(n, src, dst, t, el, nl)
    gg = tmg.Graph.load(n, src, dst, t, el, nl)
    for mo in (synth.Motif([(0, 1), (1, 0)], 400), synth.out_star(2, 60)):
        q = gg.compile(mo)
        rows = og.enumerate(mo)[0]
        for cap in sorted({0, 1, len(rows) // 2, max(0, len(rows) - 1), len(rows) + 1}):
            out = torch.full((cap, mo.k), -7, dtype=torch.int32, device="cuda")
            w = min(cap, len(rows))
            assert q.enumerate(out) == (w, len(rows), len(rows) > cap), (mo, cap)
            assert np.array_equal(out[:w].cpu().numpy(), rows[:w]) and (out[w:] == -7).all(), (mo, cap)


@pytest.mark.parametrize("m", [8191, 8193, (1 << 19) - 1, 1 << 19, 1 << 20, (1 << 20) + 1, (1 << 20) + 8193])
@pytest.mark.parametrize("span", [1, 5_000, 1 << 40])
def test_load_edges(tmg, m, span):
    """Loads around the sort's tiles, its small inputs' end and the size from which host endpoints are copied beside
    the sort, with equal, 4-byte and 8-byte times: the same graph from host and device arrays, ids in stable
    time order, invalid endpoints refused, counts against the oracle."""
    n, src, dst, t, el, nl = graph(50_000, m, span, seed=m)
    gg = tmg.Graph.load(n, src, dst, t, el, nl)
    gd = tmg.Graph.load(n, *(torch.from_numpy(x).cuda() for x in (src, dst, t, el, nl)))
    want = np.argsort(t, kind="stable")
    assert np.array_equal(gg.edge_perm(), want) and np.array_equal(gd.edge_perm(), want)
    og = oracle.Graph(n, src, dst, t, el, nl)
    for mo in (synth.Motif([(0, 1), (1, 0)], span // 9, elabel=[1, -1]), synth.Motif([(0, 1), (1, 2)], span // 9, nlabel=[0, -1, 1])):
        want = og.count(mo)
        assert gg.compile(mo).count() == want and gd.compile(mo).count() == want, mo
    for bad in (-1, n):
        for col in (src, dst):
            keep, col[m - 1] = int(col[m - 1]), bad
            with pytest.raises(tmg.TMError):
                tmg.Graph.load(n, src, dst, t, el, nl)
            col[m - 1] = keep


@pytest.mark.parametrize("extra", [-1, 0, 1, 4096])
def test_edge_permutation_parts(tmg, extra):
    """The permutation is copied out 2^22 ids at a time: around that many, into memory nobody touched before."""
    m = (1 << 22) + extra
    n, src, dst, t, el, nl = graph(1000, m, 1 << 30, seed=m)
    assert np.array_equal(tmg.Graph.load(n, src, dst, t).edge_perm(), np.argsort(t, kind="stable"))
