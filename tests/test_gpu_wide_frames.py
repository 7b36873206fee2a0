"""Frames whose windows add up to more candidates than a flattened position counts: they are
searched through a part of their parents at a time.

The library is built once more here with parts of a few thousand candidates, so that small graphs
reach every form of it (counts, per-root counts, rows, work counters, donation, the candidate
filter, pairs) and can be compared with the CPU oracle; the library itself is run on windows
that together pass 2^32, against counts worked out from the edge list.
"""
import numpy as np
import pytest

import oracle
import synth
from tests import variant

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

PART = 4096                     # above the edges of every graph searched with it


@pytest.fixture(scope="module")
def tmg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_02800_gb300 as m
    m.lib()
    return m


@pytest.fixture(scope="module")
def small_parts(tmg, tmp_path_factory):
    """The binding over a library whose frames begin at most PART candidates at a time."""
    return variant.load(tmp_path_factory.mktemp("small_parts"), "tmg_small_parts", f"TMG_FRAME_MAX={PART}u")


def check(m, gg, og, mo, n_edges):
    want, want_pr, work = (*og.count(mo, per_root=True), og.count(mo, work=True)[1])
    q = gg.compile(mo)
    pr = torch.full((n_edges,), -1, dtype=torch.int64, device="cuda")
    assert q.count() == want, mo
    assert q.count(per_root=pr) == want, mo
    assert np.array_equal(pr.cpu().numpy(), want_pr.astype(np.int64)), mo
    rows = og.enumerate(mo, cap=6_000)[0]
    out = torch.full((6_000, mo.k), -7, dtype=torch.int32, device="cuda")
    assert q.enumerate(out)[:2] == (len(rows), want), mo
    assert np.array_equal(out[: len(rows)].cpu().numpy(), rows) and bool((out[len(rows):] == -7).all()), mo
    got = q.work()
    assert got["matches"] == want, mo
    chords = mo.k > 3 and any(e in ((2, 0), (2, 1), (0, 2), (0, 3)) for e in mo.edges[3:])
    if not chords and not mo.anti:
        assert got["entries"] == [int(x) for x in work["entries"]], mo
        assert got["nodes"] == [int(x) for x in work["nodes"]], mo
    for depth in range(1, mo.k):
        q.set_tuning(4, 32, depth, 0)             # donation from every level, of any size
        assert q.count() == want, (mo, depth)
    return want


def test_disconnected_edges_in_parts(small_parts):
    """FREE levels, whose windows are the rest of the edge list, first, last and between others."""
    m = 3_000
    rng = np.random.default_rng(1)
    n = 60
    src, dst = rng.integers(0, n, m).astype(np.int32), rng.integers(0, n, m).astype(np.int32)
    t = rng.integers(0, 4 * m, m).astype(np.int64)
    el, nl = rng.integers(0, 12, m).astype(np.uint8), rng.integers(0, 2, n).astype(np.uint8)
    og, gg = oracle.Graph(n, src, dst, t, el, nl), small_parts.Graph.load(n, src, dst, t, el, nl)
    M = synth.Motif
    for mo in (M([(0, 1), (2, 3)], 9_000), M([(0, 1), (2, 3)], 9_000, elabel=[3, 4]), M([(0, 1), (2, 3), (3, 4)], 9_000, elabel=[1, 2, 3]),
               M([(0, 1), (2, 3), (4, 5)], 6_000, elabel=[5, 6, 7]), M([(0, 1), (1, 2), (3, 4)], 1_500, [600, 1_500], elabel=[-1, 1, 2]),
               M([(0, 1), (2, 3), (3, 2)], 8_000, elabel=[1, -1, -1]), M([(0, 1), (2, 3)], 9_000, nlabel=[0, 1, 1, 0]),
               M([(0, 1), (2, 3), (2, 4), (2, 5)], 2_500, elabel=[1, 2, -1, -1]),
               M([(0, 1), (2, 3)], 9_000, elabel=[3, -1], anti=[(1, 0, 0, 500)])):
        check(small_parts, gg, og, mo, m)
    qs = [gg.compile(M([(0, 1), (2, 3)], 9_000, elabel=[j, j + 1])) for j in range(9)]
    want = [og.count(M([(0, 1), (2, 3)], 9_000, elabel=[j, j + 1])) for j in range(9)]
    assert gg.count_batch(qs) == want
    tot = torch.zeros(9, dtype=torch.int64, device="cuda")
    assert gg.count_batch_noalloc(qs, tot).tolist() == want


@pytest.mark.parametrize("w", [200, 1_500])
def test_hub_lists_in_parts(small_parts, w):
    """Two hubs that send w edges each into one window: extensions, closing edges, chords behind their filter, and
    fans with windows on both sides of the longest that is counted as pairs."""
    rng = np.random.default_rng(w)
    leaves = 4 + w // 8
    n = leaves + 2

    def leaf(k):
        return rng.integers(2, n, k)

    src = np.concatenate([np.repeat([0, 1], w), leaf(leaves), leaf(leaves), np.array([0, 1, 0, 1, 0])]).astype(np.int32)
    dst = np.concatenate([leaf(2 * w), leaf(leaves), rng.integers(0, 2, leaves), np.array([1, 0, 1, 0, 0])]).astype(np.int32)
    m = len(src)
    t = rng.integers(0, 1000, m).astype(np.int64)
    t[-5:] = rng.integers(0, 60, 5)
    el, nl = rng.integers(0, 3, m).astype(np.uint8), np.zeros(n, np.uint8)
    og, gg = oracle.Graph(n, src, dst, t, el, nl), small_parts.Graph.load(n, src, dst, t, el, nl)
    M = synth.Motif
    mos = [M([(0, 1), (0, 2)], 1000), M([(0, 1), (0, 2), (2, 3)], 1000), M([(0, 1), (1, 2), (2, 0)], 1000), M([(0, 1), (1, 0), (0, 1)], 1000),
           M([(0, 1), (1, 2), (2, 3), (2, 0)], 400), M([(0, 1), (2, 1), (2, 3), (0, 2)], 400), M([(0, 1), (0, 2), (2, 3), (2, 1)], 300),
           M([(0, 1), (1, 2), (2, 3), (2, 0)], 400, anti=[(1, 0, 0, 30)]), synth.out_star(3, 100), synth.out_star(3, 400)]
    seen = sum(check(small_parts, gg, og, mo, m) > 0 for mo in mos)
    assert seen >= 7


@pytest.fixture(scope="module")
def wide():
    """140M edges, in time order: 47 rare-label roots first (and 17 self-loops among them), so that one frame holds
    32 or 47 windows of nearly all edges, 4.5 to 6.6e9 candidates."""
    m, n = 140_000_000, 1_000_000
    gen = torch.Generator(device="cuda").manual_seed(3)
    src = torch.randint(0, n, (m,), device="cuda", generator=gen, dtype=torch.int32)
    dst = torch.randint(0, n, (m,), device="cuda", generator=gen, dtype=torch.int32)
    t = torch.arange(m, device="cuda", dtype=torch.int64) // 3
    t[:64] = 0
    t[64:] += 1
    el = torch.zeros(m, device="cuda", dtype=torch.uint8)
    el[:64] = 7
    dst[:64] = (src[:64] + 1) % n
    dst[10:27] = src[10:27]
    el[torch.randint(1000, m, (40,), device="cuda", generator=gen)] = 8
    yield n, m, src, dst, t, el
    torch.cuda.empty_cache()


def roots_of(src, dst):
    return [(int(u), int(v)) for u, v in zip(src[:64].tolist(), dst[:64].tolist()) if u != v]


def test_disconnected_edges_beyond_32_bits(tmg, wide):
    n, m, src, dst, t, el = wide
    gg = tmg.Graph.load(n, src, dst, t, el)
    delta = 46_000_000
    end = int((t <= delta).sum())
    s, d = src[64:end], dst[64:end]
    roots = roots_of(src, dst)
    loop = s == d
    want = [int((~(loop | (s == u) | (s == v) | (d == u) | (d == v))).sum()) for u, v in roots]
    q = gg.compile(tmg.make_motif([(0, 1), (2, 3)], delta, elabel=[7, -1]))
    pr = torch.full((m,), -1, dtype=torch.int64, device="cuda")
    assert q.count(per_root=pr) == sum(want)
    head = pr[:64].cpu().numpy()
    assert head[head > 0].tolist() == want and int(pr.sum()) == sum(want)
    del pr
    w = q.work()
    assert w["matches"] == sum(want) and w["nodes"][1] == len(roots) and w["entries"][1] == len(roots) * (end - 64)
    # a level below: the few edges of another label, extended
    delta = 2 * int(t[-1])
    hit = (el == 8).nonzero().squeeze(1)
    want = 0
    for j in hit.tolist():
        a, b, tj = int(src[j]), int(dst[j]), int(t[j])
        if a == b:
            continue
        out = dst[(src == b) & (t > tj)].cpu().numpy()
        for u, v in roots:
            if not {a, b} & {u, v}:
                want += int((~np.isin(out, [a, b, u, v])).sum())
    q = gg.compile(tmg.make_motif([(0, 1), (2, 3), (3, 4)], delta, elabel=[7, 8, -1]))
    assert want > 0 and q.count() == want
    gg.free()


def test_hub_beyond_32_bits(tmg, wide):
    n, m, _, dst, t, el = wide
    src = torch.zeros_like(dst)                   # one hub sends everything,
    dst = dst.clone()
    dst[:64] = torch.arange(64, device="cuda", dtype=torch.int32) + 1
    dst[10:27] = 0
    few = 3_000                                   # but for the last edges, among a few nodes
    gen = torch.Generator(device="cuda").manual_seed(4)
    for col in (src, dst):
        col[-few:] = torch.randint(1, 200, (few,), device="cuda", generator=gen, dtype=torch.int32)
    el = el.clone()
    el[64:] = 0
    gg = tmg.Graph.load(n, src, dst, t, el)
    roots = [v for u, v in roots_of(src, dst)]
    delta = 2 * int(t[-1])
    hub = dst[64:m - few]
    nonzero = int((hub != 0).sum())
    per = torch.bincount(hub.long(), minlength=n).cpu().numpy()
    want = sum(nonzero - int(per[v]) for v in roots)
    q = gg.compile(tmg.make_motif([(0, 1), (0, 2)], delta, elabel=[7, -1]))
    assert q.count() == want
    # the hub's partner sends to a third node, then to the root's: found by the chord's filter
    s, d, tt = src[-few:].cpu().numpy(), dst[-few:].cpu().numpy(), t[-few:].cpu().numpy()
    want = 0
    for v in roots:
        for j in np.nonzero((d == v) & (s != v))[0]:
            x = s[j]
            between = (s == x) & (tt < tt[j]) & ~np.isin(d, [0, v, x])
            want += int(between.sum()) * int(per[x])
    q = gg.compile(tmg.make_motif([(0, 1), (0, 2), (2, 3), (2, 1)], delta, elabel=[7, -1, -1, -1]))
    assert want > 0 and q.count() == want
    gg.free()
