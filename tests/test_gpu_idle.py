"""Idle warps that give up waiting for work, in a build where they do so at once."""
import pytest

import synth
from tests import variant

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_blocks_that_gave_up_waiting_are_not_counted_idle(tmp_path):
    """4-edge paths from chunks of 4096 roots, few enough that most warps are idle from the start: with nobody
    waiting any more, the busy warps keep their work (while idle blocks stayed counted, they filled the queue's
    262,144 slots), and the count is the same."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2310_02800_gb300 as tmg
    tmg.lib()
    g = synth.powerlaw_graph(100_000, 1_000_000, 77, span=9_460_800.0)
    mo = synth.Motif([(i, i + 1) for i in range(4)], 54_000)
    gg = tmg.Graph.from_synth(g)
    want = gg.compile(mo).count()
    gg.free()
    hasty = variant.load(tmp_path, "tmg_hasty", "TMG_WAIT_NS=1ull")
    gg = hasty.Graph.from_synth(g)
    q = gg.compile(mo)
    q.set_tuning(4, 4096, 2, 0)
    assert q.count() == want
    assert hasty.last_search_stats()["reserved"] < 50_000
    q.free()
    gg.free()
