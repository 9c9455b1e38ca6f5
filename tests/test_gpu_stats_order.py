"""fw_stats after launches whose stream is gone (a capture's, the tuner's) and
after replays: it waits for the last one and reports its counts."""

import pytest
import torch

import fw_inputs as fi
from gpu_common import cached_graph, device_graph, recount

pytestmark = pytest.mark.gpu


def _requests(g, n=4000):
    s = fi.random_starts(g.n, n, 3, "cuda")
    return [dict(algo="weighted", starts=s, max_len=30, seed=1, mode="fast"),
            dict(algo="ppr", starts=s.clone(), max_len=50, seed=2, mode="fast")]


def _expect(g, outs):
    each = [recount(g, p, l) for p, l in outs]
    return sum(e[0] for e in each), sum(e[1] for e in each)


def test_stats_after_a_capture_and_its_replays():
    g = cached_graph("rmat", 12, 2)
    dg = device_graph(g)
    reqs = _requests(g)
    ex = dg.capture_multi(reqs)
    assert dg.stats()["walks"] == 0
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for k in range(1, 6):
        outs = ex.launch(stream=side)
        st = dg.stats()  # waits for the replay
        steps, rows = _expect(g, outs)
        assert (st["walks"], st["steps"], st["rows_scanned"]) == (8000 * k, steps * k, rows * k)
    ex.close()
    dg.stats_reset()
    assert dg.stats()["steps"] == 0


def test_stats_after_autotune():
    from paper_2404_08364_gb300 import _fw
    g = cached_graph("rmat", 12, 2)
    dg = device_graph(g)
    reqs = _requests(g)
    _fw.lib().fw_autotune_clear_cache()
    dg.autotune(reqs, reps=1)
    assert dg.stats()["walks"] > 0
    dg.stats_reset()
    outs = dg.walk_multi(reqs)
    st = dg.stats()
    assert (st["steps"], st["rows_scanned"]) == _expect(g, outs)
