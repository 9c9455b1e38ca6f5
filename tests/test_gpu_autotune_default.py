"""The tuner times the default launch too: its rate is at least about the
default's (the margin is for the spread between two timings)."""

import pytest
import torch

import fw_inputs as fi
from gpu_common import cached_graph, device_graph

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("algo,mode", [("node2vec", "fast"), ("node2vec", "exact"), ("ppr", "fast")])
def test_tuned_rate_is_at_least_the_default_one(algo, mode):
    from paper_2404_08364_gb300 import _fw
    _fw.lib().fw_autotune_clear_cache()
    g = cached_graph("rmat", 14, 2)
    dg = device_graph(g)
    s = fi.random_starts(g.n, 20000, 5, "cuda")
    reqs = [dict(algo=algo, starts=s, max_len=40, seed=5, mode=mode, p=2.0, q=0.5)]
    rates = []
    for _ in range(5):
        dg.stats_reset()
        dg.walk_multi(reqs)
        st = dg.stats()
        rates.append(st["steps"] / (st["last_kernel_ms"] * 1e-3))
    t = dg.autotune(reqs, reps=5)
    assert t["steps_per_s"] > 0.7 * sorted(rates)[2]
    assert dg.get_tuning() == {k: t[k] for k in ("block_threads", "slots", "d_warp", "ctas_per_sm")}
    dg.set_tuning(**dg.get_tuning())
    assert dg.autotune(reqs, reps=5)["steps_per_s"] == 0.0  # kept
