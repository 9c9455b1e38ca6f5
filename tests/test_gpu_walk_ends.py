"""Walks that end after one or two moves, by the million: a walk's end and the
claim of the next query into its slot follow each other at once, so the row
offsets asked for by the last move must have landed before the next start's
are asked for.  On a graph larger than L2, so that the two come back out of
step.  Every move has to be an edge of the row the walk stands on, and sampled
queries equal the oracle's."""

import numpy as np
import pytest
import torch

import fw_inputs as fi
from gpu_common import cached_graph, check_valid, compare_sampled, device_graph, recount

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("algo,max_len,stop", [("ppr", 100, 0.9), ("ppr", 100, 1.0), ("weighted", 1, 0.2),
                                               ("node2vec", 2, 0.2), ("metapath", 1, 0.2)])
@pytest.mark.parametrize("mode", ["exact", "fast"])
def test_short_walks_follow_each_other(orc, algo, max_len, stop, mode):
    g = cached_graph("rmat", 22, 2)
    dg = device_graph(g)
    n_q = 1 << 20
    starts = fi.random_starts(g.n, n_q, 17, "cuda")
    prm = dict(p=2.0, q=0.5, ppr_stop=stop)
    paths, plen = dg.walk(algo, starts, max_len, 29, mode=mode, **prm)
    st = dg.stats()
    check_valid(g, paths, plen, algo)
    assert torch.equal(paths[:, 0], starts)
    assert st["walks"] == n_q
    assert (st["steps"], st["rows_scanned"]) == recount(g, paths, plen)
    if mode == "exact":
        idx = np.random.default_rng(2).choice(n_q, 100, replace=False)
        compare_sampled(orc, g, algo, starts.cpu(), max_len, 29, paths.cpu(), plen.cpu(), orc.Params(**prm), idx)
