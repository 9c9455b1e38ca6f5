"""Which build of the engine a launch gets depends on the rules among its requests:
every set of rules in one launch gives each request's walks as alone."""

from itertools import combinations

import pytest
import torch

import fw_inputs as fi
from gpu_common import cached_graph, check_valid, device_graph

pytestmark = pytest.mark.gpu

ALGOS = ("weighted", "node2vec", "metapath", "ppr")


@pytest.mark.parametrize("n_q", [50, 9000])
@pytest.mark.parametrize("mode", ["exact", "fast"])
def test_every_set_of_rules_in_one_launch(mode, n_q):
    g = cached_graph("rmat", 14, 2)
    dg = device_graph(g)
    req = {a: dict(algo=a, starts=fi.random_starts(g.n, n_q + 7 * i, 5 + i, "cuda"), max_len=30, seed=11 + i, mode=mode,
                   p=2.0, q=0.5, ppr_stop=0.2) for i, a in enumerate(ALGOS)}
    alone = {a: dg.walk_multi([req[a]])[0] for a in ALGOS}
    for a in ALGOS:
        check_valid(g, *alone[a], a)
    assert int((alone["ppr"][1] - 1).sum()) < int((alone["weighted"][1] - 1).sum()) // 3  # the stop test is in
    for k in range(2, 5):
        for algos in combinations(ALGOS, k):
            for a, got in zip(algos, dg.walk_multi([req[a] for a in algos])):
                assert all(torch.equal(x, y) for x, y in zip(got, alone[a])), (algos, a)
