"""What the walk library is measured on: the calls that its users make, from one
small batch on a graph that fits in L1 up to a large batch on a graph of 10^9
entries, in both modes, for every algorithm and every form (plain launch, mixed
launch, captured launch, host-output batches, served burst, graph reload, the
samplers).

Graphs come from `fw_inputs` (R-MAT and Chung-Lu, built on the GPU from the
seed).  Every output is a whole number (vertex ids, path lengths, sampled
indices).
"""

from __future__ import annotations

import math
from functools import lru_cache

import torch

import fw_inputs as fi
from paper_2404_08364_gb300 import DeviceGraph, Server, sample

ALGOS = ("weighted", "node2vec", "metapath", "ppr")


def listed():
    return [
        # The smallest whole workload: DeepWalk-style walks on a 1,000-vertex
        # graph, one query per vertex, exact mode.  Every array fits in L1/L2,
        # so the 80 dependent steps' latency and the call itself count.
        dict(name="tiny_weighted_exact", kind="walk", graph="chunglu", size=1000, weights="int5", algo="weighted",
             mode="exact", starts="each", n_q=1000, L=80, p=1.0, q=1.0, ragged=False, resume=False),
        # An online caller's mixed-length launch, captured once and replayed:
        # three small requests (weighted, node2vec, PPR) of odd sizes.  Far
        # fewer walks than the GPU has warps: the longest chain counts.
        dict(name="small_mix_replay", kind="replay", graph="rmat", size=20, weights="grid14", mode="fast",
             n_q=129, L=40, p=2.0, q=0.5),
        # node2vec p=2 q=0.5 on R-MAT-20 (rows of about 2,000 entries).
        dict(name="node2vec_rmat20", kind="walk", graph="rmat", size=20, weights="grid14", algo="node2vec", mode="fast",
             starts="spread", n_q=1 << 17, L=80, p=2.0, q=0.5, ragged=False, resume=False),
        # The headline: node2vec p=1 q=2 on R-MAT-25, 10^9 entries, rows of
        # about 10,000 entries and hubs of several 10^5.
        dict(name="node2vec_rmat25", kind="walk", graph="rmat", size=25, weights="grid14", algo="node2vec", mode="fast",
             starts="spread", n_q=1 << 18, L=80, p=1.0, q=2.0, ragged=False, resume=False),
        # First-order walks with ragged lengths on R-MAT-22.
        dict(name="weighted_rmat22_ragged", kind="walk", graph="rmat", size=22, weights="grid14", algo="weighted",
             mode="fast", starts="random", n_q=250007, L=80, p=1.0, q=1.0, ragged=True, resume=False),
        # MetaPath (5 labels, length 80) and PPR (stop 0.2, cap 100) on the
        # labelled R-MAT-22 graph, batched in one launch.
        dict(name="metapath_ppr_rmat22", kind="multi", graph="rmat", size=22, weights="grid14", mode="fast",
             n_q=1 << 17, L=80, p=1.0, q=1.0),
        # Personalised PageRank: every walk starts at the largest hub (a row
        # of about 160,000 entries).
        dict(name="ppr_from_hub_rmat22", kind="walk", graph="rmat", size=22, weights="grid14", algo="ppr", mode="fast",
             starts="hub", n_q=1 << 16, L=100, p=1.0, q=1.0, ragged=False, resume=False),
        # The reproducible mode on the same graph and rule as above: integer
        # weights, bit-exact against a CPU walker.
        dict(name="node2vec_rmat20_exact", kind="walk", graph="rmat", size=20, weights="grid14", algo="node2vec",
             mode="exact", starts="spread", n_q=1 << 15, L=80, p=2.0, q=0.5, ragged=False, resume=False),
        # Paths larger than the device budget: host starts in, host paths out,
        # eight batches on two streams.
        dict(name="node2vec_rmat20_batched", kind="batched", graph="rmat", size=20, weights="grid14", algo="node2vec",
             mode="fast", n_q=1 << 16, L=80, p=1.0, q=2.0, batches=8),
        # A served burst: 24 requests of log-uniform size, mixed algorithms
        # and lengths, through the request loop, results on the host.
        dict(name="served_burst_rmat22", kind="served", graph="rmat", size=22, weights="grid14", mode="fast",
             n_req=24, most=32768),
        # A changed graph: a new CSR snapshot is loaded (copied and checked),
        # walked once with a small batch and dropped.
        dict(name="reload_rmat22", kind="reload", graph="rmat", size=22, weights="grid14", algo="node2vec", mode="fast",
             n_q=4096, L=10, p=2.0, q=0.5),
        # The paper's ZPRS sampler over one weight array of 2,000 entries, at
        # warp width.
        dict(name="sampler_zprs_2000", kind="sample", method="zprs", n=2000, reps=1 << 18, width=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# The work of the largest listed case, in bytes: no drawn case exceeds it.
_MOST_BYTES = 0.9e12


def draw(rng):
    while True:
        kind = rng.choices(("walk", "multi", "replay", "batched", "served", "reload", "sample"), (8, 2, 2, 1, 1, 1, 2))[0]
        if kind == "sample":
            n = _log(rng, 1, 1 << 20)
            return dict(kind="sample", method=rng.choice(("expj", "dprs", "zprs")), n=n,
                        reps=min(_log(rng, 1 << 10, 1 << 20), max(16, (1 << 29) // n)), width=rng.choice((32, 256)))
        c = dict(kind=kind, graph="rmat", size=rng.randint(10, 24), weights=rng.choice(("grid14", "grid14", "int5", "lognormal1")))
        if kind == "walk" and rng.random() < 0.2:
            c.update(graph="chunglu", size=_log(rng, 200, 5000), weights="int5")
        c["mode"] = "exact" if c["weights"] != "lognormal1" and rng.random() < 0.3 else "fast"
        if kind == "served":
            c.update(size=min(c["size"], 22), n_req=rng.randint(1, 30), most=_log(rng, 64, 20000))
            return c
        c.update(n_q=_log(rng, 1, 1 << 18), L=_log(rng, 4, 100), p=rng.choice((0.5, 1.0, 2.0, 4.0)), q=rng.choice((0.25, 0.5, 1.0, 2.0)))
        if kind == "walk":
            c.update(algo=rng.choice(ALGOS), starts=rng.choice(("spread", "random", "hub")), ragged=rng.random() < 0.4,
                     resume=rng.random() < 0.2)
        if kind == "reload":
            c.update(algo=rng.choice(ALGOS[:2]), n_q=min(c["n_q"], 8191), L=min(c["L"], 20))
        if kind == "replay":
            c.update(n_q=min(c["n_q"], 2001))
        if kind == "batched":
            c.update(algo=rng.choice(ALGOS), batches=rng.randint(1, 12))
        if c["mode"] == "exact":
            c["n_q"] = max(1, c["n_q"] // 4)
        while c["n_q"] > 1 and work(c)["bytes"] * (3 if c["mode"] == "exact" else 1) > _MOST_BYTES:
            c["n_q"] = (c["n_q"] + 1) // 2
        return c


def _graph(case, seed, labels):
    dev = "cuda"
    if case["graph"] == "chunglu":
        return fi.chung_lu(n=case["size"], sum_theta=20.0 * case["size"], seed=seed, weights=case["weights"],
                           types_seed=seed + 1 if labels else None, device=dev)
    return fi.rmat(case["size"], seed=seed, weights=case["weights"], types_seed=seed + 1 if labels else None, device=dev)


def _starts(case, g, seed):
    how, n_q = case.get("starts", "random"), case["n_q"]
    if how == "hub":
        return torch.full((n_q,), int(g.degrees().argmax()), dtype=torch.int32, device="cuda")
    if how in ("each", "spread"):
        # one query per vertex, of about every (n / n_q)-th vertex (an odd
        # stride: R-MAT ids with many zero bits are hubs); more queries than
        # vertices go round
        i = torch.arange(n_q, dtype=torch.int64, device="cuda")
        return ((i * (g.n // n_q | 1)) % g.n).to(torch.int32)
    return fi.random_starts(g.n, n_q, seed, device="cuda")


def _neighbour(g, v, seed):
    """A neighbour of each v (v itself has none: -1), as a resumed walk holds."""
    d = g.degrees()[v.long()]
    h = fi.random_starts(1 << 30, v.numel(), seed, device="cuda").long()
    at = (g.row_ptr[v.long()] + h % d.clamp(min=1)).clamp(max=max(g.m - 1, 0))
    return torch.where(d > 0, g.col[at], torch.full_like(v, -1))


def _requests(case, g, seed):
    """The requests of a mixed launch: device starts, own seeds."""
    n, n_q, L, mode = g.n, case["n_q"], case["L"], case["mode"]
    if case["kind"] == "multi":
        sizes, algos = (n_q, n_q), ("metapath", "ppr")
    else:
        sizes, algos = (max(1, n_q // 16), max(1, n_q // 4), n_q), ("weighted", "node2vec", "ppr")
    return [dict(algo=a, starts=fi.random_starts(n, k, seed + 3 * i, device="cuda"), max_len=100 if a == "ppr" else L,
                 seed=seed + i, mode=mode, p=case["p"], q=case["q"], scale=4, ppr_stop=0.2)
            for i, (k, a) in enumerate(zip(sizes, algos))]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sample":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        return dict(kind=kind, method=case["method"], reps=case["reps"], width=case["width"], seed=seed,
                    w=1.0 + 4.0 * torch.rand(case["n"], generator=gen, device="cuda"))
    labels = kind == "multi" or case.get("algo") == "metapath"
    g = _graph(case, seed, labels)
    if kind == "reload":
        return dict(kind=kind, g=g, algo=case["algo"], starts=_starts(case, g, seed),
                    kw=dict(max_len=case["L"], seed=seed, mode=case["mode"], p=case["p"], q=case["q"], scale=4))
    dg = DeviceGraph.from_graph(g)
    if kind in ("multi", "replay"):
        reqs = _requests(case, g, seed)
        return dict(kind=kind, dg=dg, reqs=reqs, exec=dg.capture_multi(reqs) if kind == "replay" else None)
    if kind == "served":
        reqs = []
        for i in range(case["n_req"]):  # sizes log-uniform, lengths uniform in [10, 80], both well spread
            n_q = max(1, int(math.exp((i * 0.618034 + 0.4) % 1.0 * math.log(case["most"]))))
            reqs.append(dict(algo=("weighted", "node2vec", "ppr")[i % 3], starts=fi.random_starts(g.n, n_q, seed + i),
                             max_len=10 + int(71 * ((i * 0.754878 + 0.1) % 1.0)), seed=seed + i, p=2.0, q=0.5))
        return dict(kind=kind, dg=dg, reqs=reqs, mode=case["mode"])
    kw = dict(max_len=case["L"], seed=seed, mode=case["mode"], p=case["p"], q=case["q"], scale=4, ppr_stop=0.2)
    starts = _starts(case, g, seed)
    if kind == "batched":
        starts = starts.cpu().pin_memory()
        return dict(kind=kind, dg=dg, algo=case["algo"], starts=starts, kw=kw,
                    budget=2 * 4 * (case["L"] + 3) * -(-case["n_q"] // case["batches"]))
    if case["ragged"]:
        kw["lengths"] = fi.uniform_lengths(case["n_q"], 0, case["L"], seed, device="cuda")
    if case["resume"]:
        kw["prev"] = _neighbour(g, starts, seed)
        kw["step0"] = torch.full((case["n_q"],), 1, dtype=torch.int32, device="cuda")
    return dict(kind=kind, dg=dg, algo=case["algo"], starts=starts, kw=kw)


def run(state):
    kind = state["kind"]
    if kind == "walk":
        return state["dg"].walk(state["algo"], state["starts"], **state["kw"])
    if kind == "multi":
        return state["dg"].walk_multi(state["reqs"])
    if kind == "replay":
        return state["exec"].launch()
    if kind == "batched":
        paths, plen, _ = state["dg"].walk_batched(state["algo"], state["starts"], budget_bytes=state["budget"], **state["kw"])
        return paths, plen
    if kind == "served":
        srv = Server(state["dg"], mode=state["mode"], mem_budget=1 << 28)
        tickets = [srv.submit(**r) for r in state["reqs"]]
        outs = [srv.result(t)[:2] for t in tickets]
        srv.close()
        return outs
    if kind == "reload":
        dg = DeviceGraph.from_graph(state["g"])
        outs = dg.walk(state["algo"], state["starts"], **state["kw"])
        dg.free()
        return outs
    return sample(state["method"], state["w"], state["reps"], seed=state["seed"], width=state["width"], timed=False)[0]


# ---------------------------------------------------------------- the work


@lru_cache(maxsize=None)
def _rows(graph, size):
    """Of a graph of this recipe: (mean row, mean row that a walk stands on,
    share of vertices with a row, entries, share of the rows that a walk stands
    on without one of five labels, longest row)."""
    if graph == "chunglu":
        th = [(i + 1.0) ** (-1.0 / 1.1) for i in range(size)]
        s = 20.0 * size / sum(th)
        th = [min(t * s, size - 1.0) for t in th]
        tot = sum(th)
        return tot / size, sum(t * t + t for t in th) / tot, sum(1.0 - math.exp(-t) for t in th) / size, tot, \
            sum(t * math.exp(-0.2 * t) for t in th) / tot, th[0]
    # R-MAT: a vertex with z zero bits meets one with n00 zeros and n11 ones in
    # common at the rate below; duplicates count once
    k, a, b, d = size, 0.57, 0.19, 0.05
    tot = sq = alive = bare = 0.0
    for z in range(k + 1):
        deg = 0.0
        for n00 in range(z + 1):
            for n11 in range(k - z + 1):
                lam = 2.0 * 16 * 2.0**k * a**n00 * b ** (k - n00 - n11) * d**n11
                deg += math.comb(z, n00) * math.comb(k - z, n11) * -math.expm1(-lam)
        c = math.comb(k, z)
        tot += c * deg
        sq += c * (deg * deg + deg)
        alive += c * -math.expm1(-deg)
        bare += c * deg * math.exp(-0.2 * deg)
    return tot / 2.0**k, sq / tot, alive / 2.0**k, tot, bare / tot, deg  # the last vertex, all zero bits, is the hub


def _walk_bytes(case, algo, n_q, L, ragged=False, hub=False):
    """The row entries of every move read once (node2vec: column and weight;
    MetaPath: weight and label; else the weight alone), the row offsets, the
    column of the pick, the start and the path."""
    mean, stood, alive, _, bare, top = _rows(case["graph"], case["size"])
    moves = L / 2.0 if ragged else float(L)
    if algo == "ppr":
        moves = (1.0 - 0.8 ** min(L, 100)) / 0.2 if not ragged else min(moves, 5.0)
    if algo == "metapath":  # a row without the wanted label ends the walk
        moves = min(moves, (1.0 - (1.0 - bare) ** moves) / bare)
    first = mean if not hub else top
    if not hub:
        n_q, idle = n_q * alive, n_q * (1 - alive)
    else:
        idle = 0.0
    per = {"node2vec": 8.0, "metapath": 5.0}.get(algo, 4.0)
    entries = n_q * (first + max(0.0, moves - 1.0) * stood)
    return per * entries + n_q * moves * 20.0 + (n_q + idle) * (4.0 * (L + 1) + 28.0)


def work(case):
    kind = case["kind"]
    if kind == "sample":
        return {"bytes": 4.0 * case["n"] + 4.0 * case["reps"], "flops": 2.0 * case["n"] * case["reps"]}
    if kind == "multi":
        b = _walk_bytes(case, "metapath", case["n_q"], case["L"]) + _walk_bytes(case, "ppr", case["n_q"], 100)
    elif kind == "replay":
        n_q = case["n_q"]
        b = (_walk_bytes(case, "weighted", max(1, n_q // 16), case["L"]) + _walk_bytes(case, "node2vec", max(1, n_q // 4), case["L"])
             + _walk_bytes(case, "ppr", n_q, 100))
    elif kind == "served":
        most = case["most"]
        each = (most - 1) / max(1e-9, math.log(most))
        b = case["n_req"] / 3.0 * (sum(_walk_bytes(case, a, each, 45) for a in ("weighted", "node2vec", "ppr")))
    else:
        b = _walk_bytes(case, case["algo"], case["n_q"], case["L"], case.get("ragged", False), case.get("starts") == "hub")
        if kind == "reload":  # every array is read and written once
            m = _rows(case["graph"], case["size"])[3]
            n = case["size"] if case["graph"] == "chunglu" else 2.0 ** case["size"]
            b += 2.0 * (12.0 * m + 8.0 * n)
    return {"bytes": b, "flops": 0.0}
