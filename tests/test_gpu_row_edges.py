"""One-step laws of rows whose lengths sit at the edges of the kernels' tiles
(quads, 128-entry halves, 256-entry stages, 512-entry pairs, 1024-entry
chunks, 16384-entry segments), at many alignments, the last row ending at the
end of arrays whose size is no multiple of 16.

Fast mode: 2^16 draws per row against w_i / sum(w), chi-square p > 1e-6 (about
100 rows and rules in all, so a false alarm has a chance below 1e-4)."""

import numpy as np
import pytest
import torch

from gpu_common import built, chi2_tv, need_gpu

pytestmark = pytest.mark.gpu

LENS = (1, 2, 3, 15, 16, 17, 31, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 1537, 4101, 16383,
        16384, 16385, 20003)
N = 1 << 16
P_MIN = 1e-6


class _G:
    pass


def edge_graph(lens=LENS, n=60000, seed=3):
    """Vertex i < len(lens) has a sorted random row of lens[i] entries."""
    rng = np.random.default_rng(seed)
    g = _G()
    g.n = n
    cols = [np.sort(rng.choice(n, k, replace=False)) for k in lens]
    g.row_ptr = np.zeros(n + 1, dtype=np.int64)
    g.row_ptr[1:len(lens) + 1] = np.cumsum(lens)
    g.row_ptr[len(lens) + 1:] = g.row_ptr[len(lens)]
    g.col = np.concatenate(cols).astype(np.int32)
    g.m = g.col.size
    g.w_u32 = rng.integers(1, 1000, g.m).astype(np.uint32)
    g.w_f32 = g.w_u32.astype(np.float32)
    g.etype = rng.integers(0, 5, g.m).astype(np.int8)
    return g


def load(g):
    need_gpu()
    built()
    from paper_2404_08364_gb300 import DeviceGraph
    t = [torch.from_numpy(x) for x in (g.row_ptr, g.col, g.w_f32, g.w_u32.view(np.int32), g.etype)]
    return DeviceGraph.from_tensors(*t, borrow=True)


@pytest.mark.parametrize("algo", ["weighted", "metapath", "ppr"])
@pytest.mark.parametrize("d_warp", [0, 1024])
def test_fast_laws_at_tile_edges(algo, d_warp):
    g = edge_graph()
    assert g.m % 16 and g.m % 4
    dg = load(g)
    if d_warp:
        dg.set_tuning(d_warp=d_warp)  # the longer rows go to the CTA sampler
    starts = torch.arange(len(LENS), dtype=torch.int32, device="cuda").repeat_interleave(N)
    paths, plen = dg.walk(algo, starts, 1, 20240501 + d_warp, mode="fast", schema=(2,), ppr_stop=0.5)
    dg.stats()
    nxt = paths[:, 1].view(len(LENS), N).cpu().numpy()
    for i, d in enumerate(LENS):
        row = slice(int(g.row_ptr[i]), int(g.row_ptr[i + 1]))
        w = g.w_f32[row].astype(np.float64) * (g.etype[row] == 2 if algo == "metapath" else 1)
        if w.sum() == 0:
            assert (nxt[i] == -1).all(), d
            continue
        at = np.searchsorted(g.col[row], nxt[i])
        assert (at < d).all() and (g.col[row][at] == nxt[i]).all(), (algo, d)
        _, p = chi2_tv(np.bincount(at, minlength=d), w / w.sum(), N)
        assert p > P_MIN, (algo, d, p)


# node2vec: rows of prev that make every kind of window: none, a few values, a
# block, several blocks, one dense against the longest and the shortest chunk
PREV_LENS = (1, 40, 128, 700, 6000, 50000)


@pytest.mark.parametrize("d_warp", [0, 1024])
def test_fast_node2vec_laws_at_chunk_edges(orc, d_warp):
    g = edge_graph(LENS + PREV_LENS)
    dg = load(g)
    if d_warp:
        dg.set_tuning(d_warp=d_warp)
    csr = orc.CSR(g)
    prm = orc.Params(p=4.0, q=3.0, scale=12)
    pairs = [(i, len(LENS) + j) for i in range(len(LENS)) for j in range(len(PREV_LENS))]
    # prev itself among cur's entries, so that the return factor is met
    for i, (cur, pv) in enumerate(pairs):
        row = g.col[g.row_ptr[cur]:g.row_ptr[cur + 1]]
        if i % 2:
            pairs[i] = (cur, int(row[len(row) // 2]) if g.row_ptr[row[len(row) // 2] + 1] > g.row_ptr[row[len(row) // 2]] else pv)
    n = N // 4
    cur = torch.tensor([a for a, _ in pairs], dtype=torch.int32, device="cuda").repeat_interleave(n)
    prev = torch.tensor([b for _, b in pairs], dtype=torch.int32, device="cuda").repeat_interleave(n)
    paths, plen = dg.walk("node2vec", cur, 2, 20240502 + d_warp, mode="fast", p=4.0, q=3.0, prev=prev,
                          step0=torch.ones_like(cur))
    dg.stats()
    nxt = paths[:, 1].view(len(pairs), n).cpu().numpy()
    for i, (c, b) in enumerate(pairs):
        row = g.col[g.row_ptr[c]:g.row_ptr[c + 1]]
        law = orc.transition(csr, "node2vec", prm, c, b, 1, mode="fast")
        at = np.searchsorted(row, nxt[i])
        assert (at < len(row)).all() and (row[at] == nxt[i]).all(), (c, b)
        _, p = chi2_tv(np.bincount(at, minlength=len(row)), law / law.sum(), n)
        assert p > P_MIN, (len(row), b, p)


@pytest.mark.parametrize("algo", ["weighted", "node2vec", "metapath", "ppr"])
@pytest.mark.parametrize("d_warp", [0, 1024])
def test_exact_picks_at_tile_edges(orc, algo, d_warp):
    """Exact mode on the same rows (and one of 40,000 entries, which is summed
    in runs of two pairs): bit-equal to the oracle."""
    g = edge_graph(LENS + PREV_LENS + (40000,))
    dg = load(g)
    if d_warp:
        dg.set_tuning(d_warp=d_warp)
    rows = len(LENS) + len(PREV_LENS) + 1
    starts = torch.arange(rows, dtype=torch.int32).repeat_interleave(96)
    kw = {}
    if algo == "node2vec":
        # prev goes over all rows too, and every third walk over cur's own middle entry
        mid = torch.from_numpy(g.col)[torch.from_numpy(g.row_ptr[:rows] + np.diff(g.row_ptr[:rows + 1]) // 2)]
        i = torch.arange(starts.numel())
        kw["prev"] = torch.where(i % 3 == 0, mid[starts.long()], ((i * 7) % rows).to(torch.int32))
    prm = orc.Params(p=2.0, q=0.5, schema=(2, 4), ppr_stop=0.5)
    rp, rl = orc.walk_exact(orc.CSR(g), algo, prm, starts.numpy(), 2, 77, **{k: v.numpy() for k, v in kw.items()})
    paths, plen = dg.walk(algo, starts.cuda(), 2, 77, mode="exact", p=2.0, q=0.5, schema=(2, 4), ppr_stop=0.5,
                          **{k: v.cuda() for k, v in kw.items()})
    dg.stats()
    assert np.array_equal(plen.cpu().numpy(), rl)
    assert np.array_equal(paths.cpu().numpy(), rp)


@pytest.mark.parametrize("mode", ["fast", "exact"])
@pytest.mark.parametrize("algo", ["weighted", "node2vec", "metapath", "ppr"])
def test_few_walks_equal_the_same_walks_in_a_large_batch(mode, algo):
    """Launches of 1, 37 and 200 walks (one walk per warp, helper warps, hub
    rows from one segment on) against the same queries of a full batch."""
    import fw_inputs as fi
    from gpu_common import cached_graph, device_graph
    g = cached_graph("rmat", 18, 2)
    dg = device_graph(g)
    assert dg.info()["d_max"] > 16384
    starts = fi.random_starts(g.n, 20000, 5, "cuda")
    starts[:5] = int((g.row_ptr[1:] - g.row_ptr[:-1]).argmax())
    kw = dict(max_len=12, seed=9, mode=mode, p=2.0, q=0.5)
    paths, plen = dg.walk(algo, starts, **kw)
    for q0, n in ((0, 1), (0, 37), (3, 200)):
        p, l = dg.walk(algo, starts[q0:q0 + n].clone(), q_id0=q0, **kw)
        dg.stats()
        assert torch.equal(l, plen[q0:q0 + n]) and torch.equal(p, paths[q0:q0 + n]), (q0, n)
