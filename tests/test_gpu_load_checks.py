"""fw_load_csr's checks: one defect at every place where the check kernels
change their code (inside a 16-byte quad, across two, across a row boundary, in
the last entries of arrays whose size is no multiple of 4)."""

import numpy as np
import pytest
import torch

from gpu_common import built, need_gpu

pytestmark = pytest.mark.gpu

LENS = (5, 0, 3, 1, 8, 1024, 0, 6)  # 1047 entries
N = 3000


def _graph():
    rng = np.random.default_rng(7)
    rp = np.concatenate([[0], np.cumsum(LENS)]).astype(np.int64)
    rp = np.concatenate([rp, np.full(N - len(LENS), rp[-1])])
    col = np.concatenate([np.sort(rng.choice(N, k, replace=False)) for k in LENS]).astype(np.int32)
    w = rng.uniform(1, 5, col.size).astype(np.float32)
    return rp, col, w, np.ones(col.size, dtype=np.int32)


def _load(rp, col, w, wu, **kw):
    need_gpu()
    built()
    from paper_2404_08364_gb300 import DeviceGraph
    return DeviceGraph.from_tensors(*(torch.from_numpy(x) for x in (rp, col, w, wu)), **kw)


def _status(*a, **kw):
    from paper_2404_08364_gb300 import _fw
    with pytest.raises(_fw.FwError) as e:
        _load(*a, **kw)
    return e.value.status


def test_descents_at_row_boundaries_are_fine():
    rp, col, w, wu = _graph()
    g = _load(rp, col, w, wu)
    assert g.info()["d_max"] == 1024 and g.info()["m"] == 1047
    # every row boundary a descent, an ascent, or equal values
    for last, first in ((2999, 0), (0, 2999), (1500, 1500)):
        c = col.copy()
        for b in rp[1:-1]:
            if 0 < b < c.size:
                c[b - 1], c[b] = last, first
        ok = all((np.diff(c[s:e]) > 0).all() for s, e in zip(rp[:-1], rp[1:]))
        if ok:
            _load(rp, c, w, wu)
        else:
            from paper_2404_08364_gb300 import _fw
            assert _status(rp, c, w, wu) == _fw.FW_EUNSORTED


@pytest.mark.parametrize("at", [0, 3, 9, 11, 15, 17, 500, 519, 1041, 1045])
@pytest.mark.parametrize("equal", [False, True])
def test_unsorted_pair_is_found(at, equal):
    from paper_2404_08364_gb300 import _fw
    rp, col, w, wu = _graph()
    row = np.searchsorted(rp, at, side="right") - 1
    assert rp[row] <= at and at + 1 < rp[row + 1]
    if equal:
        col[at] = col[at + 1]
    else:
        col[at], col[at + 1] = col[at + 1], col[at]
    assert _status(rp, col, w, wu) == _fw.FW_EUNSORTED
    _load(rp, col, w, wu, validate=False)


@pytest.mark.parametrize("at", [0, 7, 1043, 1044, 1046])
def test_bad_columns_and_weights_are_found(at):
    from paper_2404_08364_gb300 import _fw
    rp, col, w, wu = _graph()
    for bad in (-1, N, 2**31 - 1):
        c = col.copy()
        c[at] = bad
        assert _status(rp, c, w, wu, validate=False) == _fw.FW_EINVAL
    for bad in (0.0, -1.0, np.inf, np.nan):
        x = w.copy()
        x[at] = bad
        assert _status(rp, col, x, wu) == _fw.FW_EINVAL
    x = wu.copy()
    x[at] = 0
    assert _status(rp, col, w, x) == _fw.FW_EINVAL
    for k, v in ((0, 1), (3, 20), (len(rp) - 1, 1046)):
        r = rp.copy()
        r[k] = v
        assert _status(r, col, w, wu, validate=False) == _fw.FW_EINVAL


@pytest.mark.parametrize("drop", [0, 1, 2, 3])
def test_copied_arrays_walk_as_borrowed_ones(drop):
    """The arrays of a copied graph lie one behind the other: sizes with every
    remainder of 4 entries, from host and from device memory."""
    need_gpu()
    built()
    from paper_2404_08364_gb300 import DeviceGraph
    rp, col, w, wu = _graph()
    m = col.size - drop
    rp, col, w, wu = np.minimum(rp, m), col[:m], w[:m], np.arange(1, m + 1, dtype=np.int32)
    host = [torch.from_numpy(np.ascontiguousarray(x)) for x in (rp, col, w, wu, (np.arange(m) % 3).astype(np.int8))]
    dev = [x.cuda() for x in host]
    graphs = [DeviceGraph.from_tensors(*host), DeviceGraph.from_tensors(*dev), DeviceGraph.from_tensors(*dev, borrow=True)]
    starts = torch.arange(64, dtype=torch.int32).cuda() % 8
    for algo, mode in (("weighted", "fast"), ("weighted", "exact"), ("metapath", "fast"), ("metapath", "exact")):
        outs = [g.walk(algo, starts, 6, 5, mode=mode, schema=(0, 1, 2)) for g in graphs]
        for paths, plen in outs[1:]:
            assert torch.equal(paths, outs[0][0]) and torch.equal(plen, outs[0][1])
        assert int(outs[0][1].sum()) > 64  # (some walk moves)
