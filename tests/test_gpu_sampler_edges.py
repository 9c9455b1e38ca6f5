"""DPRS and ZPRS draw for draw against Alg. 3 and 4 in numpy (FP32 in the
kernels' summation order, Philox restated here), and the exponential-jump
reservoir's law, at the sizes where the samplers change their code: one element
per thread, few, groups of four, and their remainders; aligned and unaligned
weights."""

import numpy as np
import pytest
import torch

from gpu_common import built, chi2_tv, need_gpu

pytestmark = pytest.mark.gpu

SEED = 11


def _philox(c0, c1, c2, c3):
    """Philox-4x32-10 of counter arrays under key (SEED, 0): words [4, ...]."""
    m0, m1, w0, w1, lo = 0xD2511F53, 0xCD9E8D57, 0x9E3779B9, 0xBB67AE85, 0xFFFFFFFF
    x = [np.asarray(c, dtype=np.uint64) for c in np.broadcast_arrays(c0, c1, c2, c3)]
    k0, k1 = SEED, 0
    for _ in range(10):
        p0, p1 = x[0] * np.uint64(m0), x[2] * np.uint64(m1)
        x = [(p1 >> np.uint64(32)) ^ x[1] ^ np.uint64(k0), p1 & np.uint64(lo),
             (p0 >> np.uint64(32)) ^ x[3] ^ np.uint64(k1), p0 & np.uint64(lo)]
        k0, k1 = (k0 + w0) & lo, (k1 + w1) & lo
    return np.stack(x)


def _uniforms(r, k, iters):
    """u[i, j]: thread j's uniform of iteration i of draw r."""
    j, c = np.arange(k)[None, :], np.arange((iters + 3) // 4)[:, None]
    words = _philox(r, 0, j, c)                                    # [4, blocks, k]
    u = (words >> np.uint64(8)).astype(np.float32) * np.float32(2.0**-24)
    return u.transpose(1, 0, 2).reshape(-1, k)[:iters]


def _scan(v):
    """Inclusive prefix sums over k threads: shuffles inside a warp, then the
    earlier warps' totals added up in order."""
    v = v.astype(np.float32).reshape(-1, 32).copy()
    o = 1
    while o < 32:
        n = v.copy()
        n[:, o:] = v[:, o:] + v[:, :-o]
        v, o = n, 2 * o
    before = np.float32(0)
    out = []
    for row in v:
        out.append(row + before)
        before = np.float32(before + row[31])
    return np.concatenate(out)


def _draw(method, w, k, r):
    n = len(w)
    it = -(-n // k)
    x = np.zeros(it * k, np.float32)
    x[:n] = w
    x = x.reshape(it, k)
    u = _uniforms(r, k, it)
    with np.errstate(divide="ignore", invalid="ignore"):
        if method == "dprs":
            sel, wb = -1, np.float32(0)
            for i in range(it):
                s = _scan(x[i])
                hit = np.nonzero((x[i] > 0) & (u[i] < x[i] / (s + wb)))[0]
                if len(hit):
                    sel = i * k + hit[-1]
                wb = np.float32(wb + s[-1])
            return sel
        s = np.zeros(k, np.float32)
        for i in range(it):
            s = s + x[i]
        p = _scan(s) - s
        c = np.full(k, -1)
        for i in range(it):
            p = p + x[i]
            c = np.where((x[i] > 0) & (u[i] < x[i] / p), i * k + np.arange(k), c)
    top = np.nonzero(c >= 0)[0]
    return c[top[-1]] if len(top) else -1


def _weights(n, unaligned):
    gen = torch.Generator().manual_seed(n)
    w = 1.0 + 4.0 * torch.rand(n + 1, generator=gen)
    w[3::11] = 0.0
    if n > 8:
        w[7] = 1e-41  # denormal
        w[n // 2] = 900.0
    w = w.cuda()
    return w[1:] if unaligned else w[:n]


@pytest.mark.parametrize("method", ["dprs", "zprs"])
@pytest.mark.parametrize("width,n", [(32, 1), (32, 32), (32, 33), (32, 256), (32, 257), (32, 385), (32, 700),
                                     (256, 1), (256, 255), (256, 257), (256, 768), (256, 769), (256, 1025), (256, 2300)])
def test_draws_equal_the_algorithms(method, width, n):
    need_gpu()
    built()
    from paper_2404_08364_gb300 import sample
    w = _weights(n, n % 2 == 1)
    got, _ = sample(method, w, 96, seed=SEED, width=width)
    ref = [_draw(method, w.cpu().numpy(), width, r) for r in range(96)]
    assert got.cpu().tolist() == [int(x) for x in ref]


@pytest.mark.parametrize("width", [32, 256])
@pytest.mark.parametrize("n", [1, 127, 128, 129, 511, 513, 640, 641, 1153, 5000])
def test_reservoir_law(width, n):
    need_gpu()
    built()
    from paper_2404_08364_gb300 import sample
    w = _weights(n, n % 2 == 1)
    draws = 1 << 17
    got, _ = sample("expj", w, draws, seed=SEED, width=width)
    p = w.double().cpu().numpy()
    _, pv = chi2_tv(np.bincount(got.cpu().numpy(), minlength=n), p / p.sum(), draws)
    assert pv > 1e-6, (n, pv)


@pytest.mark.parametrize("width", [32, 256])
@pytest.mark.parametrize("n", [1, 2, 5, 64, 127, 128])
def test_short_reservoir_draws_as_the_general_one(width, n):
    """Zeros behind the weights are never drawn, but lead past the one-chunk kernel."""
    need_gpu()
    built()
    from paper_2404_08364_gb300 import sample
    w = _weights(n, n % 2 == 1)
    padded = torch.cat([w, torch.zeros((128 if width == 32 else 1024) + 1 - n, device=w.device)])
    a, _ = sample("expj", w, 4099, seed=SEED, width=width)
    b, _ = sample("expj", padded, 4099, seed=SEED, width=width)
    assert torch.equal(a, b)


@pytest.mark.parametrize("n", [1023, 1024, 1025])
def test_reservoir_law_where_segments_grow(n):
    test_reservoir_law(256, n)
