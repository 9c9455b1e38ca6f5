"""A tuning that is read and set again leaves the launch as it was, and a tuner
that fails leaves the graph as it found it.  Seen by which sampler takes a row of
139,000 entries: by default its walk's own warp does in fast mode, unless a
warp is idle; a threshold set below it makes it a shared row for every walk."""

import pytest
import torch

from gpu_common import built, need_gpu
from test_gpu_hub_mix import HUB_ROWS, hub_graph

pytestmark = pytest.mark.gpu

N_Q = 40000


@pytest.fixture(scope="module")
def dg():
    need_gpu()
    built()
    from paper_2404_08364_gb300 import DeviceGraph
    n, row_ptr, col, w_f32, w_u32 = hub_graph()
    return DeviceGraph.from_tensors(row_ptr, col, w_f32, w_u32)


def _shared(dg):
    dg.stats_reset()
    starts = torch.full((N_Q,), len(HUB_ROWS) - 1, dtype=torch.int32, device="cuda")
    dg.walk("weighted", starts, 1, 3, mode="fast")
    st = dg.stats()
    assert st["steps"] == N_Q
    return st["block_steps"]


def test_reading_and_setting_the_default(dg):
    dg.set_tuning()
    t = dg.get_tuning()
    assert _shared(dg) < N_Q // 2
    dg.set_tuning(**t)
    assert dg.get_tuning() == t
    assert _shared(dg) < N_Q // 2


@pytest.mark.parametrize("tuning", [dict(d_warp=4096), dict(block_threads=128), dict(block_threads=512, slots=32),
                                    dict(slots=64), dict(ctas_per_sm=1), dict(block_threads=256, d_warp=1 << 20)])
def test_reading_and_setting_a_tuning(dg, tuning):
    dg.set_tuning(**tuning)
    t = dg.get_tuning()
    # (slots alone count per 512 threads: 64 are four per warp)
    assert all(t[k] == (v if k != "slots" or "block_threads" in tuning else t["block_threads"] // 32 * v // 16)
               for k, v in tuning.items())
    own = tuning.get("d_warp", 0) == 4096
    assert (_shared(dg) == N_Q) == own
    dg.set_tuning(**t)
    assert dg.get_tuning() == t
    assert (_shared(dg) == N_Q) == own


def test_a_failing_tuner_leaves_the_tuning(dg):
    from paper_2404_08364_gb300 import _fw
    _fw.lib().fw_autotune_clear_cache()
    dg.set_tuning()
    t = dg.get_tuning()
    # a start out of range: written as an empty path and reported by the counters
    starts = torch.full((100,), -5, dtype=torch.int32, device="cuda")
    with pytest.raises(Exception):
        dg.autotune([dict(algo="weighted", starts=starts, max_len=4, seed=1, mode="fast")], reps=1)
    assert dg.get_tuning() == t
    assert _shared(dg) < N_Q // 2
