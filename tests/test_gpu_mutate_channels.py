"""Mutation at every channel count (each has code of its own), at the edges of the
rates, with rules past the first 32 and with masks of few and of many map channels
(drawn one by one, or all together), against the oracle, bit for bit."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import workload as wk
from tests.gpu_helpers import to_dev, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ONE = 1 << 24


@pytest.mark.parametrize("C", range(1, 17))
@pytest.mark.parametrize("rate,R", [(1, 1), (ONE // 7, 33), (ONE - 1, 5), (ONE, 64)])
def test_every_channel_count(C, rate, R):
    import paper_2407_04221_gb300 as av
    B, H, W = 5, 9, 7
    wl = wk.WORKLOADS[5].scaled(batch=B, H=H, W=W, C=C, n_rules=R)
    rules = wk.make_rules(wl, C)
    maps = wk.random_grids(C, B, H, W, C)
    mut = dict(p_map=rate, map_channels=(1 << C) - 1, p_rule=rate, p_reward=rate, reward_min=-9, reward_max=7,
               mutable_rules=(1 << R) - 1)
    dm = to_dev(maps)
    dr = torch.from_numpy(rules.view(np.uint8).reshape(B, R, -1).copy()).cuda()
    av.av_mutate(B, H, W, C, R, mut, 1234 + rate, dm, dr)
    want_m, want_r = oracle.mutate(H, W, C, mut, 1234 + rate, maps, rules)
    np.testing.assert_array_equal(to_np(dm), want_m)
    assert dr.cpu().numpy().tobytes() == want_r.tobytes()


@pytest.mark.parametrize("C", [1, 2, 3, 4, 8, 9, 10, 16])
@pytest.mark.parametrize("rate", [1, ONE // 3, ONE])
def test_map_channel_masks(C, rate):
    """Every number of channels, lowest and highest ones, and bits past the last channel."""
    import paper_2407_04221_gb300 as av
    B, H, W = 5, 9, 7
    maps = wk.random_grids(C, B, H, W, C)
    for n in range(1, C + 1):
        for mask in {(1 << n) - 1, ((1 << n) - 1) << (C - n), (1 << (C - 1)) | ((1 << (n - 1)) - 1)}:
            mut = dict(p_map=rate, map_channels=mask | 0xffff0000, p_rule=0, p_reward=0, reward_min=0, reward_max=0,
                       mutable_rules=0)
            dm = to_dev(maps)
            av.av_mutate(B, H, W, C, 0, mut, 99 + n, dm)
            want, _ = oracle.mutate(H, W, C, mut, 99 + n, maps, None)
            np.testing.assert_array_equal(to_np(dm), want, err_msg=f"{mask:x}")
