"""Expansion on boards of one or two long rows, whose tall rotations reach past a
plane's end in the packed table: terms on the last tile channels stay tile terms and
terms on the force stay force terms; against the oracle, bit-exact."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import workload as wk
from tests.gpu_helpers import make, to_dev, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,C", [(1, 243, 8), (243, 1, 8), (1, 256, 16), (2, 256, 10), (2, 208, 4), (1, 143, 5)])
@pytest.mark.parametrize("h,w", [(4, 1), (1, 5), (5, 2)])
def test_expand_long_rows(H, W, C, h, w):
    rng = np.random.default_rng(H + W + C)
    B, F = 3, 5
    wl = wk.WORKLOADS[3].scaled(batch=B, H=H, W=W, C=C, n_rules=3, border_wall=0)
    rules = np.zeros((B, 3), wk.RULE_DTYPE)
    rules["h"], rules["w"] = h, w
    rules["reward"] = [[1, 20, 300]]
    n = h * w
    rules["absent"][:, 0, :n] = 1 << (C - 1)         # the channel beside the force
    rules["absent"][:, 1, n - 1] = 1 << C            # the force, absent
    rules["present"][:, 2, 0] = (1 << C) | 1         # the force, present
    rules["clear"][:, 0, 0] = 4
    rules["set"][:, 1, n // 2] = 1 << (C - 1)
    rules["set"][:, 2, n - 1] = 8
    _, _, cum = wk.make(wl, 3)
    env, cfg, rules, cum = make(wl, 1, rules=rules, cum=cum)
    parents = rng.integers(0, 1 << C, size=(B, F, H, W)).astype(np.uint8 if C <= 8 else np.uint16)
    parents[:, ::2] &= ~np.array(1 << (C - 1), parents.dtype)  # half of them without the last channel
    parents[:, 1:, :, ::3] &= ~np.array(4, parents.dtype)
    ch, rew, done, hsh = env.expand(to_dev(parents))
    ech, erew, edone, ehsh = oracle.expand(cfg, rules, parents)
    np.testing.assert_array_equal(to_np(ch), ech)
    np.testing.assert_array_equal(to_np(rew), erew)
    np.testing.assert_array_equal(to_np(done), edone)
    np.testing.assert_array_equal(to_np(hsh, "hash"), ehsh)
    if min(h, w) <= min(H, W):  # the rules fit the board in some rotation
        assert (ech != parents[:, :, None]).any()
    env.sync()
    env.close()
