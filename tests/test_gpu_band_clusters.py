"""Boards over shared memory with one, two, four and eight CTAs per environment
(the count falls as the batch grows, and never exceeds the board's bands), against
the oracle on sampled environments, bit-exact."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import workload as wk
from tests.gpu_helpers import sample_envs, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,H,W", [(1, 128, 256), (608, 128, 256), (609, 128, 256), (1217, 128, 256),
                                       (2433, 128, 256), (609, 96, 70), (700, 70, 67)])
def test_ctas_per_environment(batch, H, W):
    import paper_2407_04221_gb300 as av
    wl = wk.WORKLOADS[2].scaled(batch=batch, H=H, W=W, C=5, n_rules=4, shapes=((1, 2), (3, 3)), p_present=0.06,
                                p_absent=0.04, rules_per_env=0, max_steps=5, auto_reset=1, base_game=True,
                                init="maze")
    _, rules, cum = wk.make(wl, 4)
    fields = wk.config_fields(wl)
    env = av.Env(fields, rules, cum)
    cfg = oracle.make_cfg(**fields)
    g0 = to_np(env.reset(9))
    res = env.rollout(13, 21, trajectory=True)
    g, t = (to_np(x) for x in env.get_state())
    ids = sample_envs(batch, min(batch, 5), seed=1)
    ref = oracle.rollout(cfg, rules, g0[ids], g0[ids], np.zeros(len(ids), np.int32), 13, 21, trajectory=True,
                         env_ids=ids)
    np.testing.assert_array_equal(to_np(res["obs"])[:, ids], ref["obs"])
    np.testing.assert_array_equal(to_np(res["rew"])[:, ids], ref["rew"])
    np.testing.assert_array_equal(to_np(res["done"])[:, ids], ref["done"])
    np.testing.assert_array_equal(g[ids], ref["grids"])
    np.testing.assert_array_equal(t[ids], ref["t"])
    env.close()
