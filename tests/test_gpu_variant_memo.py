"""The memoising rollout's variant step at the edges of its rule bookkeeping (rules
past the first and second 32-bit word, two plane words per lane, two-byte cells,
limits below and above a rule's match count), with every number of warps per
environment, and with rules that match nearly everywhere (keys made cell by cell),
against the oracle, bit-exact."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import workload as wk
from tests.gpu_helpers import make, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R,H,W,C", [(1, 16, 16, 4), (17, 16, 16, 8), (33, 20, 21, 10), (64, 7, 9, 5),
                                     (64, 16, 32, 16)])
@pytest.mark.parametrize("random_keys", [0, 1])
def test_variant_step(R, H, W, C, random_keys):
    import paper_2407_04221_gb300 as av
    n, steps = 6, 25
    wl = wk.WORKLOADS[3].scaled(batch=n, H=H, W=W, C=C, n_rules=R, p_present=0.08, p_absent=0.05, max_steps=9)
    env, cfg, rules, cum = make(wl, 2)
    rng = np.random.default_rng(R)
    v = dict(random_keys=random_keys, key_seed=R + 5, limit=[int(x) for x in rng.choice([0, 1, 2, 40, 255], size=R)],
             inhibit=[int(rng.integers(0, 1 << 62)) & ((1 << R) - 1) if rng.random() < 0.1 else 0 for _ in range(R)])
    v["limit"][-1] = 1
    v["inhibit"][-1] |= 1
    av.av_set_variant(env.h, **v)
    assert av.av_rollout_path(env.h) == av.AV_PATH_VARIANT
    g0 = to_np(env.reset(3))
    res = env.rollout(steps, 11, trajectory=True)
    ref = oracle.rollout(cfg, rules, g0, g0, np.zeros(n, np.int32), steps, 11, trajectory=True,
                         variant=oracle.make_variant(**v))
    np.testing.assert_array_equal(to_np(res["obs"]), ref["obs"])
    np.testing.assert_array_equal(to_np(res["rew"]), ref["rew"])
    np.testing.assert_array_equal(to_np(res["done"]), ref["done"])
    env.close()


def _check(env, cfg, rules, v, steps, seed):
    import paper_2407_04221_gb300 as av
    av.av_set_variant(env.h, **v)
    assert av.av_rollout_path(env.h) == av.AV_PATH_VARIANT
    n = env.B
    g0 = to_np(env.reset(seed))
    res = env.rollout(steps, 11, trajectory=True)
    ref = oracle.rollout(cfg, rules, g0, g0, np.zeros(n, np.int32), steps, 11, trajectory=True,
                         variant=oracle.make_variant(**v))
    for name in ("obs", "rew", "done"):
        np.testing.assert_array_equal(to_np(res[name]), ref[name], err_msg=name)
    return ref


@pytest.mark.parametrize("warps", ["1", "2", "4", "8"])
@pytest.mark.parametrize("stage", ["0", "1"])
@pytest.mark.parametrize("R,H,W,C", [(1, 5, 5, 4), (3, 16, 16, 8), (33, 20, 21, 10)])
def test_warps_per_environment(R, H, W, C, warps, stage, monkeypatch):
    monkeypatch.setenv("AV_MEMO_WARPS", warps)
    monkeypatch.setenv("AV_MEMO_STAGE", stage)
    wl = wk.WORKLOADS[3].scaled(batch=5, H=H, W=W, C=C, n_rules=R, p_present=0.08, p_absent=0.05, max_steps=9)
    env, cfg, rules, cum = make(wl, 2)
    _check(env, cfg, rules, dict(random_keys=1, key_seed=3, limit=[1 + r % 3 for r in range(R)], inhibit=[0] * R), 40, 3)
    env.close()


@pytest.mark.parametrize("n,H,W,C,R", [(1200, 5, 5, 4, 2), (2200, 4, 6, 4, 1), (4300, 5, 4, 4, 2), (600, 16, 32, 4, 33)])
@pytest.mark.parametrize("steps", [3, 33])
def test_batches_past_the_lines_of_the_choice(n, H, W, C, R, steps):
    """Batches at which the library takes other numbers of warps for short and long
    rollouts, the last environments against the oracle."""
    import paper_2407_04221_gb300 as av
    wl = wk.WORKLOADS[3].scaled(batch=n, H=H, W=W, C=C, n_rules=R, p_present=0.08, p_absent=0.05, max_steps=9)
    env, cfg, rules, cum = make(wl, 2)
    v = dict(random_keys=1, key_seed=3, limit=[1] * R, inhibit=[0] * R)
    av.av_set_variant(env.h, **v)
    g0 = to_np(env.reset(3))
    res = env.rollout(steps, 11, trajectory=True)
    ids = np.array([0, 1, n // 2, n - 2, n - 1])
    ref = oracle.rollout(cfg, rules, g0[ids], g0[ids], np.zeros(len(ids), np.int32), steps, 11, trajectory=True,
                         env_ids=ids, variant=oracle.make_variant(**v))
    for name in ("obs", "rew", "done"):
        np.testing.assert_array_equal(to_np(res[name])[:, ids], ref[name], err_msg=name)
    env.close()


@pytest.mark.parametrize("H,W,C,R", [(16, 16, 8, 8), (7, 9, 4, 9), (16, 32, 16, 12), (20, 23, 5, 64), (1, 33, 4, 8),
                                     (5, 5, 8, 8)])
@pytest.mark.parametrize("limit", [1, 3, 40, 255])
@pytest.mark.parametrize("random_keys", [0, 1])
def test_rules_that_match_in_many_places(H, W, C, R, limit, random_keys):
    """Small patterns of nothing but a few absent entries match at most anchors of every
    rotation; some rules stay rare or unlimited beside them."""
    rng = np.random.default_rng(R + limit)
    n = 4
    rules = np.zeros((n, R), wk.RULE_DTYPE)
    for e in range(n):
        for r in range(R):
            x = rules[e, r]
            x["h"], x["w"] = [(1, 1), (1, 2), (2, 2), (1, 3)][int(rng.integers(4))]
            p = int(x["h"]) * int(x["w"])
            x["reward"] = int(rng.integers(-50, 50))
            x["absent"][:p] = rng.integers(0, 1 << (C + 1), p) & rng.integers(0, 1 << (C + 1), p) & rng.integers(0, 1 << (C + 1), p)
            if r % 4 == 3:
                x["present"][0] = 1 << int(rng.integers(C))
                x["absent"][0] &= ~x["present"][0]
            x["set"][:p] = rng.integers(0, 1 << C, p) & rng.integers(0, 1 << C, p)
            x["clear"][:p] = rng.integers(0, 1 << C, p)
    wl = wk.WORKLOADS[3].scaled(batch=n, H=H, W=W, C=C, n_rules=R, max_steps=7, border_wall=0)
    _, _, cum = wk.make(wl, 3)
    env, cfg, rules, cum = make(wl, 1, rules=rules, cum=cum)
    limits = [0 if r % 5 == 4 else limit for r in range(R)]
    ref = _check(env, cfg, rules, dict(random_keys=random_keys, key_seed=R, limit=limits, inhibit=[0] * R), 12, 5)
    assert (ref["rew"] != 0).any()
    env.close()
