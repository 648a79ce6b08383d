"""The block rollout on boards of one to four 32-word groups whose rules fire here
and there: matches few enough for the queue and many enough for the match planes,
windows and outputs that reach across groups, more rules than a chunk holds; against
the oracle, bit-exact."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import workload as wk
from tests.gpu_helpers import make, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,C,R,density", [(64, 64, 16, 12, 0.05), (64, 64, 5, 6, 0.12), (23, 41, 9, 10, 0.08),
                                             (16, 256, 8, 9, 0.07), (256, 16, 8, 9, 0.07), (33, 33, 4, 4, 0.15),
                                             (48, 64, 16, 40, 0.04)])
def test_matches_across_groups(H, W, C, R, density):
    import paper_2407_04221_gb300 as av
    n, steps = 5, 70
    wl = wk.WORKLOADS[5].scaled(batch=n, H=H, W=W, C=C, n_rules=R, shapes=((1, 2), (3, 3), (5, 5)), p_present=density,
                                p_absent=density / 2, max_steps=29, auto_reset=1, base_game=True, init="maze")
    env, cfg, rules, cum = make(wl, 6)
    assert av.av_rollout_path(env.h) == av.AV_PATH_BLOCK
    g0 = to_np(env.reset(8))
    res = env.rollout(steps, 3, trajectory=True)
    ref = oracle.rollout(cfg, rules, g0, g0, np.zeros(n, np.int32), steps, 3, trajectory=True)
    np.testing.assert_array_equal(to_np(res["obs"]), ref["obs"])
    np.testing.assert_array_equal(to_np(res["rew"]), ref["rew"])
    np.testing.assert_array_equal(to_np(res["done"]), ref["done"])
    moved = (ref["obs"][1:] != ref["obs"][:-1]).any(axis=(2, 3)).mean()
    assert moved > 0.2  # boards change on many steps
    env.close()


@pytest.mark.parametrize("H,W,C,R,shapes", [(23, 41, 4, 2, ((1, 2), (3, 3))), (23, 41, 12, 9, ((1, 2), (5, 5))),
                                            (40, 40, 8, 64, ((1, 2), (3, 3))), (45, 45, 16, 64, ((5, 5),)),
                                            (63, 65, 8, 5, ((1, 2), (3, 3)))])
def test_batches_of_more_than_one_wave(H, W, C, R, shapes):
    """Batches that take one more CTA per SM where shared memory allows it (with 64 rules
    of 5 x 5 the table is read where it lies), single steps and a rollout, the first and
    last environments against the oracle."""
    from tests.gpu_helpers import to_dev
    n, steps = 460, 9
    ids = np.array([0, 1, 455, 456, 458, 459])
    wl = wk.WORKLOADS[5].scaled(batch=n, H=H, W=W, C=C, n_rules=R, shapes=shapes, p_present=0.06, p_absent=0.05,
                                max_steps=5, auto_reset=1, base_game=True, init="maze")
    env, cfg, rules, cum = make(wl, 6)
    g0 = to_np(env.reset(8))
    res = env.rollout(steps, 3, trajectory=True)
    ref = oracle.rollout(cfg, rules, g0[ids], g0[ids], np.zeros(len(ids), np.int32), steps, 3, trajectory=True,
                         env_ids=ids)
    for name in ("obs", "rew", "done"):
        np.testing.assert_array_equal(to_np(res[name])[:, ids], ref[name], err_msg=name)
    g, t = [to_np(x) for x in env.get_state()]
    acts = np.random.default_rng(1).integers(0, 5, n).astype(np.uint8)
    obs, rew, done = [to_np(x) for x in env.step(to_dev(acts))]
    eg, et, er, ed = oracle.step(cfg, rules, g[ids], g0[ids], t[ids], acts[ids], env_ids=ids)
    np.testing.assert_array_equal(obs[ids], eg)
    np.testing.assert_array_equal(rew[ids], er)
    np.testing.assert_array_equal(done[ids], ed)
    env.close()
