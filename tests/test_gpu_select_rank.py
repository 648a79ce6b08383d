"""av_select ranks few distinct candidates by counting and sorts many: the result is
av_select_static's (which sorts) at both sides of the boundary, with ties in the
cumulative reward, equal hashes, visited states and the hash 0."""
from __future__ import annotations

import numpy as np
import pytest

import workload as wk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("distinct,F,k", [(1, 1, 1), (3, 1, 5), (255, 100, 64), (256, 100, 256), (257, 100, 300),
                                          (600, 200, 256), (2000, 819, 700)])
def test_select_matches_sorted_select(distinct, F, k):
    import paper_2407_04221_gb300 as av
    B, H, W, C = 3, 16, 16, 4
    nc, cap = 5 * F, 4096
    rng = np.random.default_rng(distinct)
    pool = rng.integers(1, 1 << 62, size=distinct, dtype=np.int64)
    pool[0] = 0
    hashes = pool[rng.integers(0, distinct, size=(B, nc))]
    hashes[:, :min(nc, distinct)] = pool[:min(nc, distinct)]  # as many of them as fit
    dev = "cuda"
    up = lambda x, dt: torch.from_numpy(np.ascontiguousarray(x)).to(dev, dt)  # noqa: E731
    boards = up(rng.integers(0, 16, size=(B, F, 5, H, W)), torch.uint8)
    n_parent = up(np.array([F, max(1, F - 1), F]), torch.int32)
    cum, live = up(rng.integers(-2, 3, size=(B, F)), torch.int32), up(rng.random((B, F)) < 0.95, torch.uint8)
    rew, done = up(rng.integers(-1, 2, size=(B, F, 5)), torch.int32), up(rng.random((B, F, 5)) < 0.3, torch.uint8)
    chash = up(hashes.reshape(B, F, 5), torch.int64)

    wl = wk.WORKLOADS[4].scaled(batch=B, C=C, n_rules=2)
    _, rules, cumt = wk.make(wl, 0)
    env = av.Env(wk.config_fields(wl), rules, cumt, search_capacity=cap)
    roots = env.reset(1)
    rh, rl = torch.empty(B, dtype=torch.int64, device=dev), torch.empty(B, dtype=torch.uint8, device=dev)
    av.av_search_init(env.h, roots, rh, rl)
    visited = torch.zeros(B, cap, dtype=torch.int64, device=dev)
    visited[:, 0] = rh
    n_visited = torch.ones(B, dtype=torch.int32, device=dev)

    def outs():
        return (torch.zeros(B, k, H, W, dtype=torch.uint8, device=dev), torch.zeros(B, k, dtype=torch.int32, device=dev),
                torch.zeros(B, k, dtype=torch.int64, device=dev), torch.zeros(B, k, dtype=torch.uint8, device=dev),
                torch.zeros(B, dtype=torch.int32, device=dev))

    for call in range(2):  # the second finds the first's states visited
        a, b = outs(), outs()
        av.av_select(env.h, F, n_parent, cum, live, boards, rew, done, chash, k, *a)
        av.av_select_static(B, H, W, C, F, n_parent, cum, live, boards, rew, done, chash, k, *b, visited, n_visited, cap)
        for x, y in zip(a, b):
            np.testing.assert_array_equal(x.cpu().numpy(), y.cpu().numpy())
    env.sync()
    env.close()
