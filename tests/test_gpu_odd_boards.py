"""Boards whose cells fill no whole eight-cell units, in buffers that start at any cell:
loads of aligned words shifted into place, stores a cell a lane or byte by byte, nothing
written beside the boards; single steps, rollouts and expansions against the oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import workload as wk
from tests.gpu_helpers import make, to_dev, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _at(n_cells, dtype, offset):
    """A device buffer of n_cells starting `offset` cells into a block, and the block."""
    block = torch.full((n_cells + offset + 8,), 0x55, dtype=dtype, device="cuda")
    return block[offset:offset + n_cells], block


def _untouched(block, n, offset):
    b = to_np(block)
    assert (b[:offset] == 0x55).all() and (b[offset + n:] == 0x55).all()


# 129 and 255 cells: one-byte boards past the line between the two ways of storing
@pytest.mark.parametrize("H,W", [(1, 1), (1, 3), (5, 5), (2, 3), (7, 9), (3, 43), (15, 17), (21, 23), (23, 41)])
@pytest.mark.parametrize("C", [4, 8, 12])
@pytest.mark.parametrize("offset", [0, 1, 3, 6])
def test_odd_boards(H, W, C, offset):
    import paper_2407_04221_gb300 as av
    B, F, steps, HW = 5, 2, 6, H * W
    wl = wk.WORKLOADS[3].scaled(batch=B, H=H, W=W, C=C, n_rules=5, shapes=((1, 1), (1, 2), (2, 2)), p_present=0.1,
                                p_absent=0.1, max_steps=4, border_wall=0)
    env, cfg, rules, cum = make(wl, 4)
    rng = np.random.default_rng(HW + C)
    g0 = rng.integers(0, 1 << C, size=(B, H, W)).astype(np.uint8 if C <= 8 else np.uint16)
    grids, _ = _at(B * HW, env.cell_dtype, offset)
    grids.copy_(to_dev(g0).flatten())
    t0 = np.zeros(B, np.int32)

    acts = rng.integers(0, 5, B).astype(np.uint8)
    env.set_state(grids, set_as_init=True)
    obs, block = _at(B * HW, env.cell_dtype, offset)
    rew = torch.zeros(B, dtype=torch.int32, device="cuda")
    av.av_step(env.h, to_dev(acts), obs, rew)
    eg, et, er, ed = oracle.step(cfg, rules, g0, g0, t0, acts)[:4]
    np.testing.assert_array_equal(to_np(obs).reshape(B, H, W), eg)
    np.testing.assert_array_equal(to_np(env.get_state()[0]), eg)
    _untouched(block, B * HW, offset)

    env.set_state(grids, set_as_init=True)
    traj, block = _at(steps * B * HW, env.cell_dtype, offset)
    av.av_rollout(env.h, steps, 9, traj)
    ref = oracle.rollout(cfg, rules, g0, g0, t0, steps, 9, trajectory=True)
    np.testing.assert_array_equal(to_np(traj).reshape(steps, B, H, W), ref["obs"])
    _untouched(block, steps * B * HW, offset)

    p = rng.integers(0, 1 << C, size=(B, F, H, W)).astype(g0.dtype)
    parents, _ = _at(B * F * HW, env.cell_dtype, offset)
    parents.copy_(to_dev(p).flatten())
    children, block = _at(B * F * 5 * HW, env.cell_dtype, offset)
    hashes = torch.zeros(B, F, 5, dtype=torch.int64, device="cuda")
    av.av_expand(env.h, parents, F, children, torch.zeros(B, F, 5, dtype=torch.int32, device="cuda"), None, hashes)
    ech, _, _, ehsh = oracle.expand(cfg, rules, p)
    np.testing.assert_array_equal(to_np(children).reshape(ech.shape), ech)
    np.testing.assert_array_equal(to_np(hashes, "hash"), ehsh)
    _untouched(block, B * F * 5 * HW, offset)
    env.close()
