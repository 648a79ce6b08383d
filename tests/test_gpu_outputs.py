"""Output tensors that `Env` allocates: slots that no kernel writes read as
zero, whatever the memory held before."""
from __future__ import annotations

import numpy as np
import pytest

import workload as wk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _dirty(n_bytes: int):
    """Leave non-zero bytes in the allocator's free blocks of the sizes used here."""
    keep = [torch.full((n_bytes >> s,), 255, dtype=torch.uint8, device="cuda") for s in range(0, 12)]
    torch.cuda.synchronize()
    del keep


@pytest.mark.parametrize("C", [4, 11])
def test_unwritten_outputs_read_as_zero(C):
    import paper_2407_04221_gb300 as av
    wl = wk.WORKLOADS[4].scaled(batch=3, C=C)
    _, rules, cum = wk.make(wl, 0)
    env = av.Env(wk.config_fields(wl), rules, cum)
    roots = env.reset(5)
    _dirty(1 << 20)
    out = env.rollout(0, 1)
    assert not out["rew_sum"].cpu().numpy().any()
    F = 4
    parents = roots[:, None].expand(-1, F, -1, -1).contiguous()
    n_parent = torch.tensor([0, 2, F], dtype=torch.int32, device="cuda")
    full = [x.cpu().numpy() for x in env.expand(parents)]
    _dirty(1 << 20)
    part = [x.cpu().numpy() for x in env.expand(parents, n_parent)]
    for got, want in zip(part, full):
        for b, n in enumerate(n_parent.tolist()):
            np.testing.assert_array_equal(got[b, :n], want[b, :n])
            assert not got[b, n:].any()
    env.close()


def test_search_reads_nothing_it_did_not_write():
    """Frontiers that fill up from one board, in memory that held other bytes: every
    result, whole, as in zeroed memory."""
    import paper_2407_04221_gb300 as av
    wl = wk.WORKLOADS[4].scaled(batch=5)
    k, iters = 40, 6
    _, rules, cum = wk.make(wl, 0)
    outs = []
    for byte in (0, 255, 90):
        env = av.Env(wk.config_fields(wl), rules, cum, search_capacity=1 + k * iters)
        roots = env.reset(5)
        keep = [torch.full(((4 << 20) >> s,), byte, dtype=torch.uint8, device="cuda") for s in range(0, 17)]
        torch.cuda.synchronize()
        del keep
        outs.append({n: x.cpu().numpy() for n, x in env.search(roots, iters, k).items()})
        env.close()
    for other in outs[1:]:
        for n, x in outs[0].items():
            np.testing.assert_array_equal(other[n], x, err_msg=n)
