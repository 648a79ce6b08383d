"""`Env` calls given a stream run whole on it.  On the CPU, with torch's stream calls
and the library's entry points replaced by recorders: every allocation, fill, copy and
native call of such a call happens with that stream current, the search waits for the
caller's stream first, and arguments and results are marked for the stream they are
used on besides their own.  On the GPU: results of calls on a side stream, with the
caller's stream taking and overwriting memory at once, are those of the default stream."""
from __future__ import annotations

import contextlib

import numpy as np
import pytest

import workload as wk

torch = pytest.importorskip("torch")


class FakeStream:
    def __init__(self, handle, log):
        self.cuda_stream, self.log = handle, log

    def wait_stream(self, other):
        self.log.append(("wait", self.cuda_stream, other.cuda_stream))


@pytest.fixture
def recorded(monkeypatch):
    """An Env on the CPU and the log of (what, current stream's handle, ...)."""
    import paper_2407_04221_gb300 as av
    log, cur, capturing = [], [FakeStream(7, [])], set()
    cur[0].log = log

    @contextlib.contextmanager
    def stream(s):
        cur.append(s)
        yield
        cur.pop()

    monkeypatch.setattr(torch.cuda, "stream", stream)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: cur[-1])
    monkeypatch.setattr(torch.cuda, "ExternalStream", lambda h, dev=None: FakeStream(h, log))
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: cur[-1].cuda_stream in capturing)
    for name in ("empty", "zeros", "ones", "zeros_like"):
        real = getattr(torch, name)
        monkeypatch.setattr(torch, name, lambda *a, _r=real, _n=name, **k:
                            (log.append((_n, cur[-1].cuda_stream)), _r(*a, **k))[1])
    for name in ("copy_", "fill_", "contiguous", "clone"):
        real = getattr(torch.Tensor, name)
        monkeypatch.setattr(torch.Tensor, name, lambda t, *a, _r=real, _n=name, **k:
                            (log.append((_n, cur[-1].cuda_stream)), _r(t, *a, **k))[1])
    monkeypatch.setattr(torch.Tensor, "record_stream",
                        lambda t, s: log.append(("record", t.data_ptr(), s.cuda_stream)))
    for name in ("reset", "step", "rollout", "expand", "search_init", "select", "observe", "rule_obs", "get_state"):
        def native(*a, _n=name, stream=None, **k):
            log.append((_n, cur[-1].cuda_stream if stream is None else av._stream(stream)))
        monkeypatch.setattr(av, "av_" + name, native)
    monkeypatch.setattr(av, "av_create", lambda *a: None)
    wl = wk.WORKLOADS[4].scaled(batch=2)
    return av.Env(wk.config_fields(wl), None, device="cpu"), log, capturing


def _calls(env):
    grids = torch.zeros(2, 3, env.H, env.W, dtype=env.cell_dtype)
    n, roots = torch.ones(2, dtype=torch.int32), grids[:, 0].clone()
    return {
        "reset": lambda **k: env.reset(3, **k), "get_state": lambda **k: env.get_state(**k),
        "step": lambda **k: env.step(torch.tensor([1, 2], dtype=torch.uint8), **k),
        "rollout": lambda **k: env.rollout(4, 1, True, **k), "no_steps": lambda **k: env.rollout(0, 1, **k),
        "expand": lambda **k: env.expand(grids, **k), "expand_some": lambda **k: env.expand(grids, n, **k),
        "search": lambda **k: env.search(roots, 2, 3, **k), "observe": lambda **k: env.observe(5, **k),
        "rule_obs": lambda **k: env.rule_obs(**k),
    }


@pytest.mark.parametrize("name", ["reset", "get_state", "step", "rollout", "no_steps", "expand", "expand_some",
                                  "search", "observe", "rule_obs"])
@pytest.mark.parametrize("stream", [None, 7, 9, 0, 1])
def test_call_runs_whole_on_its_stream(recorded, name, stream):
    env, log, _ = recorded
    call = _calls(env)[name]
    del log[:]
    out = call(stream=stream)
    want = {None: 7, 1: 0}.get(stream, stream)
    outs = list(out.values()) if isinstance(out, dict) else list(out) if isinstance(out, tuple) else [out]
    work = [x for x in log if x[0] not in ("record", "wait")]
    assert {h for _, h in work} == {want}, log
    records = {x[1:] for x in log if x[0] == "record"}
    waits = [x for x in log if x[0] == "wait"]
    if want == 7:  # the current stream: nothing to mark or wait for
        assert not records and not waits
        return
    assert {(t.data_ptr(), 7) for t in outs if t is not None} <= records
    assert waits == ([("wait", want, 7)] if name == "search" else [])
    if name == "search":
        assert log[0][0] == "wait"
    if name in ("step", "expand", "expand_some", "search"):
        assert any(s == want for _, s in records)  # the arguments


def test_search_waits_only_within_one_capture(recorded):
    env, log, capturing = recorded
    for held, n in ((set(), 1), ({9}, 0), ({7}, 0), ({7, 9}, 1)):
        capturing.clear()
        capturing.update(held)
        del log[:]
        _calls(env)["search"](stream=9)
        assert len([x for x in log if x[0] == "wait"]) == n, held


def test_search_results_own_their_memory(recorded):
    """No result keeps the rows of every iteration alive."""
    env, _, _ = recorded
    for name, x in _calls(env)["search"]().items():
        assert x.untyped_storage().nbytes() == x.numel() * x.element_size(), name


@pytest.mark.gpu
def test_side_stream_results():
    """Memory of the caller's stream is taken and overwritten right after each call
    returns; the side stream is held back by queued work so that the calls are still
    to run then."""
    from tests.gpu_helpers import make, to_np
    wl = wk.WORKLOADS[4].scaled(batch=16)
    k, iters = 24, 8
    env, cfg, rules, cum = make(wl, 3, search_capacity=1 + k * iters)
    roots = env.reset(5)
    acts = torch.randint(5, (16,), dtype=torch.uint8, device="cuda")
    want_search = {n: to_np(x) for n, x in env.search(roots, iters, k).items()}
    state = env.get_state()
    want_step = [to_np(x) for x in env.step(acts)]
    ones = torch.ones(16, dtype=torch.int32, device="cuda")
    want_expand = [to_np(x) for x in env.expand(roots[:, None].contiguous(), ones)]
    want_roll = {n: to_np(x) for n, x in env.rollout(30, 2, trajectory=True).items()}
    env.set_state(*state)
    torch.cuda.synchronize()

    side = torch.cuda.Stream()
    load = torch.randn(4096, 4096, device="cuda")
    torch.cuda.synchronize()

    def held_back(call):
        with torch.cuda.stream(side):
            for _ in range(20):
                load @ load
        out = call()
        junk = [torch.full((1 << s,), 255, dtype=torch.uint8, device="cuda") for s in range(8, 23) for _ in range(6)]
        side.synchronize()
        torch.cuda.synchronize()
        del junk
        return out

    got = held_back(lambda: env.search(roots, iters, k, stream=side))
    for n, x in got.items():
        np.testing.assert_array_equal(to_np(x), want_search[n], err_msg=n)
    def ready(x):  # a temporary, made by the caller's stream
        x = x.clone()
        torch.cuda.current_stream().synchronize()
        return x

    got = held_back(lambda: env.step(ready(acts), stream=side.cuda_stream))
    for x, y in zip(got, want_step):
        np.testing.assert_array_equal(to_np(x), y)
    got = held_back(lambda: env.expand(ready(roots[:, None]), ready(ones), stream=side))
    for x, y in zip(got, want_expand):
        np.testing.assert_array_equal(to_np(x), y)
    got = held_back(lambda: env.rollout(30, 2, trajectory=True, stream=side))
    for n, x in got.items():
        np.testing.assert_array_equal(to_np(x), want_roll[n], err_msg=n)
    env.close()
