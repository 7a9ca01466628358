"""Scratch that the time-domain calls allocate belongs to the stream they run on: calls on two streams with nothing
between them do not share a block."""

import contextlib

import numpy as np
import pytest
import torch

from paper_2309_08038_gb300 import ops


class _Lib:
    """Every entry succeeds; sizes are small and not zero."""

    def __getattr__(self, name):
        return lambda *a: 1024 if name.endswith("_bytes") and "fft" in name else 512 if name.endswith("_bytes") else 0


def test_scratch_comes_from_the_stream_of_the_call(monkeypatch):
    side, active, made = object(), [None], []

    @contextlib.contextmanager
    def stream(s):
        active.append(s)
        yield
        active.pop()

    empty = torch.empty
    monkeypatch.setattr(ops._lib, "load", lambda *a: _Lib())
    monkeypatch.setattr(ops, "require", lambda t, *a, **k: t)
    monkeypatch.setattr(ops, "check", lambda status: None)
    monkeypatch.setattr(ops, "stream_handle", lambda s=None: 0)
    monkeypatch.setattr(torch.cuda, "Stream", type(side))
    monkeypatch.setattr(torch.cuda, "stream", stream)
    monkeypatch.setattr(torch.Tensor, "record_stream", lambda t, s: None)
    radar = ops.Radar(77e9, 1e14, 1e-7, 8e-6, 0.25)
    raw, out = empty(64, 32, dtype=torch.complex64), empty(32, 64, dtype=torch.complex64)
    w, o = empty(32, 4, dtype=torch.complex64), torch.zeros(4, dtype=torch.int32)
    plan = ops.TimeDomainPlan(empty(1024, dtype=torch.uint8), 64, 32, 32, 4)
    monkeypatch.setattr(torch, "empty", lambda *a, **k: (made.append(active[-1]), empty(*a, **k))[1])
    calls = [lambda **k: ops.bpa_time(raw, None, radar, 32, 4, out=out, transforms=True, **k),
             lambda **k: ops.sas_time(raw, None, w, o, radar, out=out, transforms=True, **k),
             lambda **k: ops.sas_time_planned(raw, plan, out=out, **k),
             lambda **k: ops.bpa_time_planned(raw, plan, out=out, **k)]
    for call in calls:
        made.clear()
        call()
        assert made and all(s is None for s in made)
        made.clear()
        call(stream=side)
        assert made and all(s is side for s in made)


@pytest.mark.gpu
def test_calls_on_two_streams_do_not_share_scratch():
    import synth
    from paper_2309_08038_gb300 import build
    build.build()
    import paper_2309_08038_gb300 as rosar
    r = synth.TINY.radar
    n_az, L, K = 1200, 128, 24
    api = rosar.Radar(r.fc, r.slope, r.t_sample(L), r.t_start, r.r0, r.c)
    g = torch.Generator(device="cuda").manual_seed(5)
    raws = [torch.randn(n_az, L, dtype=torch.complex64, device="cuda", generator=g) for _ in range(2)]
    w = torch.randn(L, K, dtype=torch.complex64, device="cuda", generator=g)
    o = torch.from_numpy(np.arange(-12, 12, dtype=np.int32) * 7).cuda()
    plan = rosar.sas_time_plan(None, w, o, api, n_az, L, transforms=True)
    assert plan.data.numel() != rosar.load().rosar_time_domain_plan_bytes(L, L, K)      # the form with scratch
    forms = [lambda raw, **k: rosar.sas_time_planned(raw, plan, **k), lambda raw, **k: rosar.sas_time(raw, None, w, o, api, transforms=True, **k)]
    side = torch.cuda.Stream()
    for form in forms:
        want = [form(raw) for raw in raws]
        outs = [[torch.empty_like(want[0]) for _ in range(40)] for _ in range(2)]
        torch.cuda.synchronize()
        for a, b in zip(*outs):                       # nothing waits between the two streams
            form(raws[0], out=a)
            form(raws[1], out=b, stream=side)
        torch.cuda.synchronize()
        for x, y in zip(outs, want):
            assert all(torch.equal(t, y) for t in x)
