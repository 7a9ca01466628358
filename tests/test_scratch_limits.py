"""sas_time and sas_time_plan where the memory for the transform form is not there: the tensor-core form, as before."""

import pytest
import torch

from paper_2309_08038_gb300 import ops

RADAR = ops.Radar(77e9, 1e14, 1e-7, 8e-6, 0.25)
TENSOR_CORE_PLAN = 512


class _Lib:
    def __init__(self, plan_bytes):
        self.plan_bytes, self.called = plan_bytes, []

    def __getattr__(self, name):
        if name == "rosar_time_domain_fft_pays":
            return lambda *a: 1
        if name == "rosar_time_domain_fft_plan_bytes":
            return lambda *a: self.plan_bytes
        if name.endswith("_bytes"):
            return lambda *a: TENSOR_CORE_PLAN
        return lambda *a: self.called.append(name) or 0


@pytest.mark.parametrize("plan_bytes,room,transforms", [(1 << 16, 1 << 20, True), (1 << 16, 1 << 12, False),
                                                        ((1 << 30) + 1, 1 << 40, False)])
def test_sas_time_falls_back(monkeypatch, plan_bytes, room, transforms):
    lib, empty = _Lib(plan_bytes), torch.empty
    raw, w, o = empty(64, 32, dtype=torch.complex64), empty(32, 4, dtype=torch.complex64), torch.zeros(4, dtype=torch.int32)
    out = empty(32, 64, dtype=torch.complex64)

    def bounded(shape, *a, **k):
        if isinstance(shape, int) and shape > room:
            raise torch.cuda.OutOfMemoryError("out of memory")
        return empty(min(shape, 1 << 20) if isinstance(shape, int) else shape, *a, **k)

    monkeypatch.setattr(ops._lib, "load", lambda *a: lib)
    monkeypatch.setattr(ops, "require", lambda t, *a, **k: t)
    monkeypatch.setattr(ops, "check", lambda status: None)
    monkeypatch.setattr(ops, "stream_handle", lambda s=None: 0)
    monkeypatch.setattr(torch, "empty", bounded)
    ops.sas_time(raw, None, w, o, RADAR, out=out)
    assert lib.called == (["rosar_sas_time_fft_plan", "rosar_sas_time_fft"] if transforms else ["rosar_sas_time"])
    lib.called.clear()
    plan = ops.sas_time_plan(None, w, o, RADAR, 64, 32)
    fits = plan_bytes <= room
    assert lib.called == (["rosar_sas_time_fft_plan"] if fits else ["rosar_sas_time_plan"])
    assert (plan.data.numel() == TENSOR_CORE_PLAN) == (not fits)
