"""Overlapping arguments that the time-domain calls refused before they had a form by transforms are refused with it."""

import ctypes

import pytest
import torch

from paper_2309_08038_gb300 import ops

RADAR = ops.Radar(77e9, 1e14, 1e-7, 8e-6, 0.25)


class _Lib:
    def __init__(self):
        self.called = []

    def __getattr__(self, name):
        return lambda *a: 4096 if "fft" in name and name.endswith("_bytes") else 64 if name.endswith("_bytes") else \
            self.called.append(name) or 0


@pytest.fixture
def lib(monkeypatch):
    lib = _Lib()
    monkeypatch.setattr(ops._lib, "load", lambda *a: lib)
    monkeypatch.setattr(ops, "require", lambda t, *a, **k: t)
    monkeypatch.setattr(ops, "check", lambda status: None)
    monkeypatch.setattr(ops, "stream_handle", lambda s=None: 0)
    return lib


def test_sas_time_leaves_an_overlap_to_the_direct_call(lib):
    raw = torch.empty(64, 32, dtype=torch.complex64)
    mem = torch.zeros(32 * 64 + 128, dtype=torch.complex64)
    out = mem[:32 * 64].view(32, 64)
    w, o = torch.zeros(32, 4, dtype=torch.complex64), torch.zeros(4, dtype=torch.int32)
    into_w = mem[32 * 64 - 64:32 * 64 + 64].view(32, 4)                              # its first half lies in out
    into_o = torch.view_as_real(mem[32 * 64 - 1:32 * 64 + 1]).view(torch.int32).view(-1)[:4]
    for args, names in (((w, o), ["rosar_sas_time_fft_plan", "rosar_sas_time_fft"]), ((into_w, o), ["rosar_sas_time"]),
                        ((w, into_o), ["rosar_sas_time"])):
        lib.called.clear()
        ops.sas_time(raw, None, *args, RADAR, out=out, transforms=True)
        assert lib.called == names


def test_planned_calls_refuse_an_image_inside_the_plan(lib):
    raw = torch.empty(64, 32, dtype=torch.complex64)
    data = torch.zeros(1 << 16, dtype=torch.uint8)
    out = data[-32 * 64 * 8:].view(torch.complex64).view(32, 64)                      # in the plan's last planes
    plan = ops.TimeDomainPlan(data, 64, 32, 32, 4)
    for f in (ops.sas_time_planned, ops.bpa_time_planned):
        with pytest.raises(ops._lib.RosarError):
            f(raw, plan, out=out)
    assert not lib.called


def test_entries_refuse_an_overlap_with_the_part_every_plan_has():
    from paper_2309_08038_gb300 import build
    build.build()
    import paper_2309_08038_gb300 as rosar
    lib = rosar.load()
    n_az, L, M = 3600, 256, 600
    raw, plan, far, ws = (ctypes.c_void_p(x << 32) for x in (1, 2, 3, 4))
    need = lib.rosar_time_domain_fft_workspace_bytes(1, n_az, L, L, M)
    taps, plane = 16 * L * M, 8 * L * n_az
    inside = ctypes.c_void_p((2 << 32) + ((taps + 2 * plane - 4096) & ~255))         # the end of the second plane
    assert lib.rosar_bpa_time_fft(raw, plan, n_az, L, L, M, ws, need, inside, None) == 1
    assert b"overlaps" in lib.rosar_last_error()
    assert lib.rosar_bpa_time_fft(raw, plan, n_az, L, L, M, inside, need, far, None) == 1
    assert b"overlaps" in lib.rosar_last_error()
