"""A time-domain plan is used as what it was made for: plans by transforms of BPA and of SAS are laid out differently."""


import pytest
import torch

from paper_2309_08038_gb300 import ops


@pytest.mark.parametrize("made_for_bpa", [False, True])
def test_a_plan_runs_as_its_own_kind(monkeypatch, made_for_bpa):
    called = []

    class Lib:
        def __getattr__(self, name):
            if name.endswith("_bytes"):
                return lambda *a: called.append((name, a[0])) or 512
            return lambda *a: called.append((name, a)) or 0

    monkeypatch.setattr(ops._lib, "load", lambda *a: Lib())
    monkeypatch.setattr(ops, "require", lambda t, *a, **k: t)
    monkeypatch.setattr(ops, "check", lambda status: None)
    monkeypatch.setattr(ops, "stream_handle", lambda s=None: 0)
    raw, out = torch.empty(64, 32, dtype=torch.complex64), torch.empty(32, 64, dtype=torch.complex64)
    radar = ops.Radar(77e9, 1e14, 1e-7, 8e-6, 0.25)
    monkeypatch.setattr(ops, "_scratch", lambda n, *a: torch.empty(n, dtype=torch.uint8))
    if made_for_bpa:
        plan = ops.bpa_time_plan(None, radar, 64, 32, 32, 4, device="cpu")
    else:
        plan = ops.sas_time_plan(None, torch.empty(32, 4, dtype=torch.complex64), torch.zeros(4, dtype=torch.int32), radar, 64, 32)
    plan = ops.TimeDomainPlan(torch.empty(1024, dtype=torch.uint8), *list(plan.__dict__.values())[1:])
    for f in (ops.sas_time_planned, ops.bpa_time_planned):
        called.clear()
        f(raw, plan, out=out)
        names = [n for n, _ in called]
        assert ("rosar_bpa_time_fft" if made_for_bpa else "rosar_sas_time_fft") in names
        assert ("rosar_time_domain_fft_workspace_bytes", int(made_for_bpa)) in called


@pytest.fixture(scope="module")
def rosar():
    from paper_2309_08038_gb300 import build
    build.build()
    import paper_2309_08038_gb300 as r
    return r


def _case(rosar, n_az, L, n_rng, K):
    import synth
    r = synth.TINY.radar
    api = rosar.Radar(r.fc, r.slope, r.t_sample(L), r.t_start, r.r0, r.c)
    g = torch.Generator(device="cuda").manual_seed(n_az)
    raw = torch.randn(n_az, L, dtype=torch.complex64, device="cuda", generator=g)
    w = torch.randn(n_rng, K, dtype=torch.complex64, device="cuda", generator=g)
    o = torch.arange(K, dtype=torch.int32, device="cuda") - K // 2
    return api, raw, rosar.sas_time_plan(None, w, o, api, n_az, L, transforms=True), rosar.bpa_time_plan(None, api, n_az, L, n_rng, K, transforms=True)


# 1031: the two kinds pad the row to different lengths; 360: to the same
@pytest.mark.gpu
@pytest.mark.parametrize("n_az,L,n_rng,K", [(1031, 32, 32, 172), (360, 64, 64, 60)])
def test_entries_give_nan_for_a_plan_of_another_kind_or_size(rosar, n_az, L, n_rng, K):
    api, raw, sas, bpa = _case(rosar, n_az, L, n_rng, K)
    want = {0: rosar.sas_time_planned(raw, sas), 1: rosar.bpa_time_planned(raw, bpa)}
    assert torch.equal(rosar.bpa_time_planned(raw, sas), want[0]) and torch.equal(rosar.sas_time_planned(raw, bpa), want[1])
    lib = rosar.load()
    for kind, own, other in ((0, sas, bpa), (1, bpa, sas)):
        ws = torch.empty(lib.rosar_time_domain_fft_workspace_bytes(kind, n_az, L, n_rng, K), dtype=torch.uint8, device="cuda")
        f = lib.rosar_bpa_time_fft if kind else lib.rosar_sas_time_fft
        for plan, n, good in ((own, n_rng, True), (other, n_rng, False), (own, n_rng - 1, False),
                              (torch.zeros_like(own.data), n_rng, False)):
            out = torch.zeros((n, n_az), dtype=torch.complex64, device="cuda")
            data = plan if isinstance(plan, torch.Tensor) else plan.data
            assert f(raw.data_ptr(), data.data_ptr(), n_az, L, n, K, ws.data_ptr(), ws.numel(), out.data_ptr(),
                     torch.cuda.current_stream().cuda_stream) == 0, lib.rosar_last_error()
            assert torch.equal(out, want[kind]) if good else torch.isnan(torch.view_as_real(out)).all()
