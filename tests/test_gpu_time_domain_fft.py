"""Time-domain BPA and SAS by transforms (rosar_*_time_fft, what rosar.bpa_time and rosar.sas_time take for all but the
smallest sizes) against the FP64 oracle at the edges of its sizes, and its C entries' refusals (CPU)."""

import ctypes

import numpy as np
import pytest

import oracle as O
import synth

# interpolation at most 3e-6 of a tap, three float32 transforms of about 4e-7 each, float32 coefficients and windows
# 3e-7: 5e-6 of the image; the sampled pixels may hold a quarter of its average power
TOL = 2e-5


@pytest.fixture(scope="module")
def rosar():
    from paper_2309_08038_gb300 import build
    build.build()
    import paper_2309_08038_gb300 as r
    return r


def _radars(rosar, L):
    r = synth.TINY.radar
    return (rosar.Radar(r.fc, r.slope, r.t_sample(L), r.t_start, r.r0, r.c),
            O.Radar(fc=r.fc, slope=r.slope, t_s=r.t_sample(L), t_start=r.t_start, r0=r.r0, c=r.c))


def _sample(rng, n_rng, n_az, count=40):
    rows = np.concatenate([rng.integers(0, n_rng, count), [0, 0, 1, 2, n_rng - 1, n_rng - 1]])
    thetas = np.concatenate([rng.integers(0, n_az, count), [0, n_az - 1, 1, 0, 0, n_az - 1]])
    return rows, thetas


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def _bytes(rosar, bpa, n_az, L, n_rng, K):
    api, _ = _radars(rosar, L)
    return rosar.load().rosar_time_domain_fft_plan_bytes(ctypes.byref(api.as_struct()), bpa, n_az, L, n_rng, K)


# (n_az, L, n_rng, taps): compile-time lengths (circular), lengths with room for the wrapped pulses that fit exactly or
# miss by one, run-time lengths, odd lengths, range transforms of every kind (one pass, remainder radices 2, 4, 8, three
# passes, L not a power of two), fewer rows than bins, a whole ring
SHAPES = [(360, 64, 64, 60), (720, 128, 128, 40), (301, 64, 64, 60), (302, 80, 77, 60), (480, 512, 512, 33),
          (800, 144, 100, 50), (375, 208, 208, 40), (1031, 32, 32, 172), (2187, 16, 16, 300), (97, 256, 250, 97),
          (1800, 320, 64, 128), (2000, 48, 48, 300), (4096, 64, 40, 64), (3600, 1024, 24, 64), (500, 2048, 64, 32),
          (7000, 32, 30, 40), (14400, 64, 20, 48)]


@pytest.mark.gpu
@pytest.mark.parametrize("planned", [False, True])
@pytest.mark.parametrize("n_az,L,n_rng,M", SHAPES)
def test_bpa_time(rosar, n_az, L, n_rng, M, planned):
    import torch
    if n_az * n_rng * M * L >= 4e7:
        assert _bytes(rosar, 1, n_az, L, n_rng, M) > 0
    rng = np.random.default_rng(n_az + L)
    raw = (rng.standard_normal((n_az, L)) + 1j * rng.standard_normal((n_az, L))).astype(np.complex64)
    win = rng.uniform(0.1, 1.0, L).astype(np.float32) if L != 64 else None
    api, rad = _radars(rosar, L)
    d_raw, d_win = torch.from_numpy(raw).cuda(), torch.from_numpy(win).cuda() if win is not None else None
    if planned:
        got = rosar.bpa_time_planned(d_raw, rosar.bpa_time_plan(d_win, api, n_az, L, n_rng, M))
    else:
        got = rosar.bpa_time(d_raw, d_win, api, n_rng, M)
    rows, thetas = _sample(rng, n_rng, n_az)
    ref = O.bpa_time_pixels(raw, win, rad, n_az, M, rows, thetas)
    assert _rel(got.cpu().numpy()[rows, thetas], ref) <= TOL


@pytest.mark.gpu
@pytest.mark.parametrize("centred", [False, True])
@pytest.mark.parametrize("n_az,L,n_rng,K", SHAPES)
def test_sas_time(rosar, n_az, L, n_rng, K, centred):
    """Offsets in no order over more than the ring, one repeated, some of them turns apart; planned and not."""
    import torch
    rng = np.random.default_rng(n_az + L + K)
    raw = (rng.standard_normal((n_az, L)) + 1j * rng.standard_normal((n_az, L))).astype(np.complex64)
    win = rng.uniform(0.1, 1.0, L).astype(np.float32) if L != 64 else None
    spread = n_az if L in (32, 144) else n_az // 8
    o = rng.integers(-spread, spread + 1, K).astype(np.int32)
    o[1] = o[0]
    o[2] += 3 * n_az
    o[3] -= 2 * n_az
    w = (rng.standard_normal((n_rng, K)) + 1j * rng.standard_normal((n_rng, K))).astype(np.complex64)
    api, rad = _radars(rosar, L)
    t = [None if x is None else torch.from_numpy(x).cuda() for x in (raw, win, w, o)]
    rows, thetas = _sample(rng, n_rng, n_az)
    ref = O.sas_time_pixels(raw, win, w, o, rad, n_az, rows, thetas, centred=centred)
    got = rosar.sas_time(*t, api, centred=centred)
    assert _rel(got.cpu().numpy()[rows, thetas], ref) <= TOL
    plan = rosar.sas_time_plan(t[1], t[2], t[3], api, n_az, L, centred=centred)
    assert _rel(rosar.sas_time_planned(t[0], plan).cpu().numpy()[rows, thetas], ref) <= TOL


@pytest.mark.gpu
@pytest.mark.parametrize("n_az", [360, 500, 800])
def test_pulses_that_are_not_finite_stay_where_they_are_read(rosar, n_az):
    """The tensor-core entry gives the same pixels NaN, the others agree; nothing is left of it in the next call."""
    import torch
    L, M = 80, 60
    rng = np.random.default_rng(n_az)
    raw = (rng.standard_normal((n_az, L)) + 1j * rng.standard_normal((n_az, L))).astype(np.complex64)
    clean = torch.from_numpy(raw).cuda()
    raw[3, 7] = np.nan
    raw[n_az - 1, L - 1] = 1j * np.inf
    raw[n_az // 2, 0] = -np.inf
    api, _ = _radars(rosar, L)
    bad = torch.from_numpy(raw).cuda()
    ref = torch.empty((L, n_az), dtype=torch.complex64, device="cuda")
    lib = rosar.load()
    assert lib.rosar_bpa_time(bad.data_ptr(), None, ctypes.byref(api.as_struct()), n_az, L, L, M, ref.data_ptr(),
                              torch.cuda.current_stream().cuda_stream) == 0
    before = rosar.bpa_time(clean, None, api, L, M)
    got = rosar.bpa_time(bad, None, api, L, M)
    after = rosar.bpa_time(clean, None, api, L, M)
    fine = torch.isfinite(torch.view_as_real(ref)).all(-1)
    assert torch.equal(torch.isfinite(torch.view_as_real(got)).all(-1), fine) and 0 < (~fine).sum() < ref.numel() // 2
    assert (got[fine] - ref[fine]).norm() <= 1e-4 * ref[fine].norm()
    assert torch.equal(before, after)


@pytest.mark.gpu
def test_graph_capture_and_another_stream(rosar):
    import torch
    api, _ = _radars(rosar, 64)
    raw = torch.randn(800, 64, dtype=torch.complex64, device="cuda")
    want = rosar.bpa_time(raw, None, api, 64, 130)
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    outs = []
    for _ in range(20):                       # scratch of a call on a stream that is not the current one
        outs.append(rosar.bpa_time(raw, None, api, 64, 130, stream=side))
    side.synchronize()
    assert all(torch.equal(o, want) for o in outs)
    out = torch.zeros_like(want)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        rosar.bpa_time(raw, None, api, 64, 130, out=out)
    out.zero_()
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(out, want)


def test_entries_refuse_bad_arguments(rosar):
    lib = rosar.load()
    api, _ = _radars(rosar, 256)
    st = api.as_struct()
    at = [ctypes.c_void_p(x << 32) for x in range(1, 6)]
    size = lambda *a: lib.rosar_time_domain_fft_plan_bytes(*a)  # noqa: E731
    need = size(ctypes.byref(st), 1, 3600, 256, 256, 600)
    assert need > 0 and need != lib.rosar_time_domain_plan_bytes(256, 256, 600)
    assert size(None, 1, 3600, 256, 256, 600) == 0
    assert size(ctypes.byref(st), 2, 3600, 256, 256, 600) == 0
    assert size(ctypes.byref(st), 1, 3600, 256, 256, 3601) == 0          # more taps than pulses
    assert size(ctypes.byref(st), 1, 3600, 250, 250, 600) == 0           # L % 16
    assert size(ctypes.byref(st), 1, 3600, 256, 257, 600) == 0           # more rows than bins
    assert size(ctypes.byref(st), 1, 3600, 4096, 256, 600) == 0          # L past the range transforms
    assert size(ctypes.byref(st), 0, 16001, 256, 256, 64) == 0           # no azimuth length
    assert size(ctypes.byref(st), 0, 360, 64, 64, 16) == 0               # too small to pay
    far = rosar.Radar(st.fc_hz, st.slope_hz_per_s, st.t_sample_s, st.t_start_s, 5.0, 0.0).as_struct()
    assert size(ctypes.byref(far), 0, 3600, 256, 256, 64) == 0           # an arm of 80 bins
    plan = lib.rosar_bpa_time_fft_plan
    assert plan(None, ctypes.byref(st), 3600, 256, 256, 600, at[0], need - 1, None) == 1
    assert plan(None, ctypes.byref(st), 3600, 256, 256, 600, ctypes.c_void_p((1 << 32) + 16), need, None) == 1
    assert plan(None, ctypes.byref(st), 360, 64, 64, 16, at[0], need, None) == 2
    assert lib.rosar_sas_time_fft_plan(None, None, at[1], ctypes.byref(st), 3600, 256, 256, 64, 1, at[0], need, None) == 1
    assert lib.rosar_sas_time_fft_plan(None, at[1], at[2], ctypes.byref(st), 3600, 256, 256, 64, 2, at[0], need, None) == 1
    ws = lib.rosar_time_domain_fft_workspace_bytes(1, 3600, 256, 256, 600)
    run = lib.rosar_bpa_time_fft
    assert run(at[0], at[1], 3600, 256, 256, 600, at[2], ws - 1, at[3], None) == 1
    assert run(at[0], at[1], 3600, 256, 256, 600, None, ws, at[3], None) == 1
    assert run(at[0], at[1], 3600, 256, 256, 600, at[2], ws, at[0], None) == 1      # out is raw
    assert run(at[0], at[1], 3600, 256, 256, 600, at[0], ws, at[3], None) == 1      # workspace is raw
    assert run(ctypes.c_void_p((1 << 32) + 8), at[1], 3600, 256, 256, 600, at[2], ws, at[3], None) == 1
    assert run(at[0], at[1], 16001, 256, 256, 600, at[2], ws, at[3], None) == 2
