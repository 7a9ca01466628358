"""Time-domain BPA: the Python calls give the tensor-core entries' bits unless the caller asks for transforms, and the
transforms stay at the oracle's bar."""

import ctypes

import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu

TOL_TRANSFORMS = 2e-5     # three float32 transforms and the interpolation, on sampled pixels


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


@pytest.mark.parametrize("n_az,L,n_rng,M", [(360, 64, 64, 60), (1031, 208, 200, 172), (3600, 256, 256, 600)])
def test_default_gives_the_tensor_core_bits(rosar, n_az, L, n_rng, M):
    import torch
    rng = np.random.default_rng(n_az)
    raw = torch.from_numpy((rng.standard_normal((n_az, L)) + 1j * rng.standard_normal((n_az, L))).astype(np.complex64)).cuda()
    win = torch.from_numpy(synth.hann_window(L)).cuda()
    api, _ = _radars(rosar, L)
    st, lib, s = api.as_struct(), rosar.load(), torch.cuda.current_stream().cuda_stream
    want = torch.empty((n_rng, n_az), dtype=torch.complex64, device="cuda")
    assert lib.rosar_bpa_time(raw.data_ptr(), win.data_ptr(), ctypes.byref(st), n_az, L, n_rng, M, want.data_ptr(), s) == 0
    assert torch.equal(rosar.bpa_time(raw, win, api, n_rng, M), want)
    nbytes = lib.rosar_time_domain_plan_bytes(n_rng, L, M)
    data = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
    assert lib.rosar_bpa_time_plan(win.data_ptr(), ctypes.byref(st), n_az, L, n_rng, M, data.data_ptr(), nbytes, s) == 0
    assert lib.rosar_bpa_time_planned(raw.data_ptr(), data.data_ptr(), n_az, L, n_rng, M, want.data_ptr(), s) == 0
    plan = rosar.bpa_time_plan(win, api, n_az, L, n_rng, M)
    assert plan.data.numel() == nbytes
    assert torch.equal(rosar.bpa_time_planned(raw, plan), want)


# compile-time lengths, lengths with room for the wrapped pulses, run-time lengths, every kind of range transform
@pytest.mark.parametrize("n_az,L,n_rng,M", [(360, 64, 64, 60), (301, 64, 64, 60), (302, 80, 77, 60), (480, 512, 512, 33),
                                            (1031, 32, 32, 172), (2187, 16, 16, 300), (97, 256, 250, 97), (4096, 64, 40, 64),
                                            (3600, 1024, 24, 64), (500, 2048, 64, 32), (14400, 64, 20, 48)])
def test_transforms_match_oracle(rosar, n_az, L, n_rng, M):
    import torch
    rng = np.random.default_rng(n_az + L)
    raw = (rng.standard_normal((n_az, L)) + 1j * rng.standard_normal((n_az, L))).astype(np.complex64)
    win = rng.uniform(0.1, 1.0, L).astype(np.float32)
    api, rad = _radars(rosar, L)
    t_raw, t_win = torch.from_numpy(raw).cuda(), torch.from_numpy(win).cuda()
    rows = np.concatenate([rng.integers(0, n_rng, 40), [0, 0, 1, n_rng - 1]])
    thetas = np.concatenate([rng.integers(0, n_az, 40), [0, n_az - 1, 1, n_az - 1]])
    ref = O.bpa_time_pixels(raw, win, rad, n_az, M, rows, thetas)
    got = rosar.bpa_time(t_raw, t_win, api, n_rng, M, transforms=True)
    plan = rosar.bpa_time_plan(t_win, api, n_az, L, n_rng, M, transforms=True)
    if n_az * n_rng * M * L >= 4e7:
        assert plan.data.numel() != rosar.load().rosar_time_domain_plan_bytes(n_rng, L, M)
    for y in (got, rosar.bpa_time_planned(t_raw, plan)):
        assert np.linalg.norm(y.cpu().numpy()[rows, thetas] - ref) <= TOL_TRANSFORMS * np.linalg.norm(ref)
