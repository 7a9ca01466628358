"""Time-domain forms by transforms: samples far too large for the transforms reach the pixels that read their pulse and no
others, as in the direct sums."""

import ctypes

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rosar():
    from paper_2309_08038_gb300 import build
    build.build()
    import paper_2309_08038_gb300 as r
    return r


# a compile-time length, a padded one, a run-time one for SAS (1000); L off a power of two, and one sample tile with a tail
@pytest.mark.parametrize("size", [1e25, 3e35])
@pytest.mark.parametrize("n_az,L", [(360, 80), (500, 80), (1000, 208)])
@pytest.mark.parametrize("bpa", [True, False])
def test_large_samples_stay_where_they_are_read(rosar, bpa, n_az, L, size):
    import torch
    rng = np.random.default_rng(n_az)
    K = 40
    raw = (rng.standard_normal((n_az, L)) + 1j * rng.standard_normal((n_az, L))).astype(np.complex64)
    raw[3, 7] = size
    raw[3, L - 1] = -0.5j * size
    raw[n_az - 1, 0] = size * (0.3 - 0.8j)
    clean = np.where(np.abs(raw) > 1e10, 0, raw)
    r = synth.TINY.radar
    api = rosar.Radar(r.fc, r.slope, r.t_sample(L), r.t_start, r.r0, r.c)
    st, lib, s = api.as_struct(), rosar.load(), torch.cuda.current_stream().cuda_stream
    o = np.sort(rng.choice(80, K, replace=False)).astype(np.int32) - 40
    w = (rng.standard_normal((L, K)) + 1j * rng.standard_normal((L, K))).astype(np.complex64)
    t_raw, t_clean, t_w, t_o = (torch.from_numpy(x).cuda() for x in (raw, clean, w, o))
    win = torch.from_numpy(rng.uniform(0.1, 1.0, L).astype(np.float32)).cuda()
    ref = torch.empty((L, n_az), dtype=torch.complex64, device="cuda")
    if bpa:
        M = 60
        assert lib.rosar_bpa_time(t_raw.data_ptr(), win.data_ptr(), ctypes.byref(st), n_az, L, L, M, ref.data_ptr(), s) == 0
        image = lambda x: rosar.bpa_time(x, win, api, L, M, transforms=True)  # noqa: E731
        o = np.arange(-(M // 2), M - M // 2)
    else:
        assert lib.rosar_sas_time(t_raw.data_ptr(), win.data_ptr(), t_w.data_ptr(), t_o.data_ptr(), 0, ctypes.byref(st), n_az,
                                  L, L, K, 1, ref.data_ptr(), s) == 0
        image = lambda x: rosar.sas_time(x, win, t_w, t_o, api, transforms=True)  # noqa: E731
    got, alone = image(t_raw).cpu().numpy(), image(t_clean).cpu().numpy()
    again = image(t_raw).cpu().numpy()
    ref = ref.cpu().numpy()
    reads = np.zeros(n_az, bool)
    for n in (3, n_az - 1):
        reads[(n - o) % n_az] = True
    assert 0 < reads.sum() < n_az // 2
    assert np.array_equal(got[:, ~reads], alone[:, ~reads])       # the others: as if the samples were not there
    a, b = got[:, reads].astype(np.complex128), ref[:, reads].astype(np.complex128)
    assert np.isfinite(a).all() and np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)      # the forms' parity bar
    assert np.array_equal(got, again)
