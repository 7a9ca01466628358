"""Back-projection with nominal positions in the azimuth-frequency domain (rosar_bpa on rows long enough for it)
against the FP64 oracle, at the edges of its row lengths."""

import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu

TOL_IMAGE = 1e-4     # the relative-L2 bar of the parity tests


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


def _run(rosar, S, M, n_rng, interp, **kw):
    import torch
    api, _ = _radars(rosar, S.shape[0])
    dev = {k: torch.from_numpy(v).cuda() for k, v in kw.items()}
    return rosar.bpa(torch.from_numpy(S).cuda(), api, n_rng, M, interp=interp, **dev).cpu().numpy()


# (n_az, M, L, n_rng): rows that are a plan themselves, rows whose extension fills a plan exactly or misses it by
# one, whole rings, more rows than are taken at once, rows near L (planes past the last bin read zero), and every
# length of the list
CASES = [(360, 200, 64, 64), (301, 60, 128, 120), (302, 60, 128, 120), (421, 60, 128, 128), (540, 61, 128, 100),
         (97, 97, 512, 512), (480, 480, 64, 64), (641, 80, 64, 64), (960, 131, 64, 64), (1000, 201, 64, 64),
         (1200, 150, 64, 64), (1300, 141, 64, 64), (1501, 300, 64, 64), (2000, 401, 64, 64), (2500, 381, 64, 64),
         (2100, 301, 512, 512), (3600, 600, 32, 32), (3001, 600, 512, 400), (4001, 800, 32, 32), (4800, 801, 32, 32),
         (5001, 760, 32, 32), (7200, 1200, 32, 32), (6001, 1200, 32, 32)]


@pytest.mark.parametrize("interp", ["linear", "nearest"])
@pytest.mark.parametrize("n_az,M,L,n_rng", CASES)
def test_rows_match_oracle(rosar, n_az, M, L, n_rng, interp):
    assert n_rng * n_az * M >= 2e6       # below that the direct kernel is taken
    rng = np.random.default_rng(n_az + M)
    S = (rng.standard_normal((L, n_az)) + 1j * rng.standard_normal((L, n_az))).astype(np.complex64)
    got = _run(rosar, S, M, n_rng, interp)
    assert got.shape == (n_rng, n_az)
    _, rad = _radars(rosar, L)
    dR = O.range_bin_spacing(rad, L)
    d = np.arange(-(M // 2), M - M // 2)
    checked = 0
    for r in (0, 1, 2, n_rng // 2, n_rng - 2, n_rng - 1):
        if interp == "nearest":      # a bin within 1e-4 of a tie may round either way
            x = O.slant_range(rad.r0 + r * dR, 0.0, rad.r0, O.phase_centre_angle(d, n_az)) / dR
            if np.any(np.abs(x - np.floor(x) - 0.5) < 1e-4):
                continue
        ref = O.bpa_pixels(S, rad, n_az, M, np.full(n_az, r), np.arange(n_az), interp)
        assert np.linalg.norm(got[r] - ref) <= TOL_IMAGE * np.linalg.norm(ref), r
        checked += 1
    assert checked >= 2


@pytest.mark.parametrize("interp", ["linear", "nearest"])
def test_values_that_are_not_finite_stay_where_they_are_read(rosar, interp):
    """Zero position errors take the direct kernel: the same pixels are not finite, the others agree."""
    rng = np.random.default_rng(3)
    S = (rng.standard_normal((64, 800)) + 1j * rng.standard_normal((64, 800))).astype(np.complex64)
    S[0, 5] = np.nan
    S[20, 790] = np.inf
    S[63, 400] = 1e35
    got = _run(rosar, S, 130, 64, interp)
    ref = _run(rosar, S, 130, 64, interp, dphi=np.zeros(800, np.float32))
    same = np.isfinite(ref)
    assert np.array_equal(np.isfinite(got), same) and 0 < (~same).sum() < ref.size // 4
    for r in range(64):
        ok = same[r] & (np.abs(ref[r]) < 1e30)
        assert np.linalg.norm(got[r][ok] - ref[r][ok]) <= TOL_IMAGE * np.linalg.norm(ref[r][ok]), r
