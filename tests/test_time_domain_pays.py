"""Which SAS calls go by transforms: those that measured faster so, whatever their offsets."""

import ctypes

import pytest

import synth


@pytest.fixture(scope="module")
def lib():
    from paper_2309_08038_gb300 import build
    build.build()
    import paper_2309_08038_gb300 as rosar
    return rosar.load()


# (n_az, L, n_rng, K): measured on both sides, offsets over a sixth and the whole of the ring
FASTER = [(3600, 256, 256, 64), (4500, 320, 320, 128), (720, 128, 128, 109)]
SLOWER = [(4501, 208, 208, 2), (14400, 64, 64, 2), (14400, 208, 16, 2), (4501, 64, 64, 16), (4501, 1024, 16, 16),
          (2000, 1024, 1024, 2), (500, 208, 208, 2), (432, 288, 288, 21), (360, 64, 64, 16)]


def _ask(lib, fn, L, *args):
    r = synth.TINY.radar
    from paper_2309_08038_gb300 import _lib
    st = _lib.RadarStruct(r.fc, r.slope, r.t_sample(L), r.t_start, r.r0, r.c)
    return fn(ctypes.byref(st), *args)


@pytest.mark.parametrize("n_az,L,n_rng,K", FASTER + SLOWER)
def test_rule(lib, n_az, L, n_rng, K):
    pays = _ask(lib, lib.rosar_time_domain_fft_pays, L, n_az, L, n_rng, K)
    assert pays == ((n_az, L, n_rng, K) in FASTER)
    if pays:
        assert _ask(lib, lib.rosar_time_domain_fft_plan_bytes, L, 0, n_az, L, n_rng, K) > 0


def test_nothing_pays_that_is_not_offered(lib):
    assert lib.rosar_time_domain_fft_pays(None, 3600, 256, 256, 64) == 0
    assert _ask(lib, lib.rosar_time_domain_fft_pays, 256, 3600, 250, 250, 64) == 0          # L % 16
    assert _ask(lib, lib.rosar_time_domain_fft_pays, 256, 16001, 256, 256, 64) == 0         # no azimuth length
    assert _ask(lib, lib.rosar_time_domain_fft_pays, 256, 3600, 256, 0, 64) == 0
