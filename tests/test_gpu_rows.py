"""The row filter's variants (few and many rows, compile-time and run-time plans, in place) and the launches by length
against the FP64 oracle and against each other, bit for bit where the arithmetic is the same."""

import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu

TOL_FFT_FILTER = 5e-6     # the frequency-domain filter's bar in the parity tests


@pytest.fixture(scope="module")
def rosar():
    from paper_2309_08038_gb300 import build
    build.build()
    import paper_2309_08038_gb300 as r
    return r


def _c(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


# rows of one pass, two passes, padded (powers of two) and odd lengths, the thread counts' edges (2048, 4096, 8192) and
# the compile-time plans; few rows stage H, more than 304 read it in the fused step
@pytest.mark.parametrize("n_az", [2, 15, 16, 30, 32, 81, 360, 625, 800, 1024, 1800, 2048, 2187, 3600, 4096, 4500, 7200,
                                  8192, 8640, 14400, 16384])
def test_many_rows_equal_few_rows_and_oracle(rosar, n_az):
    import torch
    rng = np.random.default_rng(n_az)
    n_rng, K = 20, 8
    n_scans = 16                                         # 320 rows in one call, 20 in each of the others
    o = rng.integers(-n_az, n_az, K).astype(np.int32)
    w = _c(rng, n_rng, K)
    S = _c(rng, n_scans, n_rng, n_az)
    P = np.exp(1j * rng.standard_normal((n_scans, n_az))).astype(np.complex64)
    t = {k: torch.from_numpy(v).cuda() for k, v in (("o", o), ("w", w), ("S", S), ("P", P))}
    H = rosar.azimuth_plan(t["w"], t["o"], n_az)
    many = rosar.sparse_azimuth_fft_scans(t["S"], H)
    for s in range(n_scans):
        assert torch.equal(many[s], rosar.sparse_azimuth_fft(t["S"][s], H)), s
    ref = O.sparse_azimuth(S[0], w, o)
    got = many[0].cpu().numpy()
    assert np.linalg.norm(got - ref) <= TOL_FFT_FILTER * np.linalg.norm(ref)
    # the adjoint with the phase applied at load and the spectrum kept
    X = torch.empty_like(t["S"])
    adj = rosar.sparse_azimuth_fft_scans_ex(t["S"], H, P=t["P"], adjoint=True, spectrum=X)
    for s in (0, n_scans - 1):
        one = torch.empty_like(X[:1])
        alone = rosar.sparse_azimuth_fft_scans_ex(t["S"][s:s + 1], H, P=t["P"][s:s + 1], adjoint=True, spectrum=one)
        assert torch.equal(adj[s], alone[0]) and torch.equal(X[s], one[0]), s


@pytest.mark.parametrize("n_az,L,n_scans", [(800, 64, 6), (1024, 32, 11), (2187, 16, 21), (9000, 64, 3), (3600, 1024, 2)])
def test_scans_in_place_equal_single_scans(rosar, n_az, L, n_scans):
    import torch
    rng = np.random.default_rng(n_az)
    w = torch.from_numpy(_c(rng, L, 8)).cuda()
    H = rosar.azimuth_plan(w, torch.arange(-4, 4, dtype=torch.int32, device="cuda"), n_az)
    win = torch.from_numpy(synth.hann_window(L)).cuda()
    raw = torch.from_numpy(_c(rng, n_scans, n_az, L)).cuda()
    got = rosar.image_fft_scans(raw, win, H)
    for s in range(n_scans):
        assert torch.equal(got[s], rosar.image_fft(raw[s], win, H)), s


@pytest.mark.parametrize("lengths", [[360, 800, 1024, 7200, 2187, 16], None])
def test_batch_by_length_equals_single_scans(rosar, lengths):
    """Every range length and several row lengths; eighteen row lengths take the persistent kernel."""
    import torch
    lengths = lengths or [n for n in range(360, 2000) if rosar.azimuth_fft_supported(n)][:18]
    rng = np.random.default_rng(len(lengths))
    scans = []
    for i, n_az in enumerate(lengths + lengths[:2]):
        L = 2 ** (4 + i % 8)
        w, o = _c(rng, L, 8), rng.integers(-n_az, n_az, 8).astype(np.int32)
        sc = {k: torch.from_numpy(v).cuda() for k, v in (("raw", _c(rng, n_az, L)), ("w", w), ("o", o))}
        sc["win"] = torch.from_numpy(synth.hann_window(L)).cuda() if i % 3 else None
        sc["H"] = rosar.azimuth_plan(sc["w"], sc["o"], n_az)
        scans.append(sc)
    b = rosar.Batch(scans)
    info = b.info()
    assert info["ctas"] >= 1 and info["range_tiles"] > 0 and info["azimuth_tiles"] == sum(2 ** (4 + i % 8)
                                                                                           for i in range(len(scans)))
    for _ in range(2):
        for out in b.outs:
            out.zero_()
        b.launch()
        b.status()
        for i, (out, sc) in enumerate(zip(b.outs, scans)):
            assert torch.equal(out, rosar.image_fft(sc["raw"], sc["win"], sc["H"])), i
    b.close()


# the migrating filter's plans of one, two and more passes, padded and odd, at the lines between its thread counts and
# (n_rng 305) between few and many rows; the gather form's bar is 2e-6 and the filter's 5e-6, each against FP64
@pytest.mark.parametrize("n_az,n_rng", [(2, 7), (16, 305), (30, 7), (81, 305), (360, 9), (675, 5), (1024, 305), (1800, 9),
                                        (1800, 305), (2048, 5), (2250, 305), (3600, 6), (4096, 3), (4500, 3), (7200, 4),
                                        (8192, 3), (8640, 305), (14400, 2), (16384, 2)])
def test_migrating_filter_equals_gather_form(rosar, n_az, n_rng):
    import torch
    rng = np.random.default_rng(n_az + n_rng)
    K = 6
    S, w = torch.from_numpy(_c(rng, n_rng + 2, n_az)).cuda(), torch.from_numpy(_c(rng, n_rng, K)).cuda()
    o = torch.from_numpy(rng.integers(-n_az // 2, n_az // 2 + 1, K).astype(np.int32)).cuda()
    dl = torch.from_numpy(rng.integers(-2, 5, (n_rng, K)).astype(np.int32)).cuda()     # rows on both sides are missing
    plan = rosar.azimuth_plan_migrating(w, o, dl, n_az)
    got = rosar.sparse_azimuth_migrating_fft(S, plan)
    ref = rosar.sparse_azimuth_migrating(S, w, o, dl)
    assert torch.linalg.norm(got - ref) <= (TOL_FFT_FILTER + 2e-6) * torch.linalg.norm(ref)


# every length (and so every number and radix of passes), pulse counts around the tiles of 4, 8, 16 and 32 pulses; the
# bar of the adjoint's parity test
@pytest.mark.parametrize("L", [8, 16, 32, 64, 128, 256, 512, 1024, 2048, 4096])
@pytest.mark.parametrize("n_az", [1, 15, 33])
def test_range_adjoint_tiles_match_oracle(rosar, L, n_az):
    import torch
    rng = np.random.default_rng(L + n_az)
    g = _c(rng, L, n_az)
    win = synth.hann_window(L)
    for w in (win, None):
        for centred in (True, False):
            got = rosar.range_compress_adjoint(torch.from_numpy(g).cuda(), None if w is None else torch.from_numpy(w).cuda(),
                                               centred=centred).cpu().numpy()
            ref = O.range_compress_adjoint(g, np.ones(L, np.float32) if w is None else w, centred)
            assert np.linalg.norm(got - ref) <= 2e-6 * np.linalg.norm(ref), centred
