"""The gather's tile widths (256 to 1536 outputs a CTA, chosen by row length and number of rows) at the edges of their
tiles, forward and adjoint, shared and per-row offsets, against an FP64 sum with the rounding bound of its products."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rosar():
    from paper_2309_08038_gb300 import build
    build.build()
    import paper_2309_08038_gb300 as r
    return r


# widths taken, in order: 1 (few rows), 1, 1, 2, 2, 3, 4, 5, 6 outputs a thread and 256 lanes
@pytest.mark.parametrize("n_az,n_rng", [(2, 1), (255, 3), (257, 3), (512, 256), (769, 320), (1536, 320), (1537, 320),
                                        (1025, 320), (1311, 256)])
@pytest.mark.parametrize("per_row", [False, True])
def test_tile_widths_match_fp64(rosar, n_az, n_rng, per_row):
    import torch
    from paper_2309_08038_gb300 import ops
    g = torch.Generator(device="cuda").manual_seed(n_az * 2 + per_row)
    K = 12
    S = torch.randn(n_rng, n_az, dtype=torch.complex64, device="cuda", generator=g)
    w = torch.randn(n_rng, K, dtype=torch.complex64, device="cuda", generator=g)
    o = torch.randint(-n_az + 1, n_az, (n_rng, K) if per_row else (K,), dtype=torch.int32, device="cuda", generator=g)
    th = torch.arange(n_az, device="cuda")
    rows = torch.arange(n_rng, device="cuda")[:, None]
    for adjoint in (False, True):
        got = rosar.sparse_azimuth(S, w, o)
        if adjoint:
            got = ops.sparse_azimuth_adjoint(S[None], None, w, o, want_w=False)[0][0]
        ref = torch.zeros(n_rng, n_az, dtype=torch.complex128, device="cuda")
        size = torch.zeros(n_rng, n_az, dtype=torch.float64, device="cuda")
        for k in range(K):
            off = (o[:, k:k + 1] if per_row else o[k]).long()
            idx = (th - off if adjoint else th + off) % n_az
            v = S[rows, idx.expand(n_rng, n_az)].to(torch.complex128)
            c = w[:, k:k + 1].to(torch.complex128)
            ref += (c.conj() if adjoint else c) * v
            size += c.abs() * v.abs()
        # two fused multiply-adds a product and component, K products in sequence: 2 K roundings of at most 2^-24 of
        # the running sum in each component
        assert ((got.to(torch.complex128) - ref).abs() <= 2 ** 0.5 * 2 * K * 2.0 ** -24 * size).all(), adjoint
