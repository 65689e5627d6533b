"""The hop with eight threads per site, and the staged pipeline at each of its depths,
against the oracle at the edges of their sizes, with ragged last blocks.

FP32 spinors run on eight threads up to 12288 sites per parity, 16-bit ones up to 4096:
840 (a last block of 8 of 32 sites), 10080, and 12600 just above (a last block of
56 of 128).  FP64 runs on it at all of these.  The staged pipeline is deepest where
two blocks of 128 per SM hold the lattice (12600: 99 blocks), then three (46656: 365),
four (72000: 563) and the full occupancy (88000: 688 of 152 x 5).  Tolerances as for the operators
(per-site relative error): FP64 1e-12, FP32 1e-5 (2e-5 for K_hat), FP16 3e-3, BF16 3e-2
(twice that for K_hat).
"""
import numpy as np
import pytest

from oracle import lattice, wilson
from paper_1702_00124_gb300 import synthetic

pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 1: 1e-5, 2: 3e-3, 3: 3e-2}
LATS = [(6, 10, 14, 2), (10, 14, 18, 8), (10, 14, 18, 10), (18, 18, 16, 18), (20, 20, 20, 18), (22, 20, 20, 20)]


@pytest.fixture(scope="module", params=LATS, ids=lambda d: "x".join(map(str, d)))
def setup(request):
    from paper_1702_00124_gb300 import wdhmc
    from tests import gpu_util as gu
    dims = request.param
    U = synthetic.gauge_field(dims, 0.5, 3000 + dims[3])
    psi = synthetic.spinor_field(dims, 4000 + dims[3])
    ref = {d: wilson.hop(U, psi, dagger=d) for d in (False, True)}
    lat = wdhmc.Lattice(dims)
    lat.wd_gauge_load(gu.dev(U))
    yield dims, U, psi, ref, lat, gu
    lat.close()


@pytest.mark.parametrize("prec,recon", [(0, 0), (1, 0), (1, 1), (2, 1), (3, 0), (3, 1)])
def test_hop_and_khat(setup, prec, recon):
    dims, U, psi, ref, lat, gu = setup
    lat.wd_set_recon(recon)
    try:
        for dagger in (False, True):
            for out_par in (0, 1):
                out = lat.half_spinor()
                lat.wd_hop(out_par, dagger, prec, gu.pack(lat, psi, 1 - out_par), out)
                got = gu.unpack(lat, out, out_par)
                # D maps one parity onto the other: the whole field's hop, masked
                assert gu.site_rel_err(got, lattice.mask(ref[dagger], dims, out_par), out_par, dims) < TOL[prec]
        out = lat.half_spinor()
        lat.mdagm_apply(0.13, prec, 1, gu.pack(lat, psi, 0), out)
        kref = wilson.apply_Khat(U, lattice.mask(psi, dims, 0), 0.13)
        assert gu.site_rel_err(gu.unpack(lat, out, 0), kref, 0, dims) < (1 if prec == 0 else 2) * TOL[prec]
    finally:
        lat.wd_set_recon(0)


@pytest.mark.parametrize("recon", [0, 1])
def test_poly_step(setup, recon):
    """The Chebyshev step fused into the last hop (FP32) against the FP64 filter."""
    dims, U, psi, ref, lat, gu = setup
    x = gu.pack(lat, psi, 0)
    a, b = lat.half_spinor(), lat.half_spinor()
    lat.poly_filter_apply(0.12, (8, 0.05, 6.0), 0, x, a)
    lat.wd_set_recon(recon)
    try:
        lat.poly_filter_apply(0.12, (8, 0.05, 6.0), 1, x, b)
    finally:
        lat.wd_set_recon(0)
    # eight K_hat at 2e-5 each bound the sum of the recurrence's steps
    assert np.linalg.norm((a - b).cpu().numpy()) < 8 * 2e-5 * np.linalg.norm(a.cpu().numpy())
