"""Operators in place, and at the edges of their launch rules.

In place: every operator call but an FP64 hop copies or reads what it needs before it writes, so input and
output may be one buffer; with FP32 the last hop stores FP64 itself.  Bit for bit the results of two
buffers.  Edges: K_hat with one block of 32 sites on either side of the early start's lines (FP64: 50, 51, 303, 304
blocks; double-float: 76, 77, 152, 153) and FP16 spinors on 18-real links where the staged pipeline takes
them (above 4096 sites per parity), against the oracle, per-site relative error: FP64 and double-float 1e-12,
FP16 6e-3 (twice that of a hop).
"""
import pytest

from oracle import lattice, wilson
from paper_1702_00124_gb300 import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(6, 10, 14, 2), (12, 12, 12, 20)], ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("prec,recon", [(0, 0), (1, 0), (1, 1), (2, 0), (3, 1), (4, 0)])
def test_in_place(dims, prec, recon):
    import torch
    from paper_1702_00124_gb300 import wdhmc as wd
    from tests import gpu_util as gu
    lat = wd.Lattice(dims)
    lat.wd_gauge_load(gu.dev(synthetic.gauge_field(dims, 0.5, 14000)))
    lat.wd_set_recon(recon)
    x = torch.randn(72 * lat.Vh, dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(14001))
    one = x[:24 * lat.Vh]

    def check(f, src):
        a, b = torch.zeros_like(src), src.clone()
        f(src, a)
        f(b, b)
        assert torch.equal(a, b)

    for dagger in (0, 1):
        if prec != 0:
            check(lambda i, o: lat.wd_hop(1, dagger, prec, i, o), one)
        check(lambda i, o: lat.wd_apply(0.13, dagger, prec, i, o), one)
    check(lambda i, o: lat.mdagm_apply(0.13, prec, 1, i, o), one)
    check(lambda i, o: lat.mdagm_apply(0.13, prec, 3, i, o), x)
    lat.close()


@pytest.mark.parametrize("dims,prec,tol", [((8, 10, 10, 4), 0, 1e-12), ((34, 6, 4, 4), 0, 1e-12), ((202, 6, 4, 4), 0, 1e-12), ((8, 8, 8, 38), 0, 1e-12),
                                           ((8, 4, 4, 38), 4, 1e-12), ((14, 22, 4, 4), 4, 1e-12), ((8, 8, 4, 38), 4, 1e-12), ((6, 6, 8, 34), 4, 1e-12),
                                           ((8, 8, 16, 8), 2, 6e-3), ((10, 14, 18, 4), 2, 6e-3), ((10, 14, 18, 10), 2, 6e-3)], ids=str)
def test_edges(dims, prec, tol):
    from paper_1702_00124_gb300 import wdhmc as wd
    from tests import gpu_util as gu
    U = synthetic.gauge_field(dims, 0.5, 14100)
    psi = lattice.mask(synthetic.spinor_field(dims, 14101), dims, 0)
    lat = wd.Lattice(dims)
    lat.wd_gauge_load(gu.dev(U))
    out = lat.half_spinor()
    for _ in range(3):                     # a chain: early starts behind one another
        lat.mdagm_apply(0.13, prec, 1, gu.pack(lat, psi, 0), out)
    err = gu.site_rel_err(gu.unpack(lat, out, 0), wilson.apply_Khat(U, psi, 0.13), 0, dims)
    lat.close()
    assert err < tol
