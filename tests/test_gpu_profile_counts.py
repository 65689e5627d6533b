"""Sampled launches of the hop kernels (wd_profile_enable, wd_profile_read).

The force of a polynomial term consists of hops outside any solve, so with every launch sampled the
samples of a format are all its hop launches, those with the shift of a factor fused in among them.
"""
import pytest

from paper_1702_00124_gb300 import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (12, 12, 12, 20)], ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("prec,recon", [(0, 0), (1, 0), (1, 1)])
def test_every_hop_is_sampled(dims, prec, recon):
    import torch
    from paper_1702_00124_gb300 import wdhmc as wd
    from tests import gpu_util as gu
    lat = wd.Lattice(dims)
    lat.wd_gauge_load(gu.dev(synthetic.gauge_field(dims, 0.3, 13000)))
    lat.wd_set_recon(recon)
    phi = torch.randn(24 * lat.Vh, dtype=torch.float64, device="cuda")
    F = lat.algebra_field()
    lat.wd_profile_enable(1)
    lat.fermion_force(wd.term(wd.POLY, 0.1, poly=(6, 0.05, 6.0)), phi, wd.cg_params(prec=prec), 1.0, F)
    got = lat.wd_profile_read(prec)
    n = lat.wd_hop_counts()[prec]
    lat.wd_profile_enable(0)
    lat.close()
    assert got["launches"] == n > 0
    assert got["ms"] > 0.0
    link = 144 if prec == 0 else 48 if recon else 72
    spinor = 192 if prec == 0 else 96
    per = 8 * link + 2 * spinor
    # in, out and links at least; y in half of the launches or more, v in some
    assert n * per * lat.Vh < got["bytes"] < n * (per + 2 * spinor) * lat.Vh
