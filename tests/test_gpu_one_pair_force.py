"""Outer products of one (Y, X) pair in FP32: the force of a plain or Hasenbusch term.

One thread per site from one block of 128 per SM on (V >= 128 x 152), a warp per direction below: values
on either side of the line and with ragged last blocks against FP64, and its time.
Tolerance: an entry of A sums 16 real products, U A six, the projection four, each rounded at 2^-24
(1.5e-6 of the sum of magnitudes); cancellation in the traceless anti-Hermitian part of random
fields costs a factor of two to three: 5e-6.
"""
import numpy as np
import pytest

from paper_1702_00124_gb300 import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(4, 4, 4, 2), (6, 10, 14, 2), (8, 8, 16, 18), (16, 8, 8, 20), (10, 14, 18, 10)], ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("kind", ["plain", "hasenbusch"])
def test_fp32_against_fp64(dims, kind):
    import torch
    from paper_1702_00124_gb300 import wdhmc as wd
    from tests import gpu_util as gu
    lat = wd.Lattice(dims)
    lat.wd_gauge_load(gu.dev(synthetic.gauge_field(dims, 0.5, 7000)))
    g = torch.Generator(device="cuda").manual_seed(7001)
    phi, X, Y = (torch.randn(24 * lat.Vh, dtype=torch.float64, device="cuda", generator=g) for _ in range(3))
    t = wd.term(wd.PLAIN, 0.13) if kind == "plain" else wd.term(wd.HASENBUSCH, 0.13, 0.12)
    F = []
    for prec in (wd.F64, wd.F32):
        F.append(torch.ones(64 * lat.Vh, dtype=torch.float64, device="cuda"))     # added to
        lat.fermion_force_xy(t, phi, X, Y, prec, 0.7, F[-1])
    a, b = ((f - 1.0).cpu().numpy() for f in F)
    lat.close()
    assert np.linalg.norm(a - b) < 5e-6 * np.linalg.norm(a)


def test_time_against_khat():
    """Two conversions, two hops and the outer products: about 1.5 K_hat (four hops) at 24^4, 2.1 with
    a warp per direction."""
    import torch
    from paper_1702_00124_gb300 import wdhmc as wd
    lat = wd.Lattice((24, 24, 24, 24))
    U = torch.eye(3, dtype=torch.complex128, device="cuda").expand(lat.V, 4, 3, 3).contiguous()
    lat.wd_gauge_load(torch.view_as_real(U).reshape(-1))
    x = torch.ones(24 * lat.Vh, dtype=torch.float64, device="cuda")
    out, F = lat.half_spinor(), lat.algebra_field()
    t = wd.term(wd.PLAIN, 0.13)

    def least(f):
        ts = []
        for _ in range(12):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            for _ in range(8):
                f()
            e[1].record()
            torch.cuda.synchronize()
            ts.append(e[0].elapsed_time(e[1]))
        return min(ts)

    khat = least(lambda: lat.mdagm_apply(0.13, wd.F32, 1, x, out))
    force = least(lambda: lat.fermion_force_xy(t, x, x, x, wd.F32, 1.0, F))
    lat.close()
    assert force < 1.8 * khat, (force, khat)
