"""The polynomial term's force, whose roots go out a segment at a time.

Degree 16: four segments of four roots; degree 70: segments of nine, which take two
launches each (at most eight roots a launch) and a last segment of seven.  Lattices of
one and of ragged blocks of 32 sites.  Tolerances (relative, Frobenius): the root
product on [0.5, 4] passes through vectors 10^2.2 (degree 16) and 10^9.2 (degree 70)
times larger than its result (largest partial product times what follows it, over the
interval), which multiplies the rounding: FP64 1e-9 and 1e-4, FP32 5e-5.
"""
import numpy as np
import pytest

from oracle import actions, force, lattice
from oracle.poly import ChebyshevFilter
from paper_1702_00124_gb300 import synthetic

pytestmark = pytest.mark.gpu

KAPPA = 0.06      # spectrum of K_hat inside the filter's interval


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (2, 6, 4, 6)], ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("n,prec,tol", [(16, 0, 1e-9), (16, 1, 5e-5), (70, 0, 1e-4)])
def test_poly_force(dims, n, prec, tol):
    from paper_1702_00124_gb300 import wdhmc as wd
    from tests import gpu_util as gu
    poly = (n, 0.5, 4.0)
    U = synthetic.gauge_field(dims, 0.5, 900 + n)
    phi = lattice.mask(synthetic.spinor_field(dims, 901 + n), dims, 0)
    ref = force.fermion_force(U, actions.term("poly", KAPPA, poly=ChebyshevFilter(*poly)), phi)
    lat = wd.Lattice(dims)
    lat.wd_gauge_load(gu.dev(U))
    F = lat.algebra_field()
    lat.fermion_force(wd.term(wd.POLY, KAPPA, poly=poly), gu.pack(lat, phi, 0), wd.cg_params(prec=prec), -2.0, F)
    got = gu.alg_to_host(lat, F) / -2.0
    lat.close()
    assert np.linalg.norm(got - ref) < tol * np.linalg.norm(ref)
