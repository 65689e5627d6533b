"""Sums that overflow are infinite, not NaN.

The action of the polynomial term on phi, P close to a multiple of one: every term of
<phi, P phi> is positive.  phi is scaled so that the sum lies below FP64's largest number,
above it in the last addition only, and above it in every block.
"""
import math

import numpy as np
import pytest

from paper_1702_00124_gb300 import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (8, 8, 8, 16)], ids=lambda d: "x".join(map(str, d)))
def test_overflowing_action(dims):
    from paper_1702_00124_gb300 import wdhmc as wd
    from tests import gpu_util as gu
    lat = wd.Lattice(dims)
    lat.wd_gauge_load(gu.dev(synthetic.gauge_field(dims, 0.3, 6000)))
    rng = np.random.default_rng(6001)
    # all components of one size: no block's sum overflows before the last
    phi = gu.dev(np.sign(rng.standard_normal(24 * lat.Vh)))
    t = wd.term(wd.POLY, 0.005, poly=(8, 0.5, 4.0))
    one = lat.pf_action(t, phi, wd.cg_params())
    assert one > 0.0
    for total in (1e300, 1.5e308):
        s = math.sqrt(total / one)
        S = lat.pf_action(t, s * phi, wd.cg_params())
        assert abs(S / one / s / s - 1.0) < 1e-12
    for scale in (math.sqrt(1.7e308) * math.sqrt(1.4 / one), 1e154, 1e160):
        assert lat.pf_action(t, scale * phi, wd.cg_params()) == math.inf
    lat.close()
