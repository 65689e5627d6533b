"""The pipeline's depth for FP32 spinors on 18-real links beyond one wave of blocks.

Four link directions and three blocks per SM; with the depths chosen as for 12 reals the Chebyshev
filter of degree 8 took 1.62 times the 12-real one at 18 x 22 x 20 x 26 (805 blocks) and 1.39 times at
24^3 x 48, where it takes 1.48 and 1.26 times (both figures against the 12-real filter with products in two chains).  Values: against the 12-real links of the same
SU(3) field, eight K_hat of FP32 rounding apart (8 x 2e-5 bounds the recurrence's steps).
"""
import pytest

from paper_1702_00124_gb300 import synthetic

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,most", [((18, 22, 20, 26), 1.55), ((24, 24, 24, 48), 1.33)], ids=str)
def test_filter_against_12_reals(dims, most):
    import torch
    from paper_1702_00124_gb300 import wdhmc as wd
    from tests import gpu_util as gu
    lat = wd.Lattice(dims)
    lat.wd_gauge_load(gu.dev(synthetic.gauge_field(dims, 0.4, 9000)))
    x = torch.randn(24 * lat.Vh, dtype=torch.float64, device="cuda", generator=torch.Generator(device="cuda").manual_seed(9001))
    out, t = [], []
    for recon in (0, 1):
        lat.wd_set_recon(recon)
        out.append(lat.half_spinor())
        ts = []
        for _ in range(10):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            for _ in range(4):
                lat.poly_filter_apply(0.12, (8, 0.05, 6.0), 1, x, out[-1])
            e[1].record()
            torch.cuda.synchronize()
            ts.append(e[0].elapsed_time(e[1]))
        t.append(min(ts))
    lat.close()
    print(dims, t)
    assert (out[0] - out[1]).norm() < 8 * 2e-5 * out[0].norm()
    assert t[0] < most * t[1], t
