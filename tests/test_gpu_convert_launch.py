"""A 16-bit hop between FP64 fields at 16^3 x 32.

Three kernels: FP64 to 16 bits site by site, the hop, 16 bits to FP64.  With the last one site by
site too, early starts piled its blocks up on some SMs: 23 to 29 us, 1.9 to 2.2 times the FP32 hop
(13 us); word by word it takes 20 us, 1.6 times.
"""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [2, 3])
def test_time_against_fp32(prec):
    import torch
    from paper_1702_00124_gb300 import wdhmc as wd
    lat = wd.Lattice((16, 16, 16, 32))
    U = torch.eye(3, dtype=torch.complex128, device="cuda").expand(lat.V, 4, 3, 3).contiguous()
    lat.wd_gauge_load(torch.view_as_real(U).reshape(-1))
    lat.wd_set_recon(1)
    x = torch.ones(24 * lat.Vh, dtype=torch.float64, device="cuda")
    out = lat.half_spinor()

    def least(p):
        ts = []
        for _ in range(14):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            for _ in range(20):
                lat.wd_hop(1, 0, p, x, out)
            e[1].record()
            torch.cuda.synchronize()
            ts.append(e[0].elapsed_time(e[1]) * 50)
        return min(ts)

    t = least(prec), least(1)
    lat.close()
    print(t)
    assert t[0] < 1.75 * t[1], t
