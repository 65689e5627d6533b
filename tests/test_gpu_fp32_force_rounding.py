"""Rounding of the FP32 forces against FP64.

Separately rounded complex products gave, relative to the FP64 force of the same fields, 7.17e-8 for the gauge
force and 1.00e-6 to 1.03e-6 for the Hasenbusch force at these sizes and hopping parameters, whatever
the lattice; chains of six products 7.47e-8 and 1.05e-6 to 1.09e-6.  The bounds lie 2 % above the
first, the scatter of the smaller lattice.  The polynomial term's groups of two pairs, more than eight roots in a segment
(degree 70: segments of nine, in several launches), agree with FP64 to the FP32 rounding of vectors
that its root product has made up to 10^2.6 times larger (K_hat inside [0.5, 4]): 5e-5.
"""
import pytest

pytestmark = pytest.mark.gpu


def _lattice(wd, torch, dims, a, seed):
    lat = wd.Lattice(dims)
    g = torch.Generator(device="cuda").manual_seed(seed)
    H = torch.randn(lat.V, 4, 3, 3, dtype=torch.complex128, device="cuda", generator=g)
    U = torch.linalg.matrix_exp(0.5j * a * (H + H.mH))
    U = U / torch.linalg.det(U)[..., None, None] ** (1 / 3)
    lat.wd_gauge_load(torch.view_as_real(U).contiguous().reshape(-1))
    phi = torch.randn(24 * lat.Vh, dtype=torch.float64, device="cuda", generator=g)
    return lat, phi


@pytest.mark.parametrize("dims", [(10, 14, 18, 8), (16, 16, 16, 32)], ids=lambda d: "x".join(map(str, d)))
def test_rounding(dims):
    import torch
    from paper_1702_00124_gb300 import wdhmc as wd
    lat, phi = _lattice(wd, torch, dims, 0.4, 12000)
    rel = []
    for force in (lambda p, F: lat.gauge_force(5.6, p, 1.0, F),
                  lambda p, F: lat.fermion_force(wd.term(wd.HASENBUSCH, 0.125, 0.117), phi, wd.cg_params(prec=p, tol=1e-11), 1.0, F)):
        F = [lat.algebra_field() for _ in range(2)]
        for p in (0, 1):
            force(p, F[p])
        rel.append(float((F[0] - F[1]).norm() / F[0].norm()))
    lat.close()
    print(dims, rel)
    assert rel[0] < 1.02 * 7.17e-8
    assert rel[1] < 1.02 * 1.03e-6
