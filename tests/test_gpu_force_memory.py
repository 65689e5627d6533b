"""Device memory of the polynomial term's force.

The force of degree m walks its root product with square-root checkpoints: with
seg = ceil(sqrt(m)) and nseg = ceil(m / seg) it holds nseg + 4 seg + 7 vectors and three
more while K_hat is applied, however many roots share a launch.  The term adds the
FP64 solution and a copy of phi.  Nothing beyond may stay with the context, so that the
calls after a force find the memory that they found without the grouping of roots.
"""
import math

import pytest

from paper_1702_00124_gb300 import synthetic

pytestmark = pytest.mark.gpu

DIMS = (16, 16, 16, 32)      # FP32 vectors of 6 MiB, FP64 of 12 MiB: whole allocation pages of 2 MiB


@pytest.mark.parametrize("m", [2, 16, 24, 70])
@pytest.mark.parametrize("prec", [0, 1])
def test_poly_force_memory(m, prec):
    import torch
    from paper_1702_00124_gb300 import wdhmc as wd
    g = torch.Generator(device="cuda").manual_seed(m)
    U = torch.view_as_real(torch.eye(3, dtype=torch.complex128, device="cuda").expand(32 * 16 ** 3, 4, 3, 3).contiguous()).reshape(-1)
    for run in range(2):         # the first run loads the kernels' code, which takes device memory too
        lat = wd.Lattice(DIMS)
        lat.wd_gauge_load(U)
        phi = torch.randn(24 * lat.Vh, dtype=torch.float64, device="cuda", generator=g)
        F = lat.algebra_field()
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        lat.fermion_force(wd.term(wd.POLY, 0.1, poly=(m, 0.05, 6.0)), phi, wd.cg_params(prec=prec), 1.0, F)
        torch.cuda.synchronize()
        used = free - torch.cuda.mem_get_info()[0]
        vh = lat.Vh
        lat.close()
    seg = math.ceil(math.sqrt(m))
    nseg = math.ceil(m / seg)
    vec = 24 * vh * (8 if prec == 0 else 4)
    # the term's own: one FP64 vector and one of the force's format
    assert 0 < used <= (nseg + 4 * seg + 7 + 3 + 1) * vec + 24 * vh * 8
