"""Layout changes between lexicographic and even-odd fields: exact for every shape, with a first or last
block of fewer than 64 sites, with the even-odd side on a 16-byte boundary and between two; and
the time of algebra fields beside that of spinors.

At 16^3 x 32 an algebra field moves 2.7 times a half spinor's bytes: 13 us against 8 us; with run-time
divisors in the index arithmetic 25 against 10 us.
"""
import numpy as np
import pytest

from oracle import lattice

pytestmark = pytest.mark.gpu


def _eo(a, dims, outer):
    """Lexicographic [V, outer, chunk, c] -> even-odd [outer, 2, chunk, Vh, c]."""
    V = int(np.prod(dims))
    par = lattice.parity(dims).reshape(-1)
    cb = np.arange(V) // 2
    eo = np.zeros((outer, 2, a.shape[2], V // 2, a.shape[3]))
    for p in (0, 1):
        m = par == p
        eo[:, p][:, :, cb[m]] = a[m].transpose(1, 2, 0, 3)
    return eo


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 4, 4, 2), (6, 10, 14, 2), (10, 6, 2, 6), (8, 8, 8, 16)], ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("shift", [0, 1])
def test_exact(dims, shift):
    import torch
    from paper_1702_00124_gb300 import wdhmc as wd
    lat = wd.Lattice(dims)
    V, rng = lat.V, np.random.default_rng(10000)

    def dev(n):
        return torch.full((n + 2,), 7.0, dtype=torch.float64, device="cuda")[shift:shift + n]

    a = rng.standard_normal((V, 4, 8, 1))                      # algebra field
    src, eo, back = torch.from_numpy(a.reshape(-1)).cuda(), dev(32 * V), dev(32 * V)
    lat.wd_algebra_pack(src, eo)
    assert np.array_equal(eo.cpu().numpy(), _eo(a, dims, 4).reshape(-1))
    lat.wd_algebra_unpack(eo, back)
    assert torch.equal(back, src)
    s = rng.standard_normal((V, 1, 12, 2))                     # spinor, one parity at a time
    src = torch.from_numpy(s.reshape(-1)).cuda()
    back = dev(24 * V)
    for p in (0, 1):
        eo = dev(12 * V)
        lat.wd_spinor_pack(p, src, eo)
        assert np.array_equal(eo.cpu().numpy(), _eo(s, dims, 1)[0, p].reshape(-1))
        before = back.clone()
        lat.wd_spinor_unpack(p, eo, back)
        m = torch.from_numpy(lattice.parity(dims).reshape(-1) == p).cuda()
        assert torch.equal(back.view(V, 24)[m], src.view(V, 24)[m])
        assert torch.equal(back.view(V, 24)[~m], before.view(V, 24)[~m])
    u = torch.from_numpy(rng.standard_normal(72 * V)).cuda()   # links there and back
    lat.wd_gauge_load(u)
    back = dev(72 * V)
    lat.wd_gauge_store(back)
    assert torch.equal(back, u)
    lat.close()


def test_time_of_algebra_fields():
    import torch
    from paper_1702_00124_gb300 import wdhmc as wd
    lat = wd.Lattice((16, 16, 16, 32))
    a, A = lat.algebra_field(), lat.algebra_field()
    s = torch.zeros(24 * lat.V, dtype=torch.float64, device="cuda")
    S = lat.half_spinor()

    def least(f):
        ts = []
        for _ in range(14):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            for _ in range(20):
                f()
            e[1].record()
            torch.cuda.synchronize()
            ts.append(e[0].elapsed_time(e[1]))
        return min(ts)

    t = [least(f) for f in (lambda: lat.wd_algebra_pack(a, A), lambda: lat.wd_algebra_unpack(A, a), lambda: lat.wd_spinor_pack(0, s, S))]
    lat.close()
    print(t)
    assert max(t[:2]) < 2.1 * t[2], t
