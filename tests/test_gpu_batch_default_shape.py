"""The batched K_hat in its default shape (128 items, one right-hand side per thread) on 18-real links.

It reads the links once per right-hand side where a lattice's own K_hat reads them once in all, but
fills the GPU with all lattices at once: 3 x 12^3 x 24 with two sides took 150 us with separately
rounded products, 164 us with one chain of six per component, 142 us with two chains of three.  Six
K_hat of a single 12^3 x 24 lattice with 18-real links take 128 us, unchanged by the shape.  Values
against the lattice's own FP32 K_hat: eight directions with 36 products each, 2e-6 relative.
"""
import pytest

pytestmark = pytest.mark.gpu


def test_default_shape():
    import torch
    from paper_1702_00124_gb300 import synthetic
    from paper_1702_00124_gb300 import wdhmc as wd
    from tests import gpu_util as gu
    dims, nr = (12, 12, 12, 24), 2
    U = gu.dev(synthetic.gauge_field(dims, 0.5, 8000))
    lats = [wd.Lattice(dims) for _ in range(3)]
    for lat in lats:
        lat.wd_gauge_load(U)
    torch.cuda.synchronize()
    batch = wd.Batch(lats, [0.13] * 3, [nr] * 3)
    g = torch.Generator(device="cuda").manual_seed(8001)
    xs = [torch.randn(24 * nr * lat.Vh, dtype=torch.float64, device="cuda", generator=g) for lat in lats]
    ys = [torch.zeros_like(x) for x in xs]
    ref = [torch.zeros_like(x) for x in xs]

    def single():
        for lat, x, r in zip(lats, xs, ref):
            lat.mdagm_apply(0.13, wd.F32, nr, x, r)

    def least(f):
        ts = []
        for _ in range(14):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            for _ in range(10):
                f()
            e[1].record()
            torch.cuda.synchronize()
            ts.append(e[0].elapsed_time(e[1]))
        return min(ts)

    t = least(lambda: batch.wd_batch_mdagm(xs, ys)), least(single)
    for y, r in zip(ys, ref):
        assert (y - r).norm() < 2e-6 * r.norm()
    batch.close()
    for lat in lats:
        lat.close()
    print(t)
    assert t[0] < 1.21 * t[1], t
