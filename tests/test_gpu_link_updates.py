"""An operator called right behind a change of the links uses the new links.

The stencils read links before they wait for the kernels ahead of them, so the first
launch behind a link write must not start early.  Two gauge fields are loaded in
turn, and a field is moved back and forth by step_T, with K_hat queued at once each time
and no wait in between; the results must be bit for bit those of K_hat called after a
synchronisation on the same links.  The same where the call in between is recorded
by a stream capture and runs later.
"""
import numpy as np
import pytest

from paper_1702_00124_gb300 import synthetic

pytestmark = pytest.mark.gpu

# eight threads per site; the staged pipeline at its deepest and at four blocks per SM
LATS = [(4, 4, 4, 4), (8, 8, 8, 16), (12, 12, 12, 24), (20, 20, 20, 18)]
PRECS = [(0, 0), (1, 0), (1, 1), (3, 1), (4, 0)]     # (precision, link storage)


@pytest.fixture(scope="module", params=LATS, ids=lambda d: "x".join(map(str, d)))
def setup(request):
    import torch
    from paper_1702_00124_gb300 import wdhmc as wd
    from tests import gpu_util as gu
    dims = request.param
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        U = [gu.dev(synthetic.gauge_field(dims, 0.5, 5000 + k)) for k in range(2)]
        lat = wd.Lattice(dims, stream)
        x = gu.pack(lat, synthetic.spinor_field(dims, 5100), 0)
        yield torch, wd, gu, dims, lat, U, x, stream
        lat.close()


@pytest.mark.parametrize("prec,recon", PRECS)
def test_loads_in_turn(setup, prec, recon):
    torch, wd, gu, dims, lat, U, x, stream = setup
    lat.wd_set_recon(recon)
    ref = []
    for u in U:
        lat.wd_gauge_load(u)
        torch.cuda.synchronize()
        ref.append(lat.half_spinor())
        lat.mdagm_apply(0.13, prec, 1, x, ref[-1])
        torch.cuda.synchronize()
    outs = [lat.half_spinor() for _ in range(12)]
    torch.cuda.synchronize()
    for k, out in enumerate(outs):
        lat.wd_gauge_load(U[k % 2])
        lat.mdagm_apply(0.13, prec, 1, x, out)
    torch.cuda.synchronize()
    lat.wd_set_recon(0)
    assert not torch.equal(ref[0], ref[1])
    for k, out in enumerate(outs):
        assert torch.equal(out, ref[k % 2]), k


@pytest.mark.parametrize("prec,recon", PRECS)
def test_link_updates(setup, prec, recon):
    torch, wd, gu, dims, lat, U, x, stream = setup
    rng = np.random.default_rng(5200)
    P = gu.dev(rng.standard_normal(64 * lat.Vh))
    lat.wd_set_recon(recon)
    runs = []
    for wait in (True, False):
        lat.wd_gauge_load(U[0])
        outs = [lat.half_spinor() for _ in range(8)]
        torch.cuda.synchronize()
        for k, out in enumerate(outs):
            lat.step_T(P, 0.3 if k % 2 == 0 else -0.2)
            if wait:
                torch.cuda.synchronize()
            lat.mdagm_apply(0.13, prec, 1, x, out)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        runs.append(outs)
    lat.wd_set_recon(0)
    for k, (a, b) in enumerate(zip(*runs)):
        assert torch.equal(a, b), k
        assert k == 0 or not torch.equal(a, runs[0][k - 1]), k


def test_capture_between_load_and_call(setup):
    torch, wd, gu, dims, lat, U, x, stream = setup
    ref = []
    for u in U:
        lat.wd_gauge_load(u)
        torch.cuda.synchronize()
        ref.append(lat.half_spinor())
        lat.mdagm_apply(0.13, 1, 1, x, ref[-1])
        torch.cuda.synchronize()
    a, b = lat.half_spinor(), lat.half_spinor()
    graph = torch.cuda.CUDAGraph()
    lat.wd_gauge_load(U[0])
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream, capture_error_mode="thread_local"):
        lat.mdagm_apply(0.13, 1, 1, x, a)
    for k in (1, 0, 1):
        lat.wd_gauge_load(U[k])
        lat.mdagm_apply(0.13, 1, 1, x, b)
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(b, ref[k])
        assert torch.equal(a, ref[k])
