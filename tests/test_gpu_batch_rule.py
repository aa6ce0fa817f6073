"""Route of small pencils in a batch, seen in the number of kernels: one persistent launch where it measured faster than
the streams, whose time is their share of a stream but never less than the largest pencil's alone."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("orders,nstreams,one_cta", [
    ([8], 8, True), ([10] * 8, 64, True), ([4] * 4, 8, True), ([16] * 16, 8, True), ([24] * 64, 8, True), ([28] * 4, 1, True),
    ([24], 1, False), ([28], 1, False), ([24] * 4, 8, False), ([64], 8, False), ([128] * 2, 8, False)])
def test_route(orders, nstreams, one_cta):
    import torch
    from paper_1504_06443_gb300 import build
    build.build()
    import paper_1504_06443_gb300 as gep
    g = torch.Generator(device="cuda").manual_seed(sum(orders))
    As, Bs = [], []
    for M in orders:
        G = torch.randn(M, M, generator=g, dtype=torch.float64, device="cuda")
        As.append(G + G.t())
        Bs.append(torch.eye(M, dtype=torch.float64, device="cuda"))
    s = gep.BatchedSolver(As, Bs, nstreams=nstreams, precision="fp64")
    s.h.launches(reset=True)
    s.run()
    torch.cuda.synchronize()
    assert s.info() == 0
    n = s.h.launches(reset=True)
    assert n <= 2 if one_cta else n >= 20 * len(orders)
    for A, (w, _) in zip(As, s.results()):
        ref = torch.linalg.eigvalsh(A)
        assert float((w - ref).abs().max()) <= 1e-11 * float(ref.abs().max())
    s.close()
