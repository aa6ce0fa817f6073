"""Routes of small pencils in a batch: one stream and many tiny pencils keep the one-CTA launch, few pencils
on many streams the staged one; both give the same eigenpairs.  Tolerances as in the batched tests (1e-11 of
the norm for eigenvalues, 1e-12 for B-orthonormality)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gep():
    import torch
    assert torch.cuda.is_available()
    from paper_1504_06443_gb300 import build
    build.build()
    import paper_1504_06443_gb300 as g
    g.load()
    return g


@pytest.mark.parametrize("count,lo,hi,nstreams", [(60, 1, 12, 1), (6, 100, 128, 8), (40, 8, 128, 2)])
def test_routes_agree(gep, count, lo, hi, nstreams):
    import torch
    g = torch.Generator(device="cuda").manual_seed(count)
    orders = [lo + (hi - lo) * i // max(count - 1, 1) for i in range(count)]
    As, Bs = [], []
    for M in orders:
        G = torch.randn(M, M, generator=g, dtype=torch.float64, device="cuda")
        H = torch.randn(M, M, generator=g, dtype=torch.float64, device="cuda")
        As.append(G + G.t())
        Bs.append(H @ H.t() / M + torch.eye(M, dtype=torch.float64, device="cuda"))
    small = gep.BatchedSolver(As, Bs, nstreams=nstreams, precision="fp64")
    staged = gep.BatchedSolver(As, Bs, nstreams=nstreams, precision="fp64", batch_small=0)
    for s in (small, staged):
        s.run()
        torch.cuda.synchronize()
        assert s.info() == 0
    for A, B, (w, Y), (w1, _) in zip(As, Bs, small.results(), staged.results()):
        n = float(torch.linalg.matrix_norm(A, 2))
        eye = torch.eye(A.shape[0], dtype=torch.float64, device="cuda")
        assert float((w - w1).abs().max()) <= 1e-11 * n
        assert float((Y.t() @ B @ Y - eye).abs().max()) <= 1e-12
        assert float((A @ Y - B @ Y * w).abs().max()) <= 1e-11 * n
