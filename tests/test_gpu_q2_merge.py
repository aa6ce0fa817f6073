"""Back-transformation with merged Q2 tiles: one level from 2560, two from 6000 rows on, with odd numbers of
tiles in a row and of rows, and a last tile of a few rows.  Residual and orthogonality of a standard problem
at the tolerances of the other two-stage tests (200 M eps)."""
import pytest

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52


@pytest.fixture(scope="module")
def gep():
    import torch
    assert torch.cuda.is_available()
    from paper_1504_06443_gb300 import build
    build.build()
    import paper_1504_06443_gb300 as g
    g.load()
    return g


@pytest.mark.parametrize("M,b,n_want", [(2560, 32, 0), (2562, 64, 0), (2817, 32, 2100), (3329, 64, 0), (3000, 48, 0),
                                        (6001, 32, 0), (6145, 64, 2048)])
def test_merged_tiles(gep, M, b, n_want):
    import torch
    g = torch.Generator(device="cuda").manual_seed(M)
    A = torch.randn(M, M, generator=g, dtype=torch.float64, device="cuda")
    A = A + A.t()
    eye = torch.eye(M, dtype=torch.float64, device="cuda")
    w, Y, info = gep.solve(A, eye, precision="fp64_emulated", sep="2stage", bandwidth=b, n_want=n_want)
    assert info == 0
    norm = float(torch.linalg.vector_norm(A)) / M ** 0.5  # about half of the 2-norm
    n = Y.shape[1]
    assert float((Y.t() @ Y - eye[:n, :n]).abs().max()) <= 200 * M * EPS
    assert float((A @ Y - Y * w[:n]).abs().max()) <= 200 * M * EPS * norm
