"""Full to band at b <= 32 with panels in one cluster: orders at the edges of the rows a warp (256, 512,
1024, 2048 below the first panel), of the panel (b - 1, b, b + 1 rows left), ragged b, and panels with zero, tiny,
graded or dependent columns.  Q^T C Q must be the band matrix: eigenvalues and orthogonality of the two-stage
route against a library eigensolver, 200 M eps of the norm as for the other stage tests."""
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


def _symmetric(M, seed):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    G = torch.randn(M, M, generator=g, dtype=torch.float64, device="cuda")
    return G + G.t()


def _check(gep, C, b):
    import torch
    M = C.shape[0]
    eye = torch.eye(M, dtype=torch.float64, device="cuda")
    w, Y, info = gep.solve(C, eye, precision="fp64_emulated", sep="2stage", bandwidth=b)
    assert info == 0
    n = float(torch.linalg.matrix_norm(C, 2))
    ref = torch.linalg.eigvalsh(C.cpu()).cuda()
    assert float((w - ref).abs().max()) <= 200 * M * EPS * n
    assert float((Y.t() @ Y - eye).abs().max()) <= 200 * M * EPS
    assert float((C @ Y - Y * w).abs().max()) <= 200 * M * EPS * n


@pytest.mark.parametrize("M,b", [(33, 32), (34, 32), (65, 32), (96, 31), (130, 7), (288, 32), (289, 32), (545, 32),
                                 (1057, 32), (2080, 32), (2082, 32)])
def test_orders(gep, M, b):
    _check(gep, _symmetric(M, M), b)


@pytest.mark.parametrize("kind", ["zero_block", "rank_one", "graded", "tiny_columns", "banded"])
def test_degenerate_panels(gep, kind):
    import torch
    M = 400
    S = _symmetric(M, 3)
    i = torch.arange(M, device="cuda")
    if kind == "zero_block":
        S[200:, :200] = 0
        S[:200, 200:] = 0
    elif kind == "rank_one":
        u = torch.linspace(1, 2, M, dtype=torch.float64, device="cuda")
        S = u[:, None] * u[None, :] + torch.diag(1e-3 * i.double())
    elif kind == "graded":
        s = torch.exp(torch.linspace(0, -40, M, dtype=torch.float64, device="cuda"))
        S = S * s[:, None] * s[None, :]
    elif kind == "tiny_columns":
        s = torch.where(i % 3 == 0, 1e-12, 1.0).double()
        S = S * s[:, None] * s[None, :]
    else:
        S = torch.where((i[:, None] - i[None, :]).abs() <= 5, S, torch.zeros_like(S))
    _check(gep, S, 32)
