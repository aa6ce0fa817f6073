"""One-launch panels of the 1-stage tridiagonalisation: orders at the edges of the tiles (32 and 64
wide), of the panels (64 columns) and of the rules (768: tile size; tiles that no longer stay in
shared memory; 4096: the per-column kernels take the first panels).  Reference: a library
eigensolver; tolerances as for the other stage tests (200 M eps of the norm)."""
import numpy as np
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


@pytest.mark.parametrize("M", [1, 2, 3, 31, 32, 33, 63, 64, 65, 66, 95, 97, 129, 193, 767, 769, 833])
def test_tridiagonal_form(gep, oracle_lib, M):
    import torch
    C = _symmetric(M, M)
    d, e, tau, Cr = gep.tridiag_1stage(C)
    Q = gep.sep_backtransform(Cr, tau, torch.eye(M, dtype=torch.float64, device="cuda"))
    T = torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1)
    n = float(torch.linalg.matrix_norm(C, 2))
    eye = torch.eye(M, dtype=torch.float64, device="cuda")
    assert float((Q.t() @ Q - eye).abs().max()) <= 200 * M * EPS
    assert float((Q.t() @ C @ Q - T).abs().max()) <= 200 * M * EPS * n


@pytest.mark.parametrize("C", ["zero", "diagonal", "banded", "tiny", "huge"])
def test_degenerate_columns(gep, C):
    import torch
    M = 150
    S = _symmetric(M, 9)
    i = torch.arange(M, device="cuda")
    C = {"zero": torch.zeros_like(S), "diagonal": torch.diag(i.double()), "tiny": S * 1e-140, "huge": S * 1e140,
         "banded": torch.where((i[:, None] - i[None, :]).abs() <= 2, S, torch.zeros_like(S))}[C]
    d, e, tau, Cr = gep.tridiag_1stage(C)
    Q = gep.sep_backtransform(Cr, tau, torch.eye(M, dtype=torch.float64, device="cuda"))
    T = torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1)
    n = float(C.abs().max()) * M
    assert bool(torch.isfinite(T).all())
    assert float((Q.t() @ C @ Q - T).abs().max()) <= 200 * M * EPS * n + 1e-300


@pytest.mark.parametrize("precision", ["fp64_emulated", "mixed_refined"])
@pytest.mark.parametrize("M", [130, 770, 2700, 4160])
def test_tensor_core_engines(gep, M, precision):
    import torch
    A = _symmetric(M, M)
    B = torch.eye(M, dtype=torch.float64, device="cuda")
    w, Y, info = gep.solve(A, B, precision=precision, sep="1stage")
    assert info == 0
    ref = torch.linalg.eigvalsh(A)
    n = float(ref.abs().max())
    assert float((w - ref).abs().max()) <= 1e-11 * n
    assert float((Y.t() @ Y - B).abs().max()) <= 1e-12
    assert float((A @ Y - Y * w).norm() / (A.norm() * M)) <= 1e-13
