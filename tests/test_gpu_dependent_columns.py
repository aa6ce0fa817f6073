"""Matrices with dependent columns: after a few reflectors what is left is rounding noise that falls off by sixteen digits a
column, down to squares that underflow.  The transformations stay orthogonal and the form holds (200 M eps of the norm,
as for the other stage tests), on every route of both reductions."""
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


def _matrix(kind, M):
    import torch
    ones = torch.ones(M, M, dtype=torch.float64, device="cuda")
    i = torch.arange(M, device="cuda")
    if kind == "ones":
        return ones
    if kind == "two_ones":
        s = torch.where(i < M // 2, 1.0, 1e-3).double()
        return torch.where((i[:, None] < M // 2) == (i[None, :] < M // 2), ones, 0 * ones) * s[:, None] * s[None, :]
    if kind == "rank_two":
        x = torch.linspace(-1, 1, M, dtype=torch.float64, device="cuda")
        return ones + 1e-4 * x[:, None] * x[None, :]
    return torch.where(i[:, None] // 5 == i[None, :] // 5, ones, 0 * ones)  # blocks of five equal columns


def _check(C, Q, d, e):
    import torch
    M = C.shape[0]
    T = torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1)
    n = float(torch.linalg.matrix_norm(C, 2))
    assert float((Q.t() @ Q - torch.eye(M, dtype=torch.float64, device="cuda")).abs().max()) <= 200 * M * EPS
    assert float((Q.t() @ C @ Q - T).abs().max()) <= 200 * M * EPS * n


@pytest.mark.parametrize("clusters", [True, False])
@pytest.mark.parametrize("kind", ["ones", "two_ones", "rank_two", "fives"])
@pytest.mark.parametrize("M", [40, 300, 600])
def test_one_stage(gep, M, kind, clusters):
    import torch
    h = gep.Handle()
    h.set_routes(clusters=clusters)
    C = _matrix(kind, M)
    d, e, tau, Cr = gep.tridiag_1stage(C, handle=h)
    _check(C, gep.sep_backtransform(Cr, tau, torch.eye(M, dtype=torch.float64, device="cuda"), handle=h), d, e)
    h.close()


@pytest.mark.parametrize("rows", [0, -1])
@pytest.mark.parametrize("clusters", [True, False])
@pytest.mark.parametrize("kind", ["ones", "two_ones", "rank_two", "fives"])
@pytest.mark.parametrize("M,b", [(100, 16), (200, 64), (520, 32), (900, 32), (900, 64)])
def test_two_stage(gep, M, b, kind, clusters, rows):
    import torch
    h = gep.Handle()
    h.set_routes(clusters=clusters)
    h.set_panel_qr(rows)
    C = _matrix(kind, M)
    d, e, tau1, q2, Cr = gep.tridiag_2stage(C, b, handle=h)
    _check(C, gep.sep_backtransform_2stage(Cr, tau1, q2, b, torch.eye(M, dtype=torch.float64, device="cuda"), handle=h), d, e)
    h.close()


@pytest.mark.parametrize("kind", ["ones", "falling", "rank_two", "signs"])
@pytest.mark.parametrize("M,b", [(30, 2), (130, 2), (257, 5), (400, 16), (400, 32), (700, 64)])
def test_tiles_of_reflections(gep, M, b, kind):
    """Reflectors whose tails vanish beside their first entry are reflections (-1 on the diagonal of a tile of Q2)."""
    import torch
    i = torch.arange(M, device="cuda", dtype=torch.float64)
    if kind == "falling":
        g = torch.Generator(device="cuda").manual_seed(M)
        G = torch.randn(M, M, generator=g, dtype=torch.float64, device="cuda")
        C = (G + G.t()) * torch.exp(-0.2 * (i[:, None] + i[None, :]))
    elif kind == "signs":  # a band of one subdiagonal and, b below the diagonal, entries beside which the others vanish
        C = torch.diag(torch.cos(i)) + 0.5 * torch.diag(torch.ones(M - 1, dtype=torch.float64, device="cuda"), -1)
        C = C + torch.diag(1e-14 * torch.ones(M - b, dtype=torch.float64, device="cuda"), -b)
        C = C.tril() + C.tril(-1).t()
    else:
        C = _matrix(kind, M)
    eye = torch.eye(M, dtype=torch.float64, device="cuda")
    w, Y, info = gep.solve(C, eye, sep="2stage", bandwidth=b, precision="fp64_emulated")
    assert info == 0
    n = float(torch.linalg.matrix_norm(C, 2))
    assert float((Y.t() @ Y - eye).abs().max()) <= 200 * M * EPS
    assert float((C @ Y - Y * w).abs().max()) <= 200 * M * EPS * n
