"""Whole solves of pencils whose norm is far from one: eigenvalues relative to it, residual and B-orthonormality do not depend
on the power of two A (or B) is multiplied with.  Tolerances of the whole-solve tests: 1e-11 of the norm, residual
1e-13 of ||A||_F M, orthonormality 1e-12."""
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


@pytest.fixture(scope="module")
def pencils():
    import torch
    out = {}
    for M in (60, 300, 700):
        g = torch.Generator().manual_seed(M)
        G, H = (torch.randn(M, M, generator=g, dtype=torch.float64) for _ in range(2))
        A, B = G + G.t(), H @ H.t() / M + torch.eye(M, dtype=torch.float64)
        L = torch.linalg.cholesky(B)
        C = torch.linalg.solve_triangular(L, torch.linalg.solve_triangular(L, A, upper=False).t(), upper=False)
        out[M] = A.cuda(), B.cuda(), torch.linalg.eigvalsh((C + C.t()) / 2).cuda()
    return out


@pytest.mark.parametrize("route", [("1stage", "fp64_emulated", "twosided"), ("2stage", "fp64_emulated", "twosided"),
                                   ("2stage", "fp64_emulated", "explicit_inv"), ("1stage", "mixed_refined", "twosided"),
                                   ("2stage", "mixed_refined", "twosided"), ("1stage", "fp64_emulated", "eigenexa"),
                                   ("1stage", "fp64", "twosided"), ("2stage", "fp64", "twosided")])
@pytest.mark.parametrize("M", [60, 300, 700])
@pytest.mark.parametrize("pa,pb", [(0, 0), (40, 0), (-40, 0), (13, 0), (-60, -30), (20, 16), (300, 0), (-300, 0)])
def test_scaled_pencil(gep, pencils, M, pa, pb, route):
    import torch
    A, B, ref = pencils[M]
    sep, precision, reducer = route
    As, Bs = A * 2.0 ** pa, B * 2.0 ** pb
    w, Y, info = gep.solve(As, Bs, sep=sep, precision=precision, reducer=reducer)
    assert info == 0
    n = float(ref.abs().max())
    w, Y = w * 2.0 ** (pb - pa), Y * 2.0 ** (pb / 2)
    assert float((w - ref).abs().max()) <= 1e-11 * n
    assert float((Y.t() @ B @ Y - torch.eye(M, dtype=torch.float64, device="cuda")).abs().max()) <= 1e-12
    assert float((A @ Y - B @ Y * w).norm() / (A.norm() * M)) <= 1e-13


@pytest.mark.parametrize("sep", ["1stage", "2stage"])
@pytest.mark.parametrize("pa", [40, -40])
def test_scaled_values_lowest_and_overwritten(gep, pencils, pa, sep):
    A, B, ref = pencils[700]
    n = float(ref.abs().max())
    w, _, info = gep.solve(A * 2.0 ** pa, B, sep=sep, precision="fp64_emulated", want_vectors=False)
    assert info == 0 and float((w * 2.0 ** -pa - ref).abs().max()) <= 1e-11 * n
    w, Y, info = gep.solve(A * 2.0 ** pa, B, sep=sep, precision="fp64_emulated", n_want=90)
    assert info == 0 and float((w * 2.0 ** -pa - ref[:90]).abs().max()) <= 1e-11 * n
    assert float((A @ Y - B @ Y * (w * 2.0 ** -pa)).norm() / (A.norm() * 700)) <= 1e-13
    w, Y, info = gep.solve(A * 2.0 ** pa, B.clone(), sep=sep, precision="fp64_emulated", overwrite=True)
    assert info == 0 and float((w * 2.0 ** -pa - ref).abs().max()) <= 1e-11 * n


@pytest.mark.parametrize("precision", ["fp64", "fp64_emulated"])
@pytest.mark.parametrize("sep,b", [("1stage", 0), ("2stage", 0), ("2stage", 48), ("2stage", 64)])
@pytest.mark.parametrize("M", [300, 700])
@pytest.mark.parametrize("p", [-660, 660])
def test_squares_beyond_the_range(gep, pencils, M, p, sep, b, precision):
    """Norms whose squares over- or underflow, with B = I."""
    import torch
    A = pencils[M][0]
    ref = torch.linalg.eigvalsh(A.cpu()).cuda()
    eye = torch.eye(M, dtype=torch.float64, device="cuda")
    n = float(ref.abs().max())
    w, Y, info = gep.solve(A * 2.0 ** p, eye, sep=sep, bandwidth=b, precision=precision)
    assert info == 0
    assert float((w * 2.0 ** -p - ref).abs().max()) <= 1e-11 * n
    assert float((Y.t() @ Y - eye).abs().max()) <= 1e-12
    assert float((gep.solve(A * 2.0 ** p, eye, sep=sep, bandwidth=b, precision=precision, want_vectors=False)[0] * 2.0 ** -p
                  - ref).abs().max()) <= 1e-11 * n


def test_no_further_off_than_unscaled(gep):
    """A dense pencil with known eigenpairs, eigenvalues in [-20, 20]: unscaled, the eigenvectors at order 8192 are
    1.02e-12 off (relative, Frobenius; 2 % between seeds); a tenth above that is allowed."""
    import importlib.util
    import pathlib
    spec = importlib.util.spec_from_file_location(
        "planted", pathlib.Path(__file__).resolve().parents[1] / "perf" / "cases.py")
    planted = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(planted)
    A, B = planted._pencil(8192, 1)
    w, Y, info = gep.solve(A, B, sep="2stage", precision="fp64_emulated", reducer="twosided")
    assert info == 0
    del A, B
    lam, Y0 = planted._eigenpairs(8192, 1)
    Y = Y.gather(0, Y.abs().argmax(0, keepdim=True)).sign() * Y
    Y0 = Y0.gather(0, Y.abs().argmax(0, keepdim=True)).sign() * Y0
    assert float((w - lam).norm() / lam.norm()) <= 1.25e-15
    assert float((Y - Y0).norm() / Y0.norm()) <= 1.1 * 1.02e-12
