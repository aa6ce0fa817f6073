"""Tridiagonalisation of trailing matrices of order <= 512 by one cluster: orders at the edges of the
cluster sizes (16, 32, 64, 128), of the rows a warp (256) and of the range (512), columns whose CTAs have no
rows left, and many launches at once.  Tolerances as for the other stage tests (200 M eps of the norm)."""
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


def _check(gep, C, tol):
    import torch
    M = C.shape[0]
    d, e, tau, Cr = gep.tridiag_1stage(C)
    eye = torch.eye(M, dtype=torch.float64, device="cuda")
    Q = gep.sep_backtransform(Cr, tau, eye)
    T = torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1)
    assert bool(torch.isfinite(T).all())
    assert float((Q.t() @ Q - eye).abs().max()) <= 200 * M * EPS
    assert float((Q.t() @ C @ Q - T).abs().max()) <= tol


@pytest.mark.parametrize("M", [4, 15, 16, 17, 47, 127, 128, 255, 256, 257, 300, 511, 512, 513, 577])
def test_tridiagonal_form(gep, M):
    import torch
    C = _symmetric(M, M)
    _check(gep, C, 200 * M * EPS * float(torch.linalg.matrix_norm(C, 2)))


@pytest.mark.parametrize("kind", ["zero", "diagonal", "banded", "tiny", "huge", "graded", "one_large"])
@pytest.mark.parametrize("M", [40, 500])
def test_degenerate_columns(gep, M, kind):
    import torch
    S = _symmetric(M, 9)
    i = torch.arange(M, device="cuda")
    s = torch.exp(torch.linspace(0, -60, M, dtype=torch.float64, device="cuda"))
    one = S * 1e-14
    one[M // 2, M // 3] = one[M // 3, M // 2] = 1.0
    C = {"zero": torch.zeros_like(S), "diagonal": torch.diag(i.double()), "tiny": S * 1e-300, "huge": S * 1e300,
         "banded": torch.where((i[:, None] - i[None, :]).abs() <= 2, S, torch.zeros_like(S)),
         "graded": S * s[:, None] * s[None, :], "one_large": one}[kind]
    scale = float(C.abs().max()) or 1.0
    _check(gep, C / scale if kind == "huge" else C, 200 * M * EPS * M * (1.0 if kind == "huge" else scale) + 1e-305)
    if kind == "huge":  # (the check's own products would overflow)
        d, e, _, _ = gep.tridiag_1stage(C)
        d1, e1, _, _ = gep.tridiag_1stage(C * 2.0 ** -997)
        assert torch.equal(d * 2.0 ** -997, d1) and torch.equal(e * 2.0 ** -997, e1)


def test_many_at_once(gep):
    """Concurrent clusters on several streams: integer sums, so every run gives the same bits.  The last
    columns have fewer rows than CTAs, where a CTA without rows must not fall behind the others."""
    import torch
    orders = [192, 160, 140, 116, 80, 500]
    mats = [_symmetric(M, M) for M in orders]
    eye = [torch.eye(M, dtype=torch.float64, device="cuda") for M in orders]
    solver = gep.BatchedSolver([m for m in mats for _ in range(4)], [b for b in eye for _ in range(4)], nstreams=8,
                               precision="fp64", batch_small=0)
    ref = None
    for _ in range(25):
        solver.run()
        torch.cuda.synchronize()
        assert solver.info() == 0
        w = [r[0].clone() for r in solver.results()]
        for q, M in enumerate(orders):
            assert all(torch.equal(w[4 * q], w[4 * q + u]) for u in range(1, 4))
        ref = ref or w
        assert all(torch.equal(a, b) for a, b in zip(ref, w))


@pytest.mark.parametrize("M", [9, 17, 40])
def test_nonfinite_tridiagonal_is_a_failure(gep, M):
    """A NaN or an infinity in the last entry, alone in its leaf for M = 9 and 17: reported, not ordered."""
    import torch
    h = gep.Handle()  # (the status stays with the handle until its next reset)
    for bad in (float("nan"), float("inf")):
        d = torch.linspace(0, 1, M, dtype=torch.float64, device="cuda")
        e = torch.full((M - 1,), 0.25, dtype=torch.float64, device="cuda")
        d[M - 1] = bad
        assert gep.tridiag_eig(d, e, handle=h)[2] != 0
    h.close()
