"""Bulge chasing at the widths of the fixed-point kernel (b = 32 and 64): orders at the edges of
its blocks, scales near both ends of the FP64 range, matrices that fill its norm bound, and the
failure path of its waits.  The reduced spectrum is held to the tolerance of the other two-stage
tests (200 M eps of the norm): an orthogonal similarity moves no eigenvalue, and 2 M / b block
updates of relative error eps each stay below it."""
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


def dev(x):
    import torch
    return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")


def _reduced_spectrum(gep, oracle_lib, C, b):
    d, e, _, q2, _ = gep.tridiag_2stage(dev(C), b=b)
    return np.sort(oracle_lib.bisect(d.cpu().numpy(), e.cpu().numpy()))


@pytest.mark.parametrize("b", [32, 64])
@pytest.mark.parametrize("M", [2, 3, 31, 33, 34, 63, 64, 65, 66, 67, 95, 97, 128, 129, 130, 161, 193, 320])
def test_block_edges(gep, oracle_lib, M, b):
    rng = np.random.default_rng(M + b)
    C = rng.standard_normal((M, M))
    C = C + C.T
    w = np.linalg.eigvalsh(C)
    wT = _reduced_spectrum(gep, oracle_lib, C, b)
    assert np.max(np.abs(wT - w)) <= 200 * M * EPS * np.max(np.abs(w))


@pytest.mark.parametrize("b", [32, 64])
@pytest.mark.parametrize("name", ["tiny", "huge", "zero", "diagonal", "ones", "one_large", "graded", "banded"])
def test_scales_and_structure(gep, oracle_lib, name, b):
    M = 200
    rng = np.random.default_rng(b)
    S = rng.standard_normal((M, M))
    S = S + S.T
    i = np.arange(M)
    C = {"tiny": S * 1e-150, "huge": S * 1e150, "zero": np.zeros((M, M)), "diagonal": np.diag(i - 7.0),
         "ones": np.ones((M, M)), "one_large": S + 1e9 * np.outer(i == 3, i == 3),
         "graded": S * np.outer(10.0 ** (-i / 20), 10.0 ** (-i / 20)),
         "banded": np.where(np.abs(i[:, None] - i[None, :]) <= b, S, 0.0)}[name]
    w = np.linalg.eigvalsh(C)
    wT = _reduced_spectrum(gep, oracle_lib, C, b)
    assert np.max(np.abs(wT - w)) <= 200 * M * EPS * np.max(np.abs(w)) + 1e-300


@pytest.mark.parametrize("b,drop", [(32, 0), (32, 5), (64, 3)])
def test_wait_that_runs_out_is_reported(gep, oracle_lib, b, drop):
    """A sweep that publishes no progress: the waits behind it give up, the status says so, and the
    same handle then reduces the matrix."""
    M = 300
    rng = np.random.default_rng(3)
    C = rng.standard_normal((M, M))
    C = C + C.T
    h = gep.Handle()
    try:
        h.set_wait_fault(drop_sweep=drop, wait_limit_s=0.2)
        gep.tridiag_2stage(dev(C), b=b, handle=h)
        assert h.info() == gep.ERR_TIMEOUT
        h.set_wait_fault(drop_sweep=-1, wait_limit_s=4.0)
        h.reset_info()
        d, e, _, _, _ = gep.tridiag_2stage(dev(C), b=b, handle=h)
        assert h.info() == 0
        w = np.linalg.eigvalsh(C)
        wT = np.sort(oracle_lib.bisect(d.cpu().numpy(), e.cpu().numpy()))
        assert np.max(np.abs(wT - w)) <= 200 * M * EPS * np.max(np.abs(w))
    finally:
        h.close()


@pytest.mark.parametrize("b", [32, 64])
def test_reflectors_give_an_orthogonal_basis(gep, b):
    """Z = Q1 Q2 I from the stored reflectors: orthogonal, and T = Z^T C Z."""
    M = 333
    rng = np.random.default_rng(b + 1)
    C = rng.standard_normal((M, M))
    C = C + C.T
    d, e, tau1, q2, Cr = gep.tridiag_2stage(dev(C), b=b)
    Z = gep.sep_backtransform_2stage(Cr, tau1, q2, b, dev(np.eye(M))).cpu().numpy()
    d, e = d.cpu().numpy(), e.cpu().numpy()
    T = np.diag(d) + np.diag(e, 1) + np.diag(e, -1)
    n = np.max(np.abs(np.linalg.eigvalsh(C)))
    assert np.max(np.abs(Z.T @ Z - np.eye(M))) <= 200 * M * EPS
    assert np.max(np.abs(Z.T @ C @ Z - T)) <= 200 * M * EPS * n


@pytest.mark.parametrize("b", [32, 64])
def test_no_drift_of_the_spectrum(gep, b):
    """A reflector that is longer or shorter than it should be by the same sign every time scales the
    whole spectrum, a little more with every sweep.  Random rounding leaves 2 to 3 eps of the norm
    per eigenvalue at this order; 6 eps (root mean square) would be a drift of 2^-60 a sweep."""
    import torch
    M = 2000
    g = torch.Generator(device="cuda").manual_seed(b)
    Q, _ = torch.linalg.qr(torch.randn(M, M, generator=g, dtype=torch.float64, device="cuda"))
    lam = torch.linspace(-20.0, 20.0, M, dtype=torch.float64, device="cuda")
    C = (Q * lam) @ Q.t()
    C = 0.5 * (C + C.t())
    w, _, info = gep.solve(C, torch.eye(M, dtype=torch.float64, device="cuda"), sep="2stage", bandwidth=b,
                           precision="fp64_emulated", want_vectors=False)
    assert info == 0
    ref = torch.linalg.eigvalsh(C)
    assert float((w - ref).norm() / ref.norm()) <= 6 * EPS


@pytest.mark.parametrize("b", [32, 64])
@pytest.mark.parametrize("M", [200, 400])
@pytest.mark.parametrize("decay", [20.0, 60.0])
def test_graded_reflectors_stay_orthogonal(gep, M, b, decay):
    """Columns far below the norm bound: the reflectors are formed from a few units of the fixed point, and
    those at the end of the matrix must not see rows beyond it."""
    import torch
    rng = np.random.default_rng(b)
    S = rng.standard_normal((M, M))
    s = np.exp(-np.linspace(0, decay, M))
    C = dev((S + S.T) * np.outer(s, s))
    d, e, tau1, q2, Cr = gep.tridiag_2stage(C, b=b)
    eye = torch.eye(M, dtype=torch.float64, device="cuda")
    Q = gep.sep_backtransform_2stage(Cr, tau1, q2, b, eye)
    T = torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1)
    assert float((Q.t() @ Q - eye).abs().max()) <= 200 * M * EPS
    assert float((Q.t() @ C @ Q - T).abs().max()) <= 200 * M * EPS * float(torch.linalg.matrix_norm(C, 2))


@pytest.mark.parametrize("b", [32, 64])
@pytest.mark.parametrize("eps", [1e-6, 1e-9, 1e-12])
def test_nearly_tridiagonal(gep, b, eps):
    """Entries far below alpha are annihilated, not dropped."""
    M = 200
    rng = np.random.default_rng(b)
    S = rng.standard_normal((M, M))
    S = S + S.T
    i = np.arange(M)
    C = np.where(np.abs(i[:, None] - i[None, :]) <= 1, S, S * eps)
    w = np.linalg.eigvalsh(C)
    d, e, _, _, _ = gep.tridiag_2stage(dev(C), b=b)
    T = np.diag(d.cpu().numpy()) + np.diag(e.cpu().numpy(), 1) + np.diag(e.cpu().numpy(), -1)
    assert np.max(np.abs(np.linalg.eigvalsh(T) - w)) <= 200 * M * EPS * np.max(np.abs(w))


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("route", ["1stage", "1stage_large", "b32", "b64"])
def test_nonfinite_shows_in_the_result(gep, route, bad):
    """The stage entry points take any matrix: a NaN or an infinity comes out as NaN, not as numbers."""
    M = 700 if route == "1stage_large" else 150
    rng = np.random.default_rng(1)
    C = rng.standard_normal((M, M))
    C = C + C.T
    C[M - 20, M - 30] = C[M - 30, M - 20] = bad
    if route.startswith("1stage"):
        d, e = gep.tridiag_1stage(dev(C))[:2]
    else:
        d, e = gep.tridiag_2stage(dev(C), b=int(route[1:]))[:2]
    assert np.isnan(d.cpu().numpy()).any()
