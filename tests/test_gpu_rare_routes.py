"""Routes that the defaults rarely take: the one-launch panels of the tridiagonalisation at orders that a cluster takes
by default (ragged and last panels, degenerate columns), the panel QR without a cluster, and the one-CTA solver at its
larger orders with its failure status.  Tolerances as for the routes' other tests."""
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


@pytest.fixture()
def no_clusters(gep):
    h = gep.Handle()
    h.set_routes(clusters=False)
    yield h
    h.close()


def _symmetric(M, seed):
    import torch
    g = torch.Generator(device="cuda").manual_seed(seed)
    G = torch.randn(M, M, generator=g, dtype=torch.float64, device="cuda")
    return G + G.t()


def _tridiagonal_form(gep, h, C, norm):
    import torch
    M = C.shape[0]
    d, e, tau, Cr = gep.tridiag_1stage(C, handle=h)
    eye = torch.eye(M, dtype=torch.float64, device="cuda")
    Q = gep.sep_backtransform(Cr, tau, eye, handle=h)
    T = torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1)
    assert bool(torch.isfinite(T).all())
    assert float((Q.t() @ Q - eye).abs().max()) <= 200 * M * EPS
    assert float((Q.t() @ C @ Q - T).abs().max()) <= 200 * M * EPS * norm + 1e-300


@pytest.mark.parametrize("M", [1, 2, 3, 31, 32, 33, 63, 64, 65, 66, 95, 97, 129, 193, 500])
def test_panels_of_small_orders(gep, no_clusters, M):
    import torch
    C = _symmetric(M, M)
    _tridiagonal_form(gep, no_clusters, C, float(torch.linalg.matrix_norm(C, 2)))


@pytest.mark.parametrize("kind", ["zero", "diagonal", "banded", "tiny", "huge"])
def test_panels_with_degenerate_columns(gep, no_clusters, kind):
    import torch
    M = 150
    S = _symmetric(M, 9)
    i = torch.arange(M, device="cuda")
    C = {"zero": torch.zeros_like(S), "diagonal": torch.diag(i.double()), "tiny": S * 1e-140, "huge": S * 1e140,
         "banded": torch.where((i[:, None] - i[None, :]).abs() <= 2, S, torch.zeros_like(S))}[kind]
    _tridiagonal_form(gep, no_clusters, C, float(C.abs().max()) * M)


def test_the_hook_changes_the_route(gep, no_clusters):
    """One cluster launch for an order of 200, several panels without it."""
    C = _symmetric(200, 1)
    n = []
    for clusters in (True, False):
        no_clusters.set_routes(clusters=clusters)
        no_clusters.launches(reset=True)
        gep.tridiag_1stage(C, handle=no_clusters)
        n.append(no_clusters.launches(reset=True))
    assert n[0] == 1 and n[1] >= 4


@pytest.mark.parametrize("M,b", [(34, 32), (65, 32), (96, 31), (130, 7), (289, 32), (545, 32), (1057, 32)])
def test_panel_qr_without_a_cluster(gep, no_clusters, M, b):
    import torch
    C = _symmetric(M, M)
    eye = torch.eye(M, dtype=torch.float64, device="cuda")
    w, Y, info = gep.solve(C, eye, precision="fp64_emulated", sep="2stage", bandwidth=b, handle=no_clusters)
    assert info == 0
    n = float(torch.linalg.matrix_norm(C, 2))
    assert float((w - torch.linalg.eigvalsh(C.cpu()).cuda()).abs().max()) <= 200 * M * EPS * n
    assert float((Y.t() @ Y - eye).abs().max()) <= 200 * M * EPS
    assert float((C @ Y - Y * w).abs().max()) <= 200 * M * EPS * n


def _one_cta(gep, As, Bs):
    import torch
    h = gep.Handle()
    h.set_routes(one_cta=True)
    s = gep.BatchedSolver(As, Bs, nstreams=2, precision="fp64", handle=h)
    h.launches(reset=True)
    s.run()
    torch.cuda.synchronize()
    assert h.launches(reset=True) <= 2
    return s


@pytest.mark.parametrize("orders", [[85], [96, 100], [127, 128], [1, 2, 3, 33, 64, 65]])
def test_one_cta_solver(gep, orders):
    import torch
    As = [_symmetric(M, M) for M in orders]
    H = [_symmetric(M, M + 1) for M in orders]
    Bs = [x @ x.t() / x.shape[0] + torch.eye(x.shape[0], dtype=torch.float64, device="cuda") for x in H]
    s = _one_cta(gep, As, Bs)
    assert s.info() == 0
    for A, B, (w, Y) in zip(As, Bs, s.results()):
        n = float(torch.linalg.matrix_norm(A, 2))
        eye = torch.eye(A.shape[0], dtype=torch.float64, device="cuda")
        assert float((Y.t() @ B @ Y - eye).abs().max()) <= 1e-12
        assert float((A @ Y - B @ Y * w).abs().max()) <= 1e-11 * n
        assert bool((w[1:] >= w[:-1]).all())
    s.h.close()


@pytest.mark.parametrize("M,minor", [(64, 11), (100, 90), (128, 128)])
def test_one_cta_status(gep, M, minor):
    """The first leading minor of B that is not positive, as the staged solve reports it; a NaN in A."""
    import torch
    A, B = _symmetric(M, 1), torch.eye(M, dtype=torch.float64, device="cuda")
    bad = B.clone()
    bad[minor - 1, minor - 1] = -1.0
    s = _one_cta(gep, [A, A], [B, bad])
    assert s.info() == minor
    assert gep.solve(A, bad, handle=s.h)[2] == minor  # (a status stays with its handle)
    s.h.close()
    nan = A.clone()
    nan[5, 3] = nan[3, 5] = float("nan")
    s = _one_cta(gep, [A, nan], [B, B])
    assert s.info() == gep.ERR_NONFINITE
    s.h.close()
