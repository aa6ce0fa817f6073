"""Divide and conquer of small and large numbers: eigenvalues and eigenvectors of a tridiagonal matrix do not depend on the
power of two it is multiplied with, as a whole or in a decoupled block.  Tolerances as for the stage's other tests
(200 M eps of the block's norm; orthogonality 200 M eps)."""
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


def _tridiagonal(M, seed):
    import torch
    g = torch.Generator().manual_seed(seed)
    return torch.randn(M, generator=g, dtype=torch.float64), torch.randn(M - 1, generator=g, dtype=torch.float64)


def _dense(d, e):
    import torch
    return torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1)


@pytest.mark.parametrize("M", [9, 16, 20, 31, 33, 100, 300, 1000])
@pytest.mark.parametrize("p", [-900, -300, -40, -8, 0, 30, 400, 900])
def test_scaled(gep, M, p):
    import torch
    d, e = _tridiagonal(M, M)
    w, Z, info = gep.tridiag_eig((d * 2.0 ** p).cuda(), (e * 2.0 ** p).cuda())
    assert info == 0
    T = _dense(d, e)
    ref = torch.linalg.eigvalsh(T)
    n = float(ref.abs().max())
    w, Z = w.cpu() * 2.0 ** -p, Z.cpu()
    assert float((w - ref).abs().max()) <= 200 * M * EPS * n
    assert float((Z.t() @ Z - torch.eye(M, dtype=torch.float64)).abs().max()) <= 200 * M * EPS
    assert float((T @ Z - Z * w).abs().max()) <= 200 * M * EPS * n


@pytest.mark.parametrize("m1,m2", [(20, 25), (64, 30), (100, 200)])
@pytest.mark.parametrize("p", [-10, -60, -400, 200])
def test_blocks(gep, m1, m2, p):
    import torch
    (d1, e1), (d2, e2) = _tridiagonal(m1, 1), _tridiagonal(m2, 2)
    s = 2.0 ** p
    zero = torch.zeros(1, dtype=torch.float64)
    w, Z, info = gep.tridiag_eig(torch.cat([d1, d2 * s]).cuda(), torch.cat([e1, zero, e2 * s]).cuda())
    assert info == 0
    w, Z = w.cpu(), Z.cpu()
    M = m1 + m2
    assert float((Z.t() @ Z - torch.eye(M, dtype=torch.float64)).abs().max()) <= 200 * M * EPS
    for rows, other, (d, e), q in ((slice(0, m1), slice(m1, M), (d1, e1), 1.0), (slice(m1, M), slice(0, m1), (d2, e2), s)):
        mine = Z[rows].abs().amax(0) > 0.5 / M  # the block's eigenvectors vanish on the other block
        T = _dense(d, e)
        ref = torch.linalg.eigvalsh(T)
        assert int(mine.sum()) == len(d) and not bool(Z[other][:, mine].any())
        assert float((w[mine] / q - ref).abs().max()) <= 200 * M * EPS * float(ref.abs().max())


def test_coupling_near_overflow(gep):
    """A coupling whose double overflows, at a tear: +-e and the rest, far below."""
    import torch
    M, big = 40, 1.2e308
    d = torch.zeros(M, dtype=torch.float64)
    e = torch.full((M - 1,), 1e290, dtype=torch.float64)
    e[7] = big
    w, Z, info = gep.tridiag_eig(d.cuda(), e.cuda())
    assert info == 0
    w, Z = w.cpu(), Z.cpu()
    assert abs(float(w[0]) + big) <= 200 * M * EPS * big and abs(float(w[-1]) - big) <= 200 * M * EPS * big
    assert float(w[1:-1].abs().max()) <= 200 * M * EPS * big
    assert float((Z.t() @ Z - torch.eye(M, dtype=torch.float64)).abs().max()) <= 200 * M * EPS


@pytest.mark.parametrize("M", [20, 40, 300])
@pytest.mark.parametrize("where", ["d", "e"])
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_not_a_number_is_a_failure(gep, M, where, bad):
    import torch
    d, e = _tridiagonal(M, M)
    for i in (0, 7, 8, M // 2):
        x, y = d.clone(), e.clone()
        (x if where == "d" else y)[i] = bad
        h = gep.Handle()
        assert gep.tridiag_eig(x.cuda(), y.cuda(), handle=h)[2] > M
        h.close()


@pytest.mark.parametrize("M", [9, 40, 300])
@pytest.mark.parametrize("ordinary", [False, True])
def test_subnormal_numbers(gep, M, ordinary):
    """A matrix (or a decoupled block) of subnormal numbers, whose reciprocals overflow."""
    import torch
    g = torch.Generator().manual_seed(M)
    d = torch.randint(-40, 41, (M,), generator=g).double()
    e = torch.randint(1, 30, (M - 1,), generator=g).double()
    ds, es = d * 2.0 ** -1000 * 2.0 ** -74, e * 2.0 ** -1000 * 2.0 ** -74
    if ordinary:
        d1, e1 = _tridiagonal(30, 1)
        ds, es = torch.cat([d1, ds]), torch.cat([e1, torch.zeros(1, dtype=torch.float64), es])
    w, Z, info = gep.tridiag_eig(ds.cuda(), es.cuda())
    assert info == 0
    w, Z = w.cpu(), Z.cpu()
    N = len(ds)
    assert float((Z.t() @ Z - torch.eye(N, dtype=torch.float64)).abs().max()) <= 200 * N * EPS
    if ordinary:  # (couplings below 2^-900 of their leaf's largest entry count as zero)
        ref = torch.sort(torch.cat([torch.linalg.eigvalsh(_dense(d1, e1)), torch.zeros(M, dtype=torch.float64)]))[0]
        assert float((w - ref).abs().max()) <= 200 * N * EPS * float(ref.abs().max())
        return
    ref = torch.linalg.eigvalsh(_dense(d, e))
    got = w * 2.0 ** 1000 * 2.0 ** 74  # every level rounds to whole units
    assert float((got - ref).abs().max()) <= 8.0
