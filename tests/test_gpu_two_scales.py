"""Reductions of matrices whose blocks lie on very different scales, and that are decoupled or coupled only through the
first column: every block keeps the accuracy that it has alone (a backward error of 200 M eps of its own norm, the
tolerance of the other stage tests), whatever arithmetic the reduction takes."""
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


def _blocks(M, m1, s, seed):
    import torch
    C = torch.zeros(M, M, dtype=torch.float64, device="cuda")
    C[:m1, :m1] = _symmetric(m1, seed)
    C[m1:, m1:] = s * _symmetric(M - m1, seed + 1)
    return C


def _backward(Q, C, T, rows):
    """Largest entry of Q^T C Q - T on a block that Q maps into itself, over the block's norm."""
    import torch
    q, c, t = Q[rows, rows], C[rows, rows], T[rows, rows]
    return float((q.t() @ c @ q - t).abs().max() / torch.linalg.matrix_norm(c, 2))


@pytest.mark.parametrize("M,m1", [(12, 5), (40, 17), (100, 99), (128, 1), (300, 100), (500, 250), (512, 480), (700, 600)])
@pytest.mark.parametrize("s", [0.25, 0.03, 1e-4, 1e-10, 1e-19, 1e-60, 1e8])
def test_tridiagonal_blocks(gep, M, m1, s):
    import torch
    C = _blocks(M, m1, s, M)
    d, e, tau, Cr = gep.tridiag_1stage(C)
    Q = gep.sep_backtransform(Cr, tau, torch.eye(M, dtype=torch.float64, device="cuda"))
    T = torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1)
    assert float(e[m1 - 1]) == 0.0
    assert not bool(Q[:m1, m1:].any()) and not bool(Q[m1:, :m1].any())
    for rows in (slice(0, m1), slice(m1, M)):
        assert _backward(Q, C, T, rows) <= 200 * M * EPS


@pytest.mark.parametrize("M", [2, 40, 300])
@pytest.mark.parametrize("s", [1e-3, 1e-30, 1e-200])
def test_decoupled_first_row(gep, M, s):
    C = _blocks(M, 1, 1.0, M)
    C[0, 0] = s
    d, e, _, _ = gep.tridiag_1stage(C)
    assert float(d[0]) == s and float(e[0]) == 0.0


@pytest.mark.parametrize("M", [33, 200, 512])
@pytest.mark.parametrize("s", [1e-3, 1e-12, 1e-25])
def test_tridiagonal_large_first_column(gep, M, s):
    """Only the first reflector sees the first column; what it leaves is on the scale of the rest."""
    import torch
    C = s * _symmetric(M, M)
    C[0, 1:] = C[1:, 0] = torch.linspace(1, 2, M - 1, dtype=torch.float64, device="cuda")
    d, e, tau, Cr = gep.tridiag_1stage(C)
    Q = gep.sep_backtransform(Cr, tau, torch.eye(M, dtype=torch.float64, device="cuda"))
    T = torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1)
    assert _backward(Q, C, T, slice(1, M)) <= 200 * M * EPS


def _block_eigenvalues(C, d, e, rows):
    """Largest error of the eigenvalues of T on a decoupled block, over the block's norm."""
    import torch
    t = (torch.diag(d) + torch.diag(e, 1) + torch.diag(e, -1))[rows, rows].cpu()
    ref = torch.linalg.eigvalsh(C[rows, rows].cpu())
    return float((torch.linalg.eigvalsh(t) - ref).abs().max() / ref.abs().max())


@pytest.mark.parametrize("M,m1", [(90, 40), (300, 96), (700, 500)])
@pytest.mark.parametrize("b", [20, 32, 64])
@pytest.mark.parametrize("s", [0.25, 1e-4, 1e-10, 1e-19, 1e8])
def test_two_stage_blocks(gep, M, m1, b, s):
    C = _blocks(M, m1, s, M)
    d, e, *_ = gep.tridiag_2stage(C, b)
    assert float(e[m1 - 1]) == 0.0
    for rows in (slice(0, m1), slice(m1, M)):
        assert _block_eigenvalues(C, d, e, rows) <= 200 * M * EPS


@pytest.mark.parametrize("b", [20, 32, 64])
@pytest.mark.parametrize("s", [1e-3, 1e-12, 1e-25])
def test_band_large_first_column(gep, b, s):
    """A band matrix whose first column alone is large: T beyond its first row stays on the scale of the rest."""
    import torch
    M = 150
    i = torch.arange(M, device="cuda")
    C = torch.where((i[:, None] - i[None, :]).abs() <= b, s * _symmetric(M, 4), torch.zeros_like(_symmetric(M, 4)))
    C[0, 1:b + 1] = C[1:b + 1, 0] = torch.linspace(1, 2, b, dtype=torch.float64, device="cuda")
    d, e, *_ = gep.tridiag_2stage(C, b)
    # the first sweep's reflector acts on rows 1.. only, so T(1:, 1:) is a similarity of C(1:, 1:)
    assert _block_eigenvalues(C, d, e, slice(1, M)) <= 200 * M * EPS


@pytest.mark.parametrize("b", [8, 32])
@pytest.mark.parametrize("M,m1", [(70, 40), (200, 100), (900, 500), (2080, 1500)])
@pytest.mark.parametrize("s", [0.2, 1e-6, 1e-12, 1e-25])
def test_panel_rows_of_two_scales(gep, M, m1, b, s):
    """Rows far below the others keep their accuracy in the reflectors of a panel: LAPACK's, row by row."""
    import torch
    D = torch.ones(M, dtype=torch.float64, device="cuda")
    D[m1:] = s
    C = D[:, None] * _symmetric(M, M) * D[None, :]
    Cr = gep.tridiag_2stage(C, b)[4]
    V = Cr[b:, :b].cpu().tril(-1)
    ref = torch.geqrf(C[b:, :b].cpu())[0].tril(-1)
    scale = ref.abs().amax(1, keepdim=True)
    assert bool(((V - ref).abs() <= 200 * M * EPS * scale).all())


@pytest.mark.parametrize("M", [300, 1000])
def test_a_slowly_falling_band_keeps_the_fast_route(gep, M):
    """A tight-binding matrix (neighbouring rows alike, the smallest of a band far below the largest): its bulge chasing is
    not the FP64 one, which takes several times as long.  Two blocks 1e-4 apart take the FP64 one."""
    import torch
    import gep_inputs as gi
    p = gi.tight_binding(M, 0)
    A, B = (torch.as_tensor(p[x], device="cuda") for x in "AB")
    h = gep.Handle()

    def chase_ms(a, b):
        t = []
        for _ in range(4):
            assert gep.solve(a, b, sep="2stage", precision="fp64_emulated", timers=True, handle=h)[2] == 0
            t.append(h.band_times()[1])
        return min(t[1:])
    eye = torch.eye(M, dtype=torch.float64, device="cuda")
    assert 1.5 * chase_ms(A, B) < chase_ms(_blocks(M, M // 2, 1e-4, 1), eye)
    h.close()
