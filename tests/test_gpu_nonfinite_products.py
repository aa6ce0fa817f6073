"""NaN and infinity in the operands of every form of the products: no output that they reach is a number (NaN on the
tensor cores; on the FP64 units, where the cheapest shapes stay, an infinity may stay one), the others are what they are
without them (rows and columns are scaled by themselves, so bit for bit)."""
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


# thin digits (fused and slab splits), square digits, two K panels, residues in one and two K panels, lower triangle
@pytest.mark.parametrize("engine,m,n,k,ta,tb,uplo,beta", [
    ("fp64_emulated", 33, 1100, 1050, "N", "N", "F", 0.0),
    ("fp64_emulated", 1100, 40, 300, "T", "T", "F", 1.0),
    ("mixed_refined", 64, 900, 700, "N", "T", "F", 0.0),
    ("fp64_emulated", 300, 300, 200, "T", "N", "F", -0.5),
    ("mixed_refined", 200, 300, 5000, "N", "N", "F", 1.0),
    ("fp64_emulated", 600, 520, 4096, "N", "T", "F", 1.0),
    ("fp64_emulated", 600, 520, 5000, "T", "N", "F", 0.0),
    ("fp64_emulated", 700, 700, 2100, "N", "N", "L", 1.0),
])
@pytest.mark.parametrize("bad", [float("nan"), float("inf"), float("-inf")])
def test_nonfinite_operands(gep, engine, m, n, k, ta, tb, uplo, beta, bad):
    import torch
    g = torch.Generator(device="cuda").manual_seed(m + n + k)
    rnd = lambda r, c: torch.randn(r, c, generator=g, dtype=torch.float64, device="cuda")
    A, B, C = rnd(m, k), rnd(k, n), rnd(m, n)
    rows, cols = [0, m // 2, m - 1], [n // 3, n - 1]
    A0, B0 = A.clone(), B.clone()
    A0[rows] = 0.0
    B0[:, cols] = 0.0
    for i, kk in zip(rows, (0, k - 1, k // 2)):
        A[i, kk] = bad
    for j, kk in zip(cols, (k - 1, 1)):
        B[kk, j] = bad
    tr = lambda X, t: X.t().contiguous() if t == "T" else X
    mul = lambda X, Y: gep.dgemm(tr(X, ta), tr(Y, tb), ta, tb, beta=beta, C=C, uplo=uplo, engine=engine)
    out, ref = mul(A, B), mul(A0, B0)
    hit = torch.zeros(m, n, dtype=torch.bool, device="cuda")
    hit[rows] = True
    hit[:, cols] = True
    if uplo == "L":
        hit = hit.tril()
    assert not bool(torch.isfinite(out[hit]).any())
    if bad != bad:
        assert bool(torch.isnan(out[hit]).all())
    assert torch.equal(out[~hit], ref[~hit])
    assert bool(torch.isfinite(ref).all())


@pytest.mark.parametrize("m,n", [(300, 200), (2000, 64)])
def test_nonfinite_symmetric_operand(gep, m, n):
    import torch
    g = torch.Generator(device="cuda").manual_seed(m)
    A = torch.randn(m, m, generator=g, dtype=torch.float64, device="cuda")
    B = torch.randn(m, n, generator=g, dtype=torch.float64, device="cuda")
    A[200, 7] = float("nan")  # lower triangle: row 200 and, mirrored, row 7
    out = gep.dgemm(A, B, "S", "N", engine="fp64_emulated")
    assert bool(torch.isnan(out[[7, 200]]).all())
    keep = torch.ones(m, dtype=torch.bool)
    keep[[7, 200]] = False
    assert bool(torch.isfinite(out[keep]).all())
