"""Deep products on the tensor cores through residues modulo 16 coprime numbers.

The integer product of the scaled operands is reconstructed exactly, so operands whose products and
sums are exact in FP64 must give the FP64 result bit for bit, whatever the order of summation.
"""
from fractions import Fraction

import numpy as np
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


def dev(x):
    import torch
    return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")


# tile edges (256), K remainders (64, 1024, panels of 4096), column blocks (2048), the lower triangle
@pytest.mark.parametrize("m,n,k,ta,tb,uplo,alpha,beta", [
    (256, 256, 4096, "N", "N", "F", 1.0, 0.0),
    (257, 255, 4095, "N", "T", "F", -1.0, 1.0),
    (129, 511, 3073, "T", "N", "F", 2.0, -0.5),
    (300, 200, 9000, "T", "T", "F", -1.0, 1.0),
    (1000, 2300, 2111, "N", "N", "F", 1.0, 1.0),
    (1031, 1031, 4161, "N", "T", "L", -1.0, 1.0),
    (2500, 2500, 1025, "T", "N", "L", 1.0, 0.0),
    (17, 2049, 8192, "N", "N", "F", 1.0, 0.0),
])
def test_exact_products(gep, m, n, k, ta, tb, uplo, alpha, beta):
    rng = np.random.default_rng(m + n + k)
    # |sum| < 2^13.2 2^38 = 2^51.2; row and column scales over 2^+-60 are powers of two, so still exact
    A = rng.integers(-2 ** 19, 2 ** 19 + 1, size=(m, k)).astype(np.float64)
    B = rng.integers(-2 ** 19, 2 ** 19 + 1, size=(k, n)).astype(np.float64)
    A[m // 2, :] = 0.0
    B[:, n // 3] = 0.0
    A[m // 3, k // 2:] = 0.0
    sr = 2.0 ** rng.integers(-60, 61, size=(m, 1))
    sc = 2.0 ** rng.integers(-60, 61, size=(1, n))
    C = rng.integers(-2 ** 20, 2 ** 20 + 1, size=(m, n)) * sr * sc
    ref = alpha * ((A @ B) * sr * sc) + beta * C
    As, Bs = A * sr, B * sc
    out = gep.dgemm(dev(As.T if ta == "T" else As), dev(Bs.T if tb == "T" else Bs), ta, tb, alpha=alpha, beta=beta,
                    C=dev(C), uplo=uplo, engine="fp64_emulated").cpu().numpy()
    if uplo == "L":
        ref = np.where(np.tril(np.ones((m, n), bool)), ref, C)
    assert np.array_equal(out, ref)


@pytest.mark.parametrize("k", [1024, 4096])
@pytest.mark.parametrize("x,y", [(2.0 - 2.0 ** -52, 2.0 - 2.0 ** -52), (-2.0 + 2.0 ** -52, 1.0), (1.0 / 3.0, -5.0 / 7.0)])
def test_largest_sums(gep, k, x, y):
    """All entries equal: the sums of the residue products and the integer product are as large as they get."""
    import torch
    A = torch.full((256, k), x, dtype=torch.float64, device="cuda")
    B = torch.full((k, 256), y, dtype=torch.float64, device="cuda")
    out = gep.dgemm(A, B, engine="fp64_emulated").cpu().numpy()
    exact = k * Fraction(x) * Fraction(y)
    assert np.all(out == out[0, 0])
    assert abs(Fraction(float(out[0, 0])) - exact) <= abs(exact) * Fraction(1, 2 ** 53) * Fraction(1025, 1024)


def test_tiny_results(gep):
    """Products far below the scale of their row and column, down to single units of the integer product."""
    rng = np.random.default_rng(5)
    m, n, k = 256, 256, 2048
    A = np.zeros((m, k))
    B = np.zeros((k, n))
    A[:, 0] = 1.0
    B[1, :] = 1.0
    ea, eb = rng.integers(1, 55, size=(m, 1)), rng.integers(1, 55, size=(1, n))
    A[:, 2:3] = 2.0 ** -ea  # the only column that meets a nonzero row of B below
    B[2:3, :] = 2.0 ** -eb
    out = gep.dgemm(dev(A), dev(B), engine="fp64_emulated").cpu().numpy()
    assert np.array_equal(out, 2.0 ** -(ea + eb).astype(np.float64))
