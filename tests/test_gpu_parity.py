"""Parity of the CUDA path with the FP64 CPU oracle, stage by stage and end to end.

Inputs are seeded (gep_inputs); expected values come from the oracle on the same
inputs.  Sizes span several 64/128-wide tiles plus a ragged tail.  Tolerances are
the solver's FP64 accuracy target (|d lambda| <= 1e-11 ||A||_2, residual
||AY - BY Lambda||_F / (||A||_F M) <= 1e-13, ||Y^T B Y - I||_max <= 1e-12) or, for
intermediate quantities, a stated multiple of M * eps relative to the input scale.
"""
import numpy as np
import pytest

import gep_inputs as gi

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52


@pytest.fixture(scope="module")
def gep():
    import torch
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    from paper_1504_06443_gb300 import build
    build.build()
    import paper_1504_06443_gb300 as g
    g.load()
    return g


@pytest.fixture(scope="module")
def torch_mod():
    import torch
    return torch


def dev(x):
    import torch
    return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")


def host(t):
    return t.detach().cpu().numpy()


def two_norm(A):
    return float(np.max(np.abs(np.linalg.eigvalsh(A))))


# ------------------------------------------------------------------ GEMM engine

@pytest.mark.parametrize("ta,tb", [("N", "N"), ("N", "T"), ("T", "N"), ("T", "T")])
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (67, 130, 33), (200, 64, 129)])
def test_dgemm_fp64(gep, ta, tb, m, n, k):
    rng = np.random.default_rng(m * n + k)
    A = rng.standard_normal((k, m) if ta == "T" else (m, k))
    B = rng.standard_normal((n, k) if tb == "T" else (k, n))
    C = rng.standard_normal((m, n))
    ref = 0.7 * (A.T if ta == "T" else A) @ (B.T if tb == "T" else B) - 0.3 * C
    out = gep.dgemm(dev(A), dev(B), ta, tb, alpha=0.7, beta=-0.3, C=dev(C))
    assert np.max(np.abs(host(out) - ref)) <= 4 * k * EPS * np.max(np.abs(A)) * np.max(np.abs(B)) * 2 + 1e-14


def test_dgemm_lower_only(gep):
    rng = np.random.default_rng(0)
    A = rng.standard_normal((150, 40))
    C = rng.standard_normal((150, 150))
    out = host(gep.dgemm(dev(A), dev(A), "N", "T", alpha=-1.0, beta=1.0, C=dev(C), uplo="L"))
    ref = C - A @ A.T
    il = np.tril_indices(150)
    iu = np.triu_indices(150, 1)
    assert np.max(np.abs(out[il] - ref[il])) <= 1e-12
    assert np.array_equal(out[iu], C[iu])


# ------------------------------------------------------------------ reducer

@pytest.mark.parametrize("M", [1, 31, 128, 129, 300, 513])
def test_cholesky_vs_oracle(gep, oracle_lib, M):
    g = gi.known_spectrum(M, seed=M)
    L_ref, info_ref = oracle_lib.cholesky(g["B"])
    L, info = gep.cholesky(dev(g["B"]))
    assert info == 0 and info_ref == 0
    Lh = np.tril(host(L))
    assert np.max(np.abs(Lh - L_ref)) <= 64 * M * EPS * np.max(np.abs(L_ref))


@pytest.mark.parametrize("k", [1, 77, 130, 256])
def test_cholesky_reports_first_bad_minor(gep, oracle_lib, k):
    M = 300
    B = gi.spd_matrix(M, seed=k)
    L0 = np.linalg.cholesky(B)
    D = np.ones(M)
    D[k - 1] = -1.0
    Bk = (L0 * D[None, :]) @ L0.T
    Bk = 0.5 * (Bk + Bk.T)
    _, info_ref = oracle_lib.cholesky(Bk)
    _, info = gep.cholesky(dev(Bk))
    assert info == info_ref == k


@pytest.mark.parametrize("variant", ["twosided", "explicit_inv"])
@pytest.mark.parametrize("M", [64, 257, 400])
def test_reduce_vs_oracle(gep, oracle_lib, variant, M):
    tb = gi.tight_binding(M if M % 4 == 0 else M - M % 4 + 4, seed=3)
    A, B = tb["A"][:M, :M], tb["B"][:M, :M]
    L_ref, _ = oracle_lib.cholesky(B)
    C_ref = oracle_lib.two_sided(A, L_ref)
    L, info = gep.cholesky(dev(B))
    assert info == 0
    C, LR = gep.reduce(dev(A), L, variant)
    Ch = host(C)
    assert np.max(np.abs(Ch - Ch.T)) == 0.0
    assert np.max(np.abs(Ch - C_ref)) <= 1e-12 * max(1.0, np.max(np.abs(C_ref)))
    if variant == "explicit_inv":
        R = np.tril(host(LR))
        assert np.max(np.abs(R @ L_ref - np.eye(M))) <= 1e-12 * M


# ---------------------------------------------------------- SEP solver stages

@pytest.mark.parametrize("M", [1, 2, 3, 64, 65, 200, 333])
def test_tridiag_vs_oracle(gep, oracle_lib, M):
    rng = np.random.default_rng(M)
    G = rng.standard_normal((M, M))
    C = 0.5 * (G + G.T)
    d_ref, e_ref, Q_ref = oracle_lib.tridiag(C)
    d, e, tau, Cr = gep.tridiag_1stage(dev(C))
    scale = max(1.0, np.max(np.abs(C)))
    assert np.max(np.abs(host(d) - d_ref)) <= 200 * M * EPS * scale
    assert np.max(np.abs(host(e) - e_ref), initial=0.0) <= 200 * M * EPS * scale
    # Q from the reflectors: back-transform the identity and compare with the oracle's Q
    Q = host(gep.sep_backtransform(Cr, tau, dev(np.eye(M))))
    assert np.max(np.abs(Q - Q_ref)) <= 200 * M * EPS


def _tridiag_cases():
    rng = np.random.default_rng(7)
    cases = []
    for M in (1, 2, 31, 32, 33, 64, 100, 257, 700):
        cases.append((f"random{M}", rng.standard_normal(M), rng.standard_normal(max(M - 1, 0))))
    n = 300
    cases.append(("diagonal", rng.standard_normal(n), np.zeros(n - 1)))
    cases.append(("constant", np.full(n, 2.0), np.full(n - 1, 1e-9)))                 # heavy deflation
    k = np.arange(n)
    cases.append(("wilkinson", np.abs(k - n // 2).astype(float), np.ones(n - 1)))      # close pairs
    cases.append(("toeplitz", np.full(n, 0.5), np.full(n - 1, -1.0)))
    d = rng.standard_normal(n)
    e = rng.standard_normal(n - 1)
    e[::37] = 0.0                                                                      # split blocks
    cases.append(("split", d, e))
    cases.append(("graded", np.logspace(-8, 2, n), np.sqrt(np.logspace(-8, 2, n - 1)) * 1e-3))
    return cases


@pytest.mark.parametrize("name,d,e", _tridiag_cases(), ids=lambda x: x if isinstance(x, str) else "")
def test_dc_vs_oracle(gep, oracle_lib, name, d, e):
    M = d.shape[0]
    w_ql, _, st = oracle_lib.tql(d, e)
    w_ref = np.sort(w_ql)
    w_bi = oracle_lib.bisect(d, e)
    T = np.diag(d) + np.diag(e, 1) + np.diag(e, -1)
    nT = max(1e-300, np.max(np.abs(w_ref)))
    w, Z, info = gep.tridiag_eig(dev(d), dev(e), want_vectors=True)
    assert info == 0
    wh, Zh = host(w), host(Z)
    assert np.all(np.diff(wh) >= 0)
    assert np.max(np.abs(wh - w_ref)) <= 64 * M * EPS * nT + 1e-300
    assert np.max(np.abs(wh - w_bi)) <= 64 * M * EPS * nT + 1e-300
    assert np.max(np.abs(Zh.T @ Zh - np.eye(M))) <= 64 * M * EPS
    assert np.max(np.abs(T @ Zh - Zh * wh[None, :])) <= 64 * M * EPS * nT
    w0, Z0, info0 = gep.tridiag_eig(dev(d), dev(e), want_vectors=False)
    assert Z0 is None and info0 == 0
    assert np.max(np.abs(host(w0) - w_bi)) <= 16 * EPS * nT * 4 + 1e-300


@pytest.mark.parametrize("variant", ["twosided", "explicit_inv"])
def test_backsub_vs_oracle(gep, oracle_lib, variant):
    M = 300
    g = gi.known_spectrum(M, seed=1)
    L_ref, _ = oracle_lib.cholesky(g["B"])
    Z = np.random.default_rng(2).standard_normal((M, 70))
    Y_ref = oracle_lib.backsub(L_ref, Z)
    L, _ = gep.cholesky(dev(g["B"]))
    if variant == "explicit_inv":
        _, LR = gep.reduce(dev(g["A"]), L, "explicit_inv")
    else:
        LR = L
    Y = host(gep.gep_backtransform(LR, dev(Z), variant))
    assert np.max(np.abs(Y - Y_ref)) <= 1e-12 * np.max(np.abs(Y_ref))


# -------------------------------------------------------------- whole workflow

def _check_solution(A, B, w, Y, w_ref):
    M = A.shape[0]
    nA = two_norm(A)
    assert np.max(np.abs(w - w_ref)) <= 1e-11 * nA
    res = np.linalg.norm(A @ Y - (B @ Y) * w[None, :]) / (np.linalg.norm(A) * M)
    orth = np.max(np.abs(Y.T @ B @ Y - np.eye(M)))
    assert res <= 1e-13, res
    assert orth <= 1e-12, orth


@pytest.mark.parametrize("precision", ["fp64", "fp64_emulated"])
@pytest.mark.parametrize("reducer", ["twosided", "explicit_inv"])
@pytest.mark.parametrize("seed", [0, 1])
def test_solve_known_spectrum_M512(gep, oracle_lib, reducer, seed, precision):
    """Workload of the M=512 known-spectrum configuration: exact lambda and the oracle."""
    g = gi.known_spectrum(512, seed)
    A, B = g["A"], g["B"]
    w_ref, Y_ref, info = oracle_lib.gep_solve(A, B)
    assert info == 0
    w, Y, info = gep.solve(dev(A), dev(B), reducer=reducer, precision=precision)
    assert info == 0
    wh, Yh = host(w), host(Y)
    _check_solution(A, B, wh, Yh, w_ref)
    assert np.max(np.abs(wh - np.sort(g["lam"]))) <= 1e-11 * two_norm(A)
    # isolated eigenpairs compare elementwise (sign convention applied by both sides)
    gaps = np.minimum(np.diff(w_ref, prepend=-np.inf), np.diff(w_ref, append=np.inf))
    iso = gaps > 1e-6 * two_norm(A)
    assert np.max(np.abs(Yh[:, iso] - Y_ref[:, iso])) <= 1e-8


@pytest.mark.parametrize("precision", ["fp64", "fp64_emulated"])
@pytest.mark.parametrize("M", [4, 36, 260, 516, 1280])
def test_solve_tight_binding_vs_oracle(gep, oracle_lib, M, precision):
    tb = gi.tight_binding(M, seed=M)
    A, B = tb["A"], tb["B"]
    w_ref, Y_ref, info = oracle_lib.gep_solve(A, B)
    assert info == 0
    w, Y, info = gep.solve(dev(A), dev(B), precision=precision)
    assert info == 0
    _check_solution(A, B, host(w), host(Y), w_ref)
    w0, Y0, info0 = gep.solve(dev(A), dev(B), want_vectors=False, precision=precision)
    assert Y0 is None and info0 == 0
    assert np.max(np.abs(host(w0) - w_ref)) <= 1e-11 * two_norm(A)


def test_solve_not_positive_definite(gep):
    M = 200
    B = np.eye(M)
    B[150, 150] = -1.0
    A = gi.random_symmetric(M, 0)
    _, _, info = gep.solve(dev(A), dev(B))
    assert info == 151


def test_solve_nonfinite_input(gep):
    M = 64
    A = gi.random_symmetric(M, 1)
    A[10, 3] = np.nan
    A[3, 10] = np.nan
    _, _, info = gep.solve(dev(A), dev(np.eye(M)))
    assert info == -102


def test_solve_host_buffers_match_device(gep):
    tb = gi.tight_binding(256, seed=9)
    w_d, Y_d, _ = gep.solve(dev(tb["A"]), dev(tb["B"]))
    w_h, Y_h, info = gep.solve_host(tb["A"], tb["B"])
    assert info == 0
    assert np.array_equal(host(w_d), w_h)
    assert np.array_equal(host(Y_d), Y_h)


def test_solve_edge_sizes(gep, oracle_lib):
    for M in (1, 2, 3, 33, 127, 129):
        rng = np.random.default_rng(M)
        A = gi.random_symmetric(M, M)
        B = gi.spd_matrix(M, M, cond=5.0)
        w_ref, _, _ = oracle_lib.gep_solve(A, B)
        w, Y, info = gep.solve(dev(A), dev(B))
        assert info == 0
        _check_solution(A, B, host(w), host(Y), w_ref)


# The FP64 product's tile choice: 16 x 16 tiles with a split depth, 32 x 32 and 64 x 64 tiles, and
# their ragged edges, each operand form; tolerance: k roundings of the largest product, twice over.
@pytest.mark.parametrize("m,n,k", [(16, 16, 4096), (17, 15, 33), (64, 64, 63), (65, 130, 1025), (130, 33, 2049),
                                   (500, 500, 96), (901, 803, 40), (1700, 1601, 20)])
@pytest.mark.parametrize("ta,tb,uplo", [("N", "N", "F"), ("N", "T", "L"), ("T", "N", "F"), ("T", "T", "F")])
def test_dgemm_fp64_tile_choices(gep, ta, tb, uplo, m, n, k):
    rng = np.random.default_rng(m + n + k)
    n = m if uplo == "L" else n
    A = rng.standard_normal((k, m) if ta == "T" else (m, k))
    B = rng.standard_normal((n, k) if tb == "T" else (k, n))
    C = rng.standard_normal((m, n))
    ref = 1.5 * (A.T if ta == "T" else A) @ (B.T if tb == "T" else B) + 0.5 * C
    if uplo == "L":
        ref = np.tril(ref) + np.triu(C, 1)
    out = host(gep.dgemm(dev(A), dev(B), ta, tb, alpha=1.5, beta=0.5, C=dev(C), uplo=uplo))
    tol = 2 * k * EPS * 1.5 * np.max(np.abs(A)) * np.max(np.abs(B)) + 1e-14
    assert np.max(np.abs(out - ref)) <= tol


def test_dgemm_fp64_symmetric_operand_split_depth(gep):
    rng = np.random.default_rng(5)
    A = rng.standard_normal((700, 700))
    S = np.tril(A) + np.tril(A, -1).T
    B = rng.standard_normal((700, 20))
    out = host(gep.dgemm(dev(np.tril(A)), dev(B), "S", "N"))
    assert np.max(np.abs(out - S @ B)) <= 2 * 700 * EPS * np.max(np.abs(A)) * np.max(np.abs(B)) + 1e-14


def _dc_edge_cases():
    """Orders at the edges of the leaves and of the merge levels, with and without a ragged or
    unmerged tail, each with rotations in chains (equal and nearly equal eigenvalues of the halves)
    and with negligible couplings."""
    rng = np.random.default_rng(11)
    cases = []
    for M in (7, 8, 9, 15, 16, 17, 24, 25, 47, 48, 49, 127, 129, 255, 256, 258, 511, 520, 770):
        cases.append((f"random{M}", rng.standard_normal(M), rng.standard_normal(M - 1)))
        cases.append((f"equal{M}", np.full(M, -3.0), np.full(M - 1, 1e-12)))
        d = np.round(rng.standard_normal(M) * 2)
        e = np.where(rng.random(M - 1) < 0.3, 1e-17, 1e-3)
        cases.append((f"chains{M}", d, e))
    return cases


@pytest.mark.parametrize("name,d,e", _dc_edge_cases(), ids=lambda x: x if isinstance(x, str) else "")
def test_dc_leaf_and_level_edges(gep, oracle_lib, name, d, e):
    M = d.shape[0]
    w_ref = oracle_lib.bisect(d, e)
    T = np.diag(d) + np.diag(e, 1) + np.diag(e, -1)
    nT = np.max(np.abs(w_ref))
    w, Z, info = gep.tridiag_eig(dev(d), dev(e))
    assert info == 0
    wh, Zh = host(w), host(Z)
    assert np.all(np.diff(wh) >= 0)
    assert np.max(np.abs(wh - w_ref)) <= 64 * M * EPS * nT
    assert np.max(np.abs(Zh.T @ Zh - np.eye(M))) <= 64 * M * EPS
    assert np.max(np.abs(T @ Zh - Zh * wh[None, :])) <= 64 * M * EPS * nT


def _bisection_cases():
    rng = np.random.default_rng(21)
    cases = []
    for M in (1, 2, 5, 63, 65, 300, 1300):
        cases.append((f"random{M}", rng.standard_normal(M), rng.standard_normal(M - 1)))
    n = 200
    i = np.arange(n)
    cases.append(("diagonal", 10.0 ** rng.uniform(-9, 3, n) * rng.choice([-1, 1], n), np.zeros(n - 1)))
    cases.append(("zero", np.zeros(n), np.zeros(n - 1)))
    cases.append(("zero_pivots", np.zeros(n), np.ones(n - 1)))                       # minors that vanish
    cases.append(("singular", np.where(i % 2, 2.0, 0.0), np.where(i[:-1] % 2, 0.0, 1e-8)))
    cases.append(("tiny", rng.standard_normal(n) * 1e-290, rng.standard_normal(n - 1) * 1e-290))
    cases.append(("huge", rng.standard_normal(n) * 1e290, rng.standard_normal(n - 1) * 1e290))
    cases.append(("steep", 10.0 ** (-i * 1.2), 10.0 ** (-i[:-1] * 1.2 - 0.6)))        # underflowing products
    cases.append(("weak", rng.standard_normal(n), np.where(rng.random(n - 1) < 0.5, 1e-170, 1e-9)))
    cases.append(("equal", np.full(n, 7.0), np.full(n - 1, 1e-15)))
    return cases


# Multisection on division-free Sturm counts: each count is exact for a matrix within a few eps of T,
# so an eigenvalue is within a few eps of the norm (the oracle's own bound is the same).
@pytest.mark.parametrize("name,d,e", _bisection_cases(), ids=lambda x: x if isinstance(x, str) else "")
def test_bisection_vs_oracle(gep, oracle_lib, name, d, e):
    # the oracle squares e as it stands: it is given T scaled by an exact power of two
    top = max(np.max(np.abs(d), initial=0.0), np.max(np.abs(e), initial=0.0))
    k = int(np.frexp(top)[1]) if top > 0 else 0
    ref = np.ldexp(oracle_lib.bisect(np.ldexp(d, -k), np.ldexp(e, -k)), k)
    nT = max(np.max(np.abs(ref)), 1e-300)
    w, Z, info = gep.tridiag_eig(dev(d), dev(e), want_vectors=False)
    assert info == 0 and Z is None
    wh = host(w)
    assert np.all(np.diff(wh) >= -16 * EPS * nT)
    assert np.max(np.abs(wh - ref)) <= 64 * EPS * nT
    if name == "diagonal":
        assert np.max(np.abs(wh - np.sort(d)) / np.abs(np.sort(d))) <= 4 * EPS
