"""The workloads this solver's speed is judged by, each a call of the public binding.

A case names an entry point ("kind"), its sizes and its options.  The pencils (A, B) have a
known spectrum, so that their eigenpairs are known without any solver:

    A = L0 S L0^T,  B = L0 L0^T,  S = Q diag(lam) Q^T,

L0 lower triangular with a band of 16 subdiagonals (diag U(1, 2), the rest N(0, 0.05^2): an
overlap matrix of orbitals with short range), Q = D1 H D2 H with H the orthonormal Hartley
transform and D1, D2 random signs (dense, entries close to normally distributed), lam spread
over [-20, 20] with the level spacing of a disordered solid (no two levels closer than half the
mean spacing).  Eigenvalues are lam and B-orthonormal eigenvectors L0^-T Q.
"""
import math

import torch

import paper_1504_06443_gb300 as gep

BAND = 16


def listed():
    return [
        # one k-point of a small unit cell, with the defaults of solve(): the smallest call,
        # where launches and synchronisations count
        dict(name="solve_64", kind="solve", M=64, sep="1stage", precision="fp64", reducer="twosided",
             vectors=True, n_want=0),
        # a molecule with the defaults of solve() (native FP64 throughout)
        dict(name="solve_fp64_500", kind="solve", M=500, sep="1stage", precision="fp64", reducer="twosided",
             vectors=True, n_want=0),
        # the two-stage workflow on a small cluster
        dict(name="solve_2stage_516", kind="solve", M=516, sep="2stage", precision="fp64_emulated",
             reducer="twosided", vectors=True, n_want=0),
        # the one-stage workflow with tensor-core products, an odd order
        dict(name="solve_1stage_1501", kind="solve", M=1501, sep="1stage", precision="fp64_emulated",
             reducer="twosided", vectors=True, n_want=0),
        # the two-stage workflow, all eigenpairs, at an ordinary order and at a large one: the
        # route of the headline benchmark
        dict(name="solve_2stage_2047", kind="solve", M=2047, sep="2stage", precision="fp64_emulated",
             reducer="twosided", vectors=True, n_want=0),
        dict(name="solve_2stage_8192", kind="solve", M=8192, sep="2stage", precision="fp64_emulated",
             reducer="twosided", vectors=True, n_want=0),
        # eigenvalues only: band structures, densities of states
        dict(name="values_4000", kind="solve", M=4000, sep="2stage", precision="fp64_emulated", reducer="twosided",
             vectors=False, n_want=0),
        # the occupied states only, with the explicit-inverse reducer
        dict(name="lowest_3000", kind="solve", M=3000, sep="2stage", precision="fp64_emulated",
             reducer="explicit_inv", vectors=True, n_want=750),
        # FP32-grade first pass and FP64 refinement
        dict(name="mixed_2048", kind="solve", M=2048, sep="2stage", precision="mixed_refined", reducer="twosided",
             vectors=True, n_want=0),
        # many small pencils (k-points, fragments), captured once and replayed
        dict(name="batched_24", kind="batched", count=24, lo=64, hi=768),
        # one step of fitting a Hamiltonian: density matrix forward, gradients backward
        dict(name="density_1000", kind="density", M=1000, n_occ=500),
        # the FP64-accurate product on its own
        dict(name="gemm_4096", kind="gemm", m=4096, n=4096, k=4096, ta="N", tb="N", engine="fp64_emulated"),
    ]


def _size(rng, lo, hi):
    """A whole number, log-uniform in [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    fam = rng.choice(["default", "1stage", "2stage", "values", "lowest", "mixed", "batched", "density", "gemm"])
    c = dict(kind="solve", sep="2stage", precision="fp64_emulated", reducer="twosided", vectors=True, n_want=0)
    if fam == "default":
        c.update(M=_size(rng, 32, 1024), sep="1stage", precision="fp64")
    elif fam == "1stage":
        c.update(M=_size(rng, 128, 3000), sep="1stage", reducer=rng.choice(["twosided", "explicit_inv"]))
    elif fam == "2stage":
        c.update(M=_size(rng, 256, 7000))
    elif fam == "values":
        c.update(M=_size(rng, 256, 6000), sep=rng.choice(["1stage", "2stage", "2stage"]), vectors=False)
    elif fam == "lowest":
        M = _size(rng, 256, 5000)
        c.update(M=M, n_want=rng.randint(M // 16, M // 2), reducer=rng.choice(["twosided", "explicit_inv"]))
    elif fam == "mixed":
        c.update(M=_size(rng, 256, 3000))
    elif fam == "batched":
        return dict(kind="batched", count=rng.randint(4, 32), lo=rng.randint(48, 96), hi=_size(rng, 128, 1024))
    elif fam == "density":
        M = _size(rng, 64, 2048)
        return dict(kind="density", M=M, n_occ=rng.randint(M // 8, M // 2))
    else:
        return dict(kind="gemm", m=_size(rng, 64, 6000), n=_size(rng, 64, 6000), k=_size(rng, 64, 6000),
                    ta=rng.choice(["N", "T"]), tb=rng.choice(["N", "T"]),
                    engine=rng.choice(["fp64_emulated", "fp64_emulated", "mixed_refined"]))
    return c


# ------------------------------------------------------------------ inputs

def _hartley(X, dim):
    F = torch.fft.fft(X, dim=dim)
    return (F.real - F.imag) / math.sqrt(X.shape[dim])


def _factors(M, seed):
    """lam (ascending), the signs of D1 and D2, and the subdiagonals 0..BAND of L0, on the GPU."""
    g = torch.Generator().manual_seed(int(seed) * 1000003 + M)
    f8 = torch.float64
    u = torch.rand(M, generator=g, dtype=f8)
    lam = -20.0 + 40.0 * (torch.arange(M, dtype=f8) + 0.25 + 0.5 * u) / M
    s1 = torch.randint(0, 2, (M,), generator=g).to(f8) * 2 - 1
    s2 = torch.randint(0, 2, (M,), generator=g).to(f8) * 2 - 1
    sub = 0.05 * torch.randn(BAND + 1, M, generator=g, dtype=f8)
    sub[0] = 1.0 + torch.rand(M, generator=g, dtype=f8)
    return lam.cuda(), s1.cuda(), s2.cuda(), sub.cuda()


def _apply_L0(sub, X):
    """L0 X, L0(i + o, i) = sub[o, i]."""
    M = X.shape[0]
    out = sub[0][:, None] * X
    for o in range(1, min(BAND, M - 1) + 1):
        out[o:] += sub[o, : M - o, None] * X[: M - o]
    return out


def _pencil(M, seed):
    lam, s1, s2, sub = _factors(M, seed)
    S = _hartley(_hartley(torch.diag(lam), 0), 1)
    S = _hartley(_hartley(s2[:, None] * S * s2[None, :], 0), 1)
    S = s1[:, None] * S * s1[None, :]
    A = _apply_L0(sub, _apply_L0(sub, S).t().contiguous())
    A = 0.5 * (A + A.t())
    B = _apply_L0(sub, _apply_L0(sub, torch.eye(M, dtype=torch.float64, device="cuda")).t().contiguous())
    B = 0.5 * (B + B.t())
    return A.contiguous(), B.contiguous()


def _eigenpairs(M, seed):
    """(lam ascending, Y = L0^-T Q with each column's largest entry positive)."""
    lam, s1, s2, sub = _factors(M, seed)
    Q = _hartley(torch.eye(M, dtype=torch.float64, device="cuda"), 0)
    Q = s1[:, None] * _hartley(s2[:, None] * Q, 0)
    L0 = _apply_L0(sub, torch.eye(M, dtype=torch.float64, device="cuda"))
    Y = torch.linalg.solve_triangular(L0.t(), Q, upper=True)
    top = Y.gather(0, Y.abs().argmax(0, keepdim=True))
    return lam, Y * torch.where(top < 0, -1.0, 1.0)


def _orders(case):
    """count orders, spread over the logarithm of [lo, hi]."""
    n, lo, hi = case["count"], case["lo"], case["hi"]
    return [int(round(math.exp(math.log(lo) + (math.log(hi) - math.log(lo)) * ((7 * i) % n + 0.5) / n)))
            for i in range(n)]


def _cotangents(case, seed):
    """The loss of the density case: sum lbar_k lambda_k + <W, P>."""
    M, n = case["M"], case["n_occ"]
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 17)
    lbar = torch.zeros(M, dtype=torch.float64, device="cuda")
    lbar[:n] = 1.0
    G = torch.randn(M, M, generator=g, dtype=torch.float64, device="cuda")
    return lbar, (G + G.t()) / math.sqrt(2.0)


def _factors_of_product(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 29)
    m, n, k = case["m"], case["n"], case["k"]
    a = torch.randn((k, m) if case["ta"] == "N" else (m, k), generator=g, dtype=torch.float64, device="cuda").t()
    b = torch.randn((n, k) if case["tb"] == "N" else (k, n), generator=g, dtype=torch.float64, device="cuda").t()
    return a, b  # column-major, as the library takes them


def prepare(case, seed):
    if case["kind"] == "gemm":
        a, b = _factors_of_product(case, seed)
        return dict(case=case, a=a, b=b)
    if case["kind"] == "batched":
        orders = _orders(case)
        pencils = [_pencil(m, int(seed) * 64 + i) for i, m in enumerate(orders)]
        bs = gep.BatchedSolver([p[0] for p in pencils], [p[1] for p in pencils], nstreams=16,
                               precision="fp64_emulated", seps=["2stage" if m > 512 else "1stage" for m in orders])
        bs.capture()
        return dict(case=case, solver=bs)
    A, B = _pencil(case["M"], seed)
    if case["kind"] == "density":
        lbar, W = _cotangents(case, seed)
        return dict(case=case, A=A.requires_grad_(), B=B.requires_grad_(), lbar=lbar, W=W)
    return dict(case=case, A=A, B=B)


def run(state):
    c = state["case"]
    if c["kind"] == "gemm":
        return gep.dgemm(state["a"], state["b"], c["ta"], c["tb"], engine=c["engine"])
    if c["kind"] == "batched":
        state["solver"].replay()
        return [list(p) for p in state["solver"].results()]
    if c["kind"] == "density":
        A, B = state["A"], state["B"]
        A.grad = B.grad = None
        lam, P = gep.eigh_density(A, B, c["n_occ"])
        ((state["lbar"] * lam).sum() + (state["W"] * P).sum()).backward()
        return lam.detach(), P.detach(), A.grad, B.grad
    return gep.solve(state["A"], state["B"], reducer=c["reducer"], sep=c["sep"], precision=c["precision"],
                     want_vectors=c["vectors"], n_want=c["n_want"])


def exact(case, seed):
    if case["kind"] == "gemm":
        a, b = _factors_of_product(case, seed)
        return (a if case["ta"] == "N" else a.t()) @ (b if case["tb"] == "N" else b.t())
    if case["kind"] == "batched":
        return [list(_eigenpairs(m, int(seed) * 64 + i)) for i, m in enumerate(_orders(case))]
    M = case["M"]
    lam, Y = _eigenpairs(M, seed)
    if case["kind"] == "solve":
        n = case["n_want"] or M
        return lam[:n], Y[:, :n] if case["vectors"] else None, None
    # first-order perturbation: dlambda_k = y_k^T (dA - lambda_k dB) y_k and, with P = Y_o Y_o^T,
    # dP through the occupied-empty rotations and the B-normalisation of the occupied block
    n = case["n_occ"]
    lbar, W = _cotangents(case, seed)
    P = Y[:, :n] @ Y[:, :n].t()
    F = Y.t() @ W @ Y
    G = torch.diag(lbar)
    H = -torch.diag(lbar * lam)
    lo, le = lam[:n, None], lam[None, n:]
    R = F[:n, n:] / (lo - le)
    G[:n, n:] = R
    G[n:, :n] = R.t()
    H[:n, :n] -= F[:n, :n]
    H[:n, n:] = -R * lo
    H[n:, :n] = (-R * lo).t()
    H = 0.5 * (H + H.t())
    return lam, P, Y @ G @ Y.t(), Y @ H @ Y.t()


def work(case):
    if case["kind"] == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 8.0 * (m * k + k * n + m * n), "flops": 2.0 * m * n * k}
    if case["kind"] == "batched":
        parts = [_solve_work(m, m) for m in _orders(case)]
        return {key: sum(p[key] for p in parts) for key in ("bytes", "flops")}
    M = case["M"]
    if case["kind"] == "density":
        w, n = _solve_work(M, M), case["n_occ"]
        # P, Y^T W Y on the occupied rows, Y G Y^T and Y H Y^T (symmetric results)
        return {"bytes": w["bytes"] + 8.0 * 4 * M * M, "flops": w["flops"] + M * M * n + 4.0 * M * M * n + 4.0 * M ** 3}
    return _solve_work(M, (case["n_want"] or M) if case["vectors"] else 0)


def _solve_work(M, n):
    """Cholesky M^3/3, reduction M^3, tridiagonalisation 4/3 M^3; with n eigenvectors the
    tridiagonal ones (at most 4/3 M^3, for all of them) and 3 M^2 n of back-transformation."""
    flops = (8.0 / 3.0) * M ** 3 + (4.0 / 3.0 * M * M * n + 3.0 * M * M * n if n else 0.0)
    return {"bytes": 8.0 * (2 * M * M + M * n + (n or M)), "flops": flops}
