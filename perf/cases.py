"""Performance cases: the calls a user of this package makes, on inputs made on the GPU.

A case names an entry point ("call") and its sizes; ``prepare`` draws the problem and the
vectors, ``run`` makes the one call, ``exact`` gives the same outputs from plain torch in 64
bits where that is quick enough, and ``work`` counts the bytes and operations of the call.

The problem is H = [[A, B], [-conj(B), -conj(A)]] with A = Q diag(d) Q^* hermitian and
B = G + G^T symmetric scaled to ||B||_2 = beta min(d), as in the repository's workloads; Q is
a product of Fourier (for real problems: Hartley) transforms and random phases (signs), a
dense unitary that costs O(n^2 log n), so that a problem of any size takes milliseconds.
The largest singular value of G + G^T for complex Gaussian G is 4 sqrt(n) to a few per cent.
"""
import math

import numpy as np
import torch

import paper_2601_10557_gb300 as cb

DEV = "cuda:0"


def listed():
    return [
        # The check of a handful of eigenpairs of a small problem: the smallest call, a few
        # launches whose latency is the time.
        dict(name="residuals_small", call="residuals", n=64, k=6),
        # The residual check of all the pairs of the n = 4096 workload in FP64.
        dict(name="residuals_n4096", call="residuals", n=4096, k=200),
        # The filter of the n = 512 workload (20 + 10 vectors, degree 20) in the default
        # precision.
        dict(name="filter_fp64_n512", call="filter", n=512, k=30, deg_lo=20, deg_hi=20, precision="fp64",
             spec="uniform", beta=0.3),
        # An FP64 filter with adaptive degrees and sizes that fit no tile, as later
        # iterations of a solve with part of the block locked have them.
        dict(name="filter_fp64_ragged", call="filter", n=1301, k=67, deg_lo=4, deg_hi=20, precision="fp64",
             spec="uniform", beta=0.3),
        # The FP64-accurate filter on the tensor cores.
        dict(name="filter_fp64tc_n2048", call="filter", n=2048, k=130, deg_lo=8, deg_hi=12, precision="fp64_tc",
             spec="groups8", beta=0.3),
        # The tensor-core filter, odd sizes and adaptive degrees (8 to 36).
        dict(name="filter_mixed_ragged", call="filter", n=3001, k=83, deg_lo=8, deg_hi=36, precision="mixed",
             spec="uniform", beta=0.3),
        # The tensor-core filter of the n = 4096 workload's first iteration.
        dict(name="filter_mixed_n4096", call="filter", n=4096, k=260, deg_lo=20, deg_hi=20, precision="mixed",
             spec="groups8", beta=0.3),
        # The tensor-core filter of the benchmark's n = 16384 workload over its whole block,
        # at the smallest degree of its adaptive range.
        dict(name="filter_mixed_n16384", call="filter", n=16384, k=1300, deg_lo=8, deg_hi=8, precision="mixed",
             spec="gapband", beta=0.3),
        # One Rayleigh-Ritz step in FP64 on a search space of 128 + 128 vectors.
        dict(name="rr_n2048", call="rr", n=2048, k=256),
        # The adjoint of the n = 8192 gradient workload's 100 eigenvalues.
        dict(name="grad_n8192", call="grad", n=8192, k=100),
        # A training step on the n = 512 workload: eigenvalues by a solve in the default
        # precision, and the gradient of a loss of them.  The tolerance leaves the gradient's
        # digits to FP64 rounding rather than to where the iteration stopped.
        dict(name="train_n512", call="train", n=512, nev=20, nex=20, deg=20, deg_hi=36, tol=1e-12,
             precision="fp64", spec="uniform", beta=0.3),
        # A whole mixed-precision solve of the n = 4096 workload.
        dict(name="solve_mixed_n4096", call="solve", n=4096, nev=200, nex=60, deg=20, deg_hi=36, tol=1e-10,
             precision="mixed", spec="groups8", beta=0.3),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["residuals", "filter", "filter", "filter", "filter", "rr", "grad", "train", "solve"])
    if call == "residuals":
        n = _log(rng, 64, 4096)
        return dict(call=call, n=n, k=_log(rng, 4, max(4, min(200, n // 8))))
    if call == "filter":
        precision = rng.choice(["fp64", "fp64_tc", "mixed", "mixed", "bf16x6"])
        top = {"fp64": 2048, "fp64_tc": 4096, "mixed": 8192, "bf16x6": 4096}[precision]
        n = _log(rng, 64, top)
        k = _log(rng, 6, max(6, min(n // 8, 600 if precision != "fp64" else 96)))
        lo = rng.choice([4, 8, 12, 20])
        return dict(call=call, n=n, k=k, deg_lo=lo, deg_hi=max(lo, rng.choice([lo, 20, 36])), precision=precision,
                    spec=rng.choice(["uniform", "groups8", "gapband"]), beta=rng.choice([0.3, 0.3, 0.4]),
                    real=rng.random() < 0.2)
    if call == "rr":
        n = _log(rng, 128, 2048)
        return dict(call=call, n=n, k=2 * _log(rng, 8, max(8, min(128, n // 8))))
    if call == "grad":
        n = _log(rng, 256, 8192)
        return dict(call=call, n=n, k=_log(rng, 8, max(8, min(200, n // 16))))
    n = _log(rng, 96, 768 if call == "train" else 2048)
    nev = _log(rng, 6, max(6, n // 24))
    if call == "train":
        return dict(call=call, n=n, nev=nev, nex=max(8, nev), deg=rng.choice([12, 20]), deg_hi=36, tol=1e-12,
                    precision=rng.choice(["fp64", "mixed"]), spec="uniform", beta=0.3)
    return dict(call=call, n=n, nev=nev, nex=max(8, nev // 2), deg=rng.choice([12, 20]), deg_hi=36, tol=1e-10,
                precision=rng.choice(["mixed", "mixed", "fp64_tc"]), spec=rng.choice(["uniform", "groups8"]),
                beta=0.3)


# ------------------------------------------------------------------------------- inputs
def _rand(gen, *shape):
    return torch.randn(shape, generator=gen, dtype=torch.complex128, device=DEV) * math.sqrt(2.0)


def _spectrum(kind, n, rng):
    """The spectra of the repository's workloads: U[1, 10]; eight bands of width 4.375 with
    gaps of 0.5 on [1, 39.5]; U[1, 50] with 5 % of the values in [1, 1.49]."""
    if kind == "uniform":
        return rng.uniform(1.0, 10.0, n)
    if kind == "groups8":
        band = (np.arange(n) * 8) // n
        return 1.0 + 4.875 * band + rng.uniform(0.0, 4.375, n)
    d = rng.uniform(1.0, 50.0, n)
    low = rng.choice(n, max(1, n // 20), replace=False)
    d[low] = rng.uniform(1.0, 1.49, len(low))
    return d


def _problem(case, seed, gen):
    """A, B on the GPU and the bounds (mu1, mu_nevex, muN) a filter of this spectrum has."""
    n, real = case["n"], bool(case.get("real", False))
    rng = np.random.default_rng(seed + 17)
    d = _spectrum(case.get("spec", "uniform"), n, rng)
    A = torch.zeros((n, n), dtype=torch.complex128, device=DEV)
    A.diagonal().copy_(torch.from_numpy(d))
    for _ in range(2):
        if real:
            s = torch.randint(0, 2, (n,), generator=gen, device=DEV) * 2.0 - 1.0
            for dim in (0, 1):
                F = torch.fft.fft(A, dim=dim, norm="ortho")
                A = (F.real - F.imag).to(torch.complex128) * (s[:, None] if dim == 0 else s[None, :])
        else:
            p = torch.polar(torch.ones(n, dtype=torch.float64, device=DEV),
                            2 * math.pi * torch.rand(n, generator=gen, dtype=torch.float64, device=DEV))
            A = torch.fft.fft(A, dim=0, norm="ortho") * p[:, None]
            A = torch.fft.ifft(A, dim=1, norm="ortho") * p.conj()[None, :]
    A = (A + A.conj().T) * 0.5
    G = _rand(gen, n, n)
    if real:
        G = G.real.to(torch.complex128)
    B = G + G.T
    norm = (2.0 * math.sqrt(2.0) if real else 4.0) * math.sqrt(n)
    beta = case.get("beta", 0.3)
    B *= beta * float(d.min()) / norm
    sd = np.sort(d)
    k = case.get("k", case.get("nev", 0) + case.get("nex", 0))
    mune = float(sd[min(n - 1, max(k, n // 16))])
    mu1 = min(0.93 * float(sd[0]), 0.5 * mune)
    return A.contiguous(), B.contiguous(), (mu1, mune, float(sd[-1]) + beta * float(sd[0]))


def _degrees(case, seed):
    rng = np.random.default_rng(seed + 5)
    return [int(x) for x in rng.integers(case["deg_lo"], case["deg_hi"] + 1, size=case["k"])]


def prepare(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    n = case["n"]
    s = dict(case=dict(case), seed=seed)
    if case["call"] == "grad":  # eigenvectors: a large upper and a small lower half
        V = _rand(gen, case["k"], 2 * n)
        V[:, n:] *= 0.1
        s["V"] = V / torch.linalg.vector_norm(V, dim=1, keepdim=True)
        s["w"] = torch.randn(case["k"], generator=gen, dtype=torch.float64, device=DEV)
        return s
    s["A"], s["B"], s["mu"] = _problem(case, seed, gen)
    if case["call"] == "residuals":
        W = _rand(gen, case["k"], 2 * n)
        s["W"] = W / torch.linalg.vector_norm(W, dim=1, keepdim=True)
        s["lam"] = torch.linspace(1.0, 3.0, case["k"], dtype=torch.float64, device=DEV)
    elif case["call"] == "filter":
        W = _rand(gen, case["k"], 2 * n)
        W[:, n:] *= 1e-3  # the solver's start block
        s["W"] = W
        s["degs"] = _degrees(case, seed)
    elif case["call"] == "rr":
        # an orthonormal basis closed under w -> K conj(w): [W, K conj(W)]
        W = _rand(gen, case["k"] // 2, 2 * n)
        W[:, n:] *= 1e-3
        both = torch.cat([W, torch.cat([W[:, n:], W[:, :n]], dim=1).conj()])
        for _ in range(2):
            L = torch.linalg.cholesky(both.conj() @ both.T)  # Gram matrix of the rows
            both = torch.linalg.solve_triangular(L.conj(), both, upper=False)
        s["Q"] = both.contiguous()
    elif case["call"] == "train":
        s["A"].requires_grad_(True)
        s["B"].requires_grad_(True)
        s["w"] = torch.randn(case["nev"], generator=gen, dtype=torch.float64, device=DEV)
    return s


# --------------------------------------------------------------------------------- calls
def _single(case):
    """The mixed filters work on single-precision iterates: a program that takes them keeps
    the block in complex64."""
    return case["precision"] in ("mixed", "bf16x6")


def run(s):
    case = s["case"]
    call = case["call"]
    if call == "residuals":
        return cb.residuals(s["A"], s["B"], s["W"], s["lam"])
    if call == "filter":
        mu1, mune, muN = s["mu"]
        W = cb.filter(s["A"], s["B"], s["W"].clone(), s["degs"], mu1, mune, muN, precision=case["precision"])
        return W.to(torch.complex64) if _single(case) else W
    if call == "rr":
        ritz, W = cb.rayleigh_ritz(s["A"], s["B"], s["Q"])
        return {"ritz": ritz, "W": W}
    if call == "grad":
        gA, gB = cb.grad(s["V"], s["w"])
        return {"gA": gA, "gB": gB}
    if call == "train":
        A, B = s["A"], s["B"]
        A.grad = B.grad = None
        lam = cb.eigvals(A, B, case["nev"], case["nex"], case["deg"], case["tol"], precision=case["precision"],
                         deg_max=case["deg_hi"], maxiter=50, seed=7)
        (lam * s["w"]).sum().backward()
        return {"lam": lam.detach(), "gA": A.grad, "gB": B.grad}
    # the eigenvectors are good to the tolerance over the gap, single precision
    lam, V, _ = cb.solve(s["A"], s["B"], case["nev"], case["nex"], case["deg"], case["tol"],
                         precision=case["precision"], deg_max=case["deg_hi"], maxiter=50, seed=7)
    return {"lam": lam, "V": V.to(torch.complex64)}


# --------------------------------------------------------------------- 64-bit reference
def _hop(A, B, W):
    """H w for the rows w = [x, y] of W."""
    n = A.shape[0]
    X, Y = W[:, :n], W[:, n:]
    return torch.cat([X @ A.T + Y @ B.T, -(X @ B.conj().T) - (Y @ A.conj().T)], dim=1)


def _spectral(A, B):
    """Positive eigenvalues (ascending) and right eigenvectors (rows) of H from the Cholesky
    factor of S H = [[A, B], [conj(B), conj(A)]] = L L^*: L^* S L y = lambda y."""
    n = A.shape[0]
    SH = torch.cat([torch.cat([A, B], 1), torch.cat([B.conj(), A.conj()], 1)])
    L = torch.linalg.cholesky(SH)
    sgn = torch.ones(2 * n, dtype=torch.float64, device=DEV)
    sgn[n:] = -1.0
    M = L.conj().T @ (sgn[:, None] * L)
    lam, y = torch.linalg.eigh((M + M.conj().T) * 0.5)
    v = sgn[:, None] * (L @ y[:, n:])
    return lam[n:], (v / torch.linalg.vector_norm(v, dim=0, keepdim=True)).T


def _adjoint(V, w):
    n = V.shape[1] // 2
    X, Y = V[:, :n], V[:, n:]
    c = w / (X.abs().square().sum(1) - Y.abs().square().sum(1))
    gA = (X.T * c) @ X.conj() + (Y.conj().T * c) @ Y
    gB = (X.T * c) @ Y.conj() + (Y.conj().T * c) @ X
    return gA, gB


def exact(case, seed):
    call, n = case["call"], case["n"]
    if call == "filter" and 256.0 * n * n * sum(_degrees(case, seed)) > 2.5e13:
        return None
    if call in ("train", "solve") and n > 1024:
        return None
    s = prepare(case, seed)
    if call == "grad":
        gA, gB = _adjoint(s["V"], s["w"])
        return {"gA": gA, "gB": gB}
    A, B = s["A"].detach(), s["B"].detach()
    if call == "residuals":
        R = _hop(A, B, s["W"]) - s["lam"][:, None] * s["W"]
        return torch.linalg.vector_norm(R, dim=1)
    if call == "filter":
        mu1, mune, muN = s["mu"]
        c, e = 0.5 * (mune ** 2 + muN ** 2), 0.5 * (muN ** 2 - mune ** 2)
        s1 = e / (mu1 ** 2 - c)
        degs = torch.tensor(s["degs"], device=DEV)
        prev, cur, sig = None, s["W"], s1
        out = torch.empty_like(cur)
        for j in range(int(degs.max())):
            T = _hop(A, B, _hop(A, B, cur)) - c * cur
            if j == 0:
                prev, cur = cur, (s1 / e) * T
            else:
                sn = 1.0 / (2.0 / s1 - sig)
                prev, cur = cur, (2.0 * sn / e) * T - sig * sn * prev
                sig = sn
            out[degs == j + 1] = cur[degs == j + 1]
        return out
    if call == "rr":
        Q = s["Q"].T
        sgn = torch.ones(2 * n, dtype=torch.float64, device=DEV)
        sgn[n:] = -1.0
        M = Q.conj().T @ (sgn[:, None] * _hop(A, B, s["Q"]).T)
        L = torch.linalg.cholesky((M + M.conj().T) * 0.5)
        N = Q.conj().T @ (sgn[:, None] * Q)
        Z = torch.linalg.solve_triangular(L, N, upper=False)
        G = torch.linalg.solve_triangular(L, Z.conj().T, upper=False)
        theta = torch.linalg.eigvalsh((G + G.conj().T) * 0.5)
        ritz = 1.0 / theta[case["k"] // 2:].flip(0)
        return {"ritz": ritz.cpu().numpy(), "W": None}  # each vector is free up to a phase
    lam, V = _spectral(A, B)
    nev = case["nev"]
    lam, V = lam[:nev], V[:nev]
    if call == "train":
        gA, gB = _adjoint(V, s["w"])
        return {"lam": lam, "gA": gA, "gB": gB}
    top = V[:, :n]
    big = torch.gather(top, 1, top.abs().argmax(1, keepdim=True))
    return {"lam": lam, "V": V * (big.conj() / big.abs())}


def work(case):
    """Bytes: A and B once, each block in and out once.  Operations: one application of H to
    a vector is a real 2n x 2n matrix on two real vectors of 2n entries, 16 n^2 (w = [x; y] is
    a sum of two vectors [z; conj z], for which H needs A z + B conj(z) alone)."""
    call, n = case["call"], float(case["n"])
    mat = 32.0 * n * n
    if call == "residuals":
        return {"bytes": mat + 32.0 * n * case["k"], "flops": 16.0 * n * n * case["k"]}
    if call == "filter":
        total = 0.5 * (case["deg_lo"] + case["deg_hi"]) * case["k"]
        out = 16.0 if _single(case) else 32.0
        return {"bytes": mat + (32.0 + out) * n * case["k"], "flops": 32.0 * n * n * total}
    if call == "rr":
        k = float(case["k"])  # H Q, two hermitian k x k products, W = Q Z; the k x k work
        return {"bytes": mat + 32.0 * n * k + 16.0 * n * k,
                "flops": 16.0 * n * n * k + 8.0 * n * k * k + 4.0 * n * k * k + 8.0 * n * k * k + 40.0 * k ** 3}
    if call == "grad":  # two n x n matrices of rank 2 nev, hermitian and symmetric
        return {"bytes": mat + 32.0 * n * case["k"], "flops": 16.0 * n * n * case["k"]}
    nevex = case["nev"] + case["nex"]  # about six filters over half the block, and the Rayleigh-Ritz steps
    k = 2.0 * nevex
    flops = 32.0 * n * n * 3.0 * case["deg"] * nevex + 6.0 * (16.0 * n * n * k + 28.0 * n * k * k + 40.0 * k ** 3)
    grads = mat + 16.0 * n * n * case["nev"] if call == "train" else 0.0
    return {"bytes": mat + 32.0 * n * case["nev"] + (mat if call == "train" else 0.0), "flops": flops + grads}
