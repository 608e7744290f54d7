"""Performance cases of the DFC-LRR library, each through its public entry
points (paper_1304_5583_gb300.binding): the singular-value thresholding on its
own, whole LRR / DFC-LRR solves in the three precisions, many small problems
at once, the tensor-core products and the differentiable unrolled iteration.

listed()              the named cases
draw(rng)             one more case of the same ranges
prepare(case, seed)   inputs and options on the GPU
run(state)            one pass, returning its outputs
work(case)            bytes and flops a pass cannot do without
exact(case, seed)     the outputs in 64 bits, by plain numpy / torch
"""
import math

import numpy as np
import torch

from paper_1304_5583_gb300 import binding, synth

TAU = 0.05          # threshold of the stand-alone SVT cases


def listed():
    return [
        # --- singular-value thresholding alone (lrr_svt): the solver's inner step offered by itself
        # a small matrix inside a user's own loop: launches and latency
        {"name": "svt_f32_60x80", "kind": "svt", "dtype": "f32", "rows": 60, "cols": 80, "rank": 12, "no_alloc": False},
        # one block of the 500 x 5000 problem: r = 350, 256 columns
        {"name": "svt_f32_350x256", "kind": "svt", "dtype": "f32", "rows": 350, "cols": 256, "rank": 100,
         "no_alloc": False},
        # one block of the 1000 x 20000 problem: r = 1000, 487 columns, 400 directions kept
        {"name": "svt_f32_1000x487", "kind": "svt", "dtype": "f32", "rows": 1000, "cols": 487, "rank": 400,
         "no_alloc": False},
        # wide, float64, fixed scratch: the shape of the 100 x 500 problem
        {"name": "svt_f64_100x500", "kind": "svt", "dtype": "f64", "rows": 100, "cols": 500, "rank": 25,
         "no_alloc": True},
        # --- whole solves
        # plain LRR in float64 to 1e-8 (the 100 x 500 problem)
        {"name": "lrr_f64_100x500", "kind": "solve", "precision": "f64", "m": 100, "subspaces": 5, "dim": 5,
         "points": 100, "outliers": 0.10, "blocks": 1, "min_cols": 0, "lam": 0.1, "eps": 1e-8, "autotune": False},
        # a small DFC problem, three blocks: launch-bound
        {"name": "dfc_f32_60x240", "kind": "solve", "precision": "f32", "m": 60, "subspaces": 4, "dim": 3,
         "points": 60, "outliers": 0.05, "blocks": 3, "min_cols": 64, "lam": 0.2, "eps": 1e-6, "autotune": False},
        # the 500 x 5000 problem, ten uneven blocks, float32
        {"name": "dfc_f32_500x5000", "kind": "solve", "precision": "f32", "m": 500, "subspaces": 10, "dim": 10,
         "points": 500, "outliers": 0.05, "blocks": 10, "min_cols": 200, "lam": 0.1, "eps": 1e-6, "autotune": False},
        # a batch of twelve blocks of 400 and more columns, mixed precision with the autotuner, as the benchmark runs
        {"name": "dfc_mixed_600x6000", "kind": "solve", "precision": "mixed", "m": 600, "subspaces": 10, "dim": 10,
         "points": 600, "outliers": 0.05, "blocks": 12, "min_cols": 400, "lam": 0.1, "eps": 1e-6, "autotune": True},
        # many small independent problems on concurrent streams (the phase-transition sweep)
        {"name": "batch_f32_8x60x100", "kind": "batch", "problems": 8, "m": 60, "subspaces": 3, "dim": 3, "points": 30,
         "outliers": 0.10, "lam": 0.5},
        # --- the tensor-core products by themselves
        # U^T P of the 1000 x 20000 problem for the whole batch
        {"name": "gemm_bf16_1000x20000x1000", "kind": "gemm", "dtype": "bf16", "M": 1000, "N": 20000, "K": 1000},
        # the same product of the 500 x 5000 problem, ragged, float32 operands (split TF32)
        {"name": "gemm_f32_350x5003x500", "kind": "gemm", "dtype": "f32", "M": 350, "N": 5003, "K": 500},
        # --- the differentiable unrolled iteration: forward and backward of a training step in float64
        {"name": "unrolled_f64_100x500", "kind": "unrolled", "m": 100, "subspaces": 5, "dim": 5, "points": 100,
         "outliers": 0.05, "K": 10, "lam": 0.1},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["svt", "svt", "svt", "solve", "solve", "batch", "gemm", "gemm", "unrolled"])
    if kind == "svt":
        if rng.random() < 0.25:
            small, large = _log_int(rng, 24, 120), _log_int(rng, 60, 500)
            dtype = "f64"
        else:
            small, large = _log_int(rng, 24, 500), _log_int(rng, 60, 1000)
            dtype = "f32"
        rows, cols = (small, large) if rng.random() < 0.5 else (large, small)
        p = min(rows, cols)
        return {"kind": "svt", "dtype": dtype, "rows": rows, "cols": cols,
                "rank": max(1, int(p * rng.uniform(0.1, 0.85))), "no_alloc": rng.random() < 0.3}
    if kind == "solve":
        if rng.random() < 0.2:
            k, d = rng.randint(3, 5), rng.randint(2, 5)
            return {"kind": "solve", "precision": "f64", "m": rng.randint(60, 100), "subspaces": k, "dim": d,
                    "points": rng.randint(40, 400 // k), "outliers": 0.1, "blocks": 1, "min_cols": 0, "lam": 0.1,
                    "eps": 1e-8, "autotune": False}
        m = _log_int(rng, 60, 600)
        k = rng.randint(3, 10)
        d = max(2, min(10, m // (5 * k), rng.randint(3, 10)))
        width = max(64, _log_int(rng, 3 * k * d, 500))        # columns of a block, on average
        t = rng.randint(2, 12)
        pts = max(20, width * t // k)
        return {"kind": "solve", "precision": rng.choice(["f32", "mixed"]), "m": m, "subspaces": k, "dim": d,
                "points": pts, "outliers": 0.05, "blocks": t, "min_cols": int(0.7 * (pts * k // t)),
                "lam": 0.2 if m < 200 else 0.1, "eps": 1e-6, "autotune": rng.random() < 0.3}
    if kind == "batch":
        return {"kind": "batch", "problems": rng.randint(2, 12), "m": rng.randint(40, 80), "subspaces": 3, "dim": 3,
                "points": rng.randint(20, 40), "outliers": rng.choice([0.05, 0.1, 0.2]), "lam": 0.5}
    if kind == "gemm":
        return {"kind": "gemm", "dtype": rng.choice(["bf16", "f32"]), "M": _log_int(rng, 60, 1000),
                "N": _log_int(rng, 200, 20000), "K": _log_int(rng, 60, 1000)}
    return {"kind": "unrolled", "m": rng.randint(40, 100), "subspaces": 4, "dim": rng.randint(2, 5),
            "points": rng.randint(30, 110), "outliers": 0.05, "K": rng.randint(4, 10), "lam": 0.1}


def _device(M, dtype):
    return torch.from_numpy(np.asfortranarray(M)).to(dtype).cuda()


def _svt_input(c, seed):
    # low rank plus noise below the threshold: what the J-step meets once the
    # kept directions have emerged
    g = torch.Generator(device="cuda").manual_seed(seed)
    kw = dict(generator=g, device="cuda", dtype=torch.float64)
    rows, cols, k = c["rows"], c["cols"], c["rank"]
    A = torch.randn(rows, k, **kw) @ torch.randn(k, cols, **kw) / math.sqrt(rows * cols)
    A += 1e-2 * torch.randn(rows, cols, **kw) / math.sqrt(max(rows, cols))
    dt = torch.float64 if c["dtype"] == "f64" else torch.float32
    return A.to(dt).t().contiguous().t()


def _solve_input(c, seed):
    d = synth.union_of_subspaces(seed, c["m"], c["subspaces"], c["dim"], c["points"], c["outliers"])
    perm, off = synth.column_partition(seed + 1, d.M.shape[1], c["blocks"], min_cols=c["min_cols"] or None, alpha=4.0)
    return d.M, perm, off


def _batch_input(c, seed):
    return [synth.union_of_subspaces(seed * 1009 + i, c["m"], c["subspaces"], c["dim"], c["points"], c["outliers"],
                                     recipe="paper").M for i in range(c["problems"])]


def _gemm_input(c, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    align = 8 if c["dtype"] == "bf16" else 1
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    ld = (c["K"] + align - 1) // align * align
    return (torch.randn(c["M"], ld, generator=g, device="cuda").to(dt),
            torch.randn(c["N"], ld, generator=g, device="cuda").to(dt))


def _unrolled_input(c, seed):
    d = synth.union_of_subspaces(seed, c["m"], c["subspaces"], c["dim"], c["points"], c["outliers"])
    n = d.M.shape[1]
    W = np.random.default_rng(seed + 1).standard_normal((n, n))
    return d.M, W


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "svt":
        return {"case": c, "A": _svt_input(c, seed)}
    if kind == "solve":
        M, perm, off = _solve_input(c, seed)
        dt = torch.float64 if c["precision"] == "f64" else torch.float32
        o = binding.options(c["lam"], eps=c["eps"], precision=c["precision"], autotune=c["autotune"])
        Md = _device(M, dt)
        ws = torch.empty(binding.workspace_bytes(Md, perm, off, o), dtype=torch.uint8, device="cuda")
        return {"case": c, "M": Md, "perm": perm, "off": off, "opts": o, "ws": ws}
    if kind == "batch":
        return {"case": c, "Ms": [_device(M, torch.float32) for M in _batch_input(c, seed)],
                "opts": binding.options(c["lam"], precision="f32")}
    if kind == "gemm":
        A, B = _gemm_input(c, seed)
        return {"case": c, "A": A, "B": B}
    M, W = _unrolled_input(c, seed)
    return {"case": c, "M": _device(M, torch.float64).requires_grad_(True), "W": _device(W, torch.float64),
            "lam": torch.tensor(c["lam"], dtype=torch.float64, device="cuda", requires_grad=True)}


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "svt":
        J, rank = binding.svt(state["A"], TAU, no_alloc=c["no_alloc"])
        return J, rank
    if kind == "solve":
        if c["blocks"] == 1:
            r = binding.lrr_solve(state["M"], state["perm"], state["opts"], workspace=state["ws"])
        else:
            r = binding.dfc_lrr_solve(state["M"], state["perm"], state["off"], state["opts"], workspace=state["ws"])
        return r.Z, r.S
    if kind == "batch":
        outs, _ = binding.solve_batch(state["Ms"], state["opts"])
        return [(Z, S) for Z, S, _ in outs]
    if kind == "gemm":
        f = binding.gemm_bf16 if c["dtype"] == "bf16" else binding.gemm_f32
        return f(state["A"], state["B"], c["M"], c["N"], c["K"])
    M, lam = state["M"], state["lam"]
    M.grad = lam.grad = None
    Z = binding.unrolled_lrr(M, lam, c["K"], mu0=0.1)
    ((Z * state["W"]) ** 2).sum().backward()
    return Z.detach(), M.grad, lam.grad


def _solve_work(m, n, t, el, iters):
    # the iteration's two m x r x l products for every block, and for the
    # iterations whose SVT acts (about half) its Gram, one eigensolve sweep
    # and the reconstruction
    r = min(m, n)
    l = n / t
    p = min(r, l)
    flops = iters * (4.0 * m * r * n + 0.5 * t * (4.0 * max(r, l) * p * p + 4.0 * p ** 3))
    return el * (2.0 * m * n + n * n), flops


def work(case):
    c, kind = case, case["kind"]
    if kind == "svt":
        el = 8 if c["dtype"] == "f64" else 4
        L, p = max(c["rows"], c["cols"]), min(c["rows"], c["cols"])
        return {"bytes": 2.0 * el * L * p, "flops": 4.0 * L * p * p + 4.0 * p ** 3}
    if kind == "solve":
        b, f = _solve_work(c["m"], c["subspaces"] * c["points"], c["blocks"], 8 if c["precision"] == "f64" else 4, 200)
        return {"bytes": b, "flops": f}
    if kind == "batch":
        n = c["subspaces"] * c["points"] / (1.0 - c["outliers"])
        b, f = _solve_work(c["m"], n, 1, 4, 200)
        return {"bytes": c["problems"] * b, "flops": c["problems"] * f}
    if kind == "gemm":
        el = 2 if c["dtype"] == "bf16" else 4
        return {"bytes": float(el * c["K"] * (c["M"] + c["N"]) + 4 * c["M"] * c["N"]),
                "flops": 2.0 * c["M"] * c["N"] * c["K"]}
    m, n = c["m"], c["subspaces"] * c["points"]
    r = min(m, n)
    # forward, its recomputation, and the reverse (about twice a forward) of K iterations
    per = 8.0 * m * n * n + 4.0 * r * n * n + 4.0 * n * r * r + 4.0 * r ** 3
    return {"bytes": 8.0 * (2 * m * n + 3 * n * n), "flops": 4.0 * c["K"] * per}


# ---------------------------------------------------------------- 64 bits
def _svt64(A, tau):
    U, s, Vh = torch.linalg.svd(A, full_matrices=False)
    k = int((s > tau).sum())
    return (U[:, :k] * (s[:k] - tau)) @ Vh[:k], U[:, :k]


def _alm64(M, cols, V, sig, lam, eps, rho=1.1, mu=1e-6, mu_max=1e10, max_iter=1000):
    """Inexact ALM of one block, min ||Z||_* + lam ||S||_{2,1} s.t. C = M Z + S, C = M[:, cols]; Z = V Zt with V, sig
    the right singular vectors and the singular values of M.  Returns Zt, S and the left factor of the last J."""
    C = M[:, cols]
    U = M @ V / sig
    g = 1.0 / (1.0 + sig * sig)
    Zt = torch.zeros(V.shape[1], len(cols), dtype=torch.float64, device=M.device)
    Y2, E, Y1 = torch.zeros_like(Zt), torch.zeros_like(C), torch.zeros_like(C)
    basis = None
    for _ in range(max_iter):
        J, basis = _svt64(Zt + Y2 / mu, 1.0 / mu) if float(torch.linalg.norm(Zt + Y2 / mu)) > 1.0 / mu else (
            torch.zeros_like(Zt), torch.zeros(V.shape[1], 0, dtype=torch.float64, device=M.device))
        Zt = g[:, None] * (sig[:, None] * (U.T @ (C - E + Y1 / mu)) + J - Y2 / mu)
        R = C - U @ (sig[:, None] * Zt)
        X = R + Y1 / mu
        nrm = torch.linalg.norm(X, dim=0)
        E = X * torch.where(nrm > lam / mu, 1.0 - lam / mu / nrm, torch.zeros_like(nrm))
        if max(float((R - E).abs().max()), float((V @ (Zt - J)).abs().max())) < eps:
            break
        Y1 = Y1 + mu * (R - E)
        Y2 = Y2 + mu * (Zt - J)
        mu = min(rho * mu, mu_max)
    return Zt, E, basis


def _solve64(Mh, perm, off, lam, eps):
    M = torch.from_numpy(Mh)
    _, s, Vh = torch.linalg.svd(M, full_matrices=False)
    r = int((s > 1e-6 * s[0]).sum())
    V, sig = Vh[:r].T.contiguous(), s[:r]
    Zs, Ss, Q = [], [], None
    for i in range(len(off) - 1):
        Zt, E, basis = _alm64(M, perm[off[i]:off[i + 1]], V, sig, lam, eps)
        Zs.append(Zt)
        Ss.append(E)
        Q = basis if i == 0 else Q
    Zt = torch.cat(Zs, 1)
    if len(off) > 2:
        Zt = Q @ (Q.T @ Zt)
    Z, S = torch.zeros(M.shape[1], M.shape[1], dtype=torch.float64), torch.zeros_like(M)
    Z[:, perm] = V @ Zt
    S[:, perm] = torch.cat(Ss, 1)
    return Z, S


class _SvtGrad(torch.autograd.Function):
    @staticmethod
    def forward(ctx, A, tau):
        U, s, Vh = torch.linalg.svd(A)
        ctx.save_for_backward(U, s, Vh)
        ctx.tau = tau
        return (U * torch.clamp(s - tau, min=0.0)) @ Vh

    @staticmethod
    def backward(ctx, G):
        U, s, Vh = ctx.saved_tensors
        f = torch.clamp(s - ctx.tau, min=0.0)
        P = U.T @ G @ Vh.T
        d = s[:, None] - s[None, :]
        on = (s > ctx.tau).to(s.dtype)
        gp = torch.where(d == 0, on[:, None].expand_as(d), (f[:, None] - f[None, :]) / torch.where(d == 0, 1.0, d))
        t = s[:, None] + s[None, :]
        gm = torch.where(t > 0, (f[:, None] + f[None, :]) / torch.where(t > 0, t, 1.0), torch.zeros_like(t))
        core = gp * 0.5 * (P + P.T) + gm * 0.5 * (P - P.T)
        return U @ core @ Vh, None


def _unrolled64(Mh, W, lam, K, mu=0.1, rho=1.1, mu_max=1e10):
    M = torch.from_numpy(Mh).requires_grad_(True)
    lam = torch.tensor(lam, dtype=torch.float64, requires_grad=True)
    n = M.shape[1]
    S = torch.eye(n, dtype=torch.float64) + M.T @ M
    Z, Y2 = torch.zeros(n, n, dtype=torch.float64), torch.zeros(n, n, dtype=torch.float64)
    E, Y1 = torch.zeros_like(Mh_t := M.detach()), torch.zeros_like(Mh_t)
    for _ in range(K):
        J = _SvtGrad.apply(Z + Y2 / mu, 1.0 / mu)
        Z = torch.linalg.solve(S, M.T @ (M - E + Y1 / mu) + J - Y2 / mu)
        R = M - M @ Z
        X = R + Y1 / mu
        nrm = torch.linalg.norm(X, dim=0)
        keep = nrm > lam.detach() / mu
        E = X * torch.where(keep, 1.0 - lam / mu / torch.where(keep, nrm, 1.0), torch.zeros_like(nrm))
        Y1 = Y1 + mu * (R - E)
        Y2 = Y2 + mu * (Z - J)
        mu = min(rho * mu, mu_max)
    ((Z * torch.from_numpy(W)) ** 2).sum().backward()
    return Z.detach(), M.grad, lam.grad


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "svt":
        J, U = _svt64(_svt_input(c, seed).double(), TAU)
        return J, U.shape[1]
    if kind == "solve":
        M, perm, off = _solve_input(c, seed)
        if c["precision"] != "f64":
            # the iterate returned is the one at which a float32 stop test
            # fired, often one iteration before or after the 64-bit run's, so
            # a free-running 64-bit solve is not its value (and past a few
            # hundred columns it takes minutes)
            return None
        return _solve64(M, perm, off, c["lam"], c["eps"])
    if kind == "batch":
        out = []
        for M in _batch_input(c, seed):
            n = M.shape[1]
            out.append(_solve64(M.astype(np.float32).astype(np.float64), np.arange(n), np.array([0, n]), c["lam"], 1e-6))
        return out
    if kind == "gemm":
        A, B = _gemm_input(c, seed)
        return A[:, :c["K"]].double() @ B[:, :c["K"]].double().t()
    M, W = _unrolled_input(c, seed)
    return _unrolled64(M, W, c["lam"], c["K"])
