"""The library's own work, as a program that uses it calls it.

Each case is one call (or one training step) through the package's public entry points, on seeded
synthetic inputs with the shapes and distributions of the workloads in
`paper_2207_06856_gb300/workloads.py`:

  mvm       gp_kmvm, the kernel MVM inside every solve, per precision option;
  mean      gp_kmvm on test points: the posterior mean of a solved system;
  backward  gp_kmvm_vjp_prec, the gradient of u^T K w that a training step ends with;
  precond   gp_pivchol_precond, once per hyperparameter setting;
  solve     gp_cg_solve with the preconditioner it was given;
  step      one training step: factor, solves and gradient through torch autograd.

`prepare` makes what such a program holds before the call, `run` is the call, `exact` restates the
result in plain FP64 torch.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2207_06856_gb300 import autograd, gpk

KERNEL = {"rbf": gpk.RBF, "matern32": gpk.MATERN32, "matern52": gpk.MATERN52}

# MVM options as the solvers, the server and the benchmark set them
OPTION = {
    "fp16": gpk.FP16,                                              # default: kernel values rounded once
    "hilo": gpk.FP16 | gpk.MVM_PSPLIT | gpk.MVM_XSPLIT,            # first phase of the relaxed solve
    "fp32pv": gpk.FP16 | gpk.MVM_XSPLIT | gpk.MVM_FP32_PV,         # the server's: FP32 value product, R <= 4
    "fp32": gpk.FP32,                                              # true-residual checks, the mean
}


def listed() -> list:
    return [
        # the smallest request a server gets (N log-uniform from 1,000; d in {4, 8, 16}): one CG step's MVM
        {"name": "mvm_request_smallest", "op": "mvm", "option": "fp32pv", "kernel": "rbf", "N": 1000, "d": 4, "R": 1,
         "inputs": "normal"},
        # a large request: the MVM that sets the server's tail
        {"name": "mvm_request_large", "op": "mvm", "option": "fp32pv", "kernel": "matern32", "N": 100_003, "d": 16,
         "R": 1, "inputs": "normal"},
        # the headline solve's MVM: Kin40K-like, [y, z_1..z_16]
        {"name": "mvm_solve", "op": "mvm", "option": "fp16", "kernel": "rbf", "N": 65_536, "d": 8, "R": 17,
         "inputs": "normal"},
        # the same solve's first phase (kernel tile and inputs as hi + lo), on an odd number of points
        {"name": "mvm_solve_hilo", "op": "mvm", "option": "hilo", "kernel": "rbf", "N": 50_021, "d": 8, "R": 17,
         "inputs": "normal"},
        # HouseElectric-like training MVM (d = 11, Matern-3/2), the largest that takes tens of milliseconds
        {"name": "mvm_training", "op": "mvm", "option": "fp16", "kernel": "matern32", "N": 196_613, "d": 11, "R": 17,
         "inputs": "mixture"},
        # the FP32 MVM of every true-residual check
        {"name": "mvm_check_fp32", "op": "mvm", "option": "fp32", "kernel": "rbf", "N": 32_768, "d": 8, "R": 17,
         "inputs": "normal"},
        # the posterior mean at 1,024 test points after a large solve
        {"name": "mean_request", "op": "mean", "option": "fp32", "kernel": "matern32", "N": 150_001, "d": 16, "R": 1,
         "n_test": 1024, "inputs": "normal"},
        # the gradient of a training step (Elevators-like, d = 18), inputs' gradient included
        {"name": "backward_training", "op": "backward", "kernel": "rbf", "N": 65_536, "d": 18, "R": 17,
         "inputs": "mixture"},
        # the headline solve's rank-100 preconditioner
        {"name": "precond_rank100", "op": "precond", "kernel": "rbf", "N": 65_536, "d": 8, "rank": 100,
         "inputs": "normal"},
        # a small request's whole solve, a fixed budget of steps: launches and the host's part count
        {"name": "solve_request", "op": "solve", "option": "fp32pv", "kernel": "matern32", "N": 2000, "d": 8, "R": 1,
         "rank": 20, "iters": 25, "inputs": "normal"},
        # the paper's budget of CG steps on 17 right-hand sides
        {"name": "solve_17rhs", "op": "solve", "option": "hilo", "kernel": "rbf", "N": 32_768, "d": 8, "R": 17,
         "rank": 100, "iters": 30, "inputs": "normal"},
        # one step of the training loop: factor, 17 solves, gradient, log-determinant
        {"name": "training_step", "op": "step", "kernel": "rbf", "N": 20_011, "d": 18, "R": 17, "rank": 100,
         "iters": 12, "inputs": "mixture"},
    ]


def _log_uniform(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    """One more case of the listed ranges: N over its logarithm, every d, R and kernel of the listed workloads."""
    op = rng.choice(["mvm", "mvm", "mvm", "mvm", "mean", "backward", "precond", "solve", "step"])
    kernel = rng.choice(["rbf", "matern32"])
    c = {"op": op, "kernel": kernel, "d": rng.choice([4, 8, 11, 16, 18]),
         "inputs": "mixture" if op in ("backward", "step") else rng.choice(["normal", "mixture"])}
    if op == "mvm":
        option = rng.choice(["fp16", "hilo", "fp32pv", "fp32"])
        hi = {"fp16": 196_613, "hilo": 100_003, "fp32pv": 196_613, "fp32": 50_021}[option]
        return {**c, "option": option, "N": _log_uniform(rng, 1000, hi), "R": 1 if option == "fp32pv" else rng.randint(1, 17)}
    if op == "mean":
        return {**c, "option": "fp32", "N": _log_uniform(rng, 1000, 200_000), "R": 1, "n_test": _log_uniform(rng, 100, 4096)}
    if op == "backward":
        return {**c, "N": _log_uniform(rng, 2000, 131_101), "R": rng.randint(2, 17)}
    if op == "precond":
        return {**c, "N": _log_uniform(rng, 1000, 196_613), "rank": rng.choice([20, 100])}
    if op == "solve":
        if rng.random() < 0.5:
            return {**c, "option": "fp32pv", "N": _log_uniform(rng, 1000, 20_000), "R": 1, "rank": 20,
                    "iters": rng.randint(10, 25)}
        return {**c, "option": "hilo", "N": _log_uniform(rng, 1000, 50_021), "R": rng.randint(2, 17), "rank": 100,
                "iters": rng.randint(10, 25)}
    return {**c, "N": _log_uniform(rng, 2000, 30_011), "R": rng.randint(5, 17), "rank": 100, "iters": 12}


# ---- inputs ------------------------------------------------------------------------------------

_ctx = None


def _context() -> gpk.Context:
    """The program's one library context (a handle that it keeps)."""
    global _ctx
    if _ctx is None:
        _ctx = gpk.Context(0, 64 << 20)
    return _ctx


def _inputs(case: dict, seed: int) -> dict:
    """X, X*, targets, probes and hyperparameters on the GPU, in the library's layouts."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    N, d = case["N"], case["d"]

    def normal(*shape):
        return torch.randn(shape, generator=g, device="cuda")

    if case["inputs"] == "mixture":   # the training workloads
        means, std = 2.0 * normal(8, d), 0.3 + 0.9 * torch.rand((8, d), generator=g, device="cuda")
        lab = torch.randint(0, 8, (N,), generator=g, device="cuda")
        X = means[lab] + std[lab] * normal(N, d)
    else:
        X = normal(N, d)
    X = (X - X.mean(0)) / X.std(0)
    y = torch.sin(2.0 * math.pi * X.mean(1)) + 0.1 * normal(N)
    R = case.get("R", 1)
    Z = (torch.randint(0, 2, (max(R - 1, 1), N), generator=g, device="cuda") * 2 - 1).float()
    r = np.random.default_rng(int(seed))
    if case["op"] == "mean" or case.get("option") == "fp32pv":
        hyp = (r.uniform(0.8, 2.0), r.uniform(0.5, 2.0), r.uniform(0.05, 0.1))   # a request's own hyperparameters
    else:
        hyp = (1.0 if d < 16 else 2.0, 1.0, 0.05)
    ls = np.full(d, hyp[0]) * r.uniform(0.9, 1.1, size=d)
    return {"X": X.float().contiguous(), "y": y.float().contiguous(), "Z": Z.contiguous(), "normal": normal,
            "hyp": gpk.Hyper(KERNEL[case["kernel"]], ls, float(hyp[1]), float(hyp[2]))}


def prepare(case: dict, seed: int) -> dict:
    i = _inputs(case, seed)
    X, y, Z, normal, hyp = i["X"], i["y"], i["Z"], i["normal"], i["hyp"]
    op, R = case["op"], case.get("R", 1)
    s = {"op": op, "case": case, "ctx": _context(), "hyp": hyp, "X": X}
    if op in ("mvm", "solve"):
        s["V"] = torch.cat([y[None], Z])[:R].contiguous()
    if op == "mean":
        s["Xt"] = normal(case["n_test"], case["d"])
        s["V"] = (y + 0.3 * normal(case["N"]))[None].contiguous()   # the solution of the request's system
    if op == "backward":
        # [u_1..u_M, u_0] and [z_1/(2M).., -u_0/2] of the pseudo-loss
        Z = Z[:R - 1]
        u0 = (y + 0.3 * normal(case["N"]))[None]
        s["U"] = torch.cat([0.7 * Z + 0.5 * normal(*Z.shape), u0]).contiguous()
        s["W"] = torch.cat([Z / (2 * (R - 1)), -0.5 * u0]).contiguous()
    if op == "solve":
        s["precond"] = _factor(X, hyp, case["rank"])
    if op == "step":
        s["y"], s["Z"] = y, normal(R - 1, case["N"])
        s["E"] = normal(R - 1, case["rank"])
        s["theta"] = [torch.tensor(hyp.lengthscale, requires_grad=True),
                      torch.tensor(hyp.outputscale, dtype=torch.float32, requires_grad=True),
                      torch.tensor(hyp.noise, dtype=torch.float32, requires_grad=True)]
        s["cfg"] = autograd.FitConfig(ctx=s["ctx"], kernel=hyp.kernel, rank=case["rank"], tol=1.0,
                                      max_iter=case["iters"], min_iter=case["iters"])
    return s


def run(s: dict):
    case, op = s["case"], s["op"]
    if op == "mvm":
        return gpk.kmvm(s["ctx"], s["hyp"], s["X"], s["V"], precision=OPTION[case["option"]], add_noise=True)
    if op == "mean":
        return gpk.kmvm(s["ctx"], s["hyp"], s["Xt"], s["V"], Xc=s["X"], precision=OPTION[case["option"]])
    if op == "backward":
        g, gX = gpk.kmvm_vjp(s["ctx"], s["hyp"], s["X"], s["U"], s["W"], want_X=True, precision="fp16")
        return {"theta": torch.from_numpy(g).float(), "X": gX}   # the parameters are float32
    if op == "precond":
        p = gpk.pivchol_precond(s["ctx"], s["hyp"], s["X"], case["rank"])
        return {"L": p.L, "core": p.core, "piv": p.piv}
    if op == "solve":
        U, status, info = gpk.cg_solve(s["ctx"], s["hyp"], s["X"], s["V"], s["precond"], tol=1e-6,
                                       max_iter=case["iters"], precision=OPTION[case["option"]])
        return U
    for t in s["theta"]:
        t.grad = None
    loss = autograd.MarginalLikelihood.apply(*s["theta"], s["X"], s["y"], s["Z"], s["E"], s["cfg"])
    loss.backward()
    return {"loss": float(loss.detach()), "lengthscale": s["theta"][0].grad, "outputscale": s["theta"][1].grad,
            "noise": s["theta"][2].grad}


# ---- work: what a pass cannot do without ---------------------------------------------------------


def _pairs(case: dict) -> float:
    return float(case.get("n_test") or case["N"]) * case["N"]


def work(case: dict) -> dict:
    op, N, d, R = case["op"], case["N"], case["d"], case.get("R", 1)
    if op in ("mvm", "mean"):
        rows = case.get("n_test") or N
        # inputs and vectors in, products out; per pair: squared distance, kernel value, R multiply-adds
        return {"bytes": 4.0 * (N * d + (rows * d if op == "mean" else 0) + R * N + R * rows),
                "flops": _pairs(case) * (2 * d + 4 + 2 * R)}
    if op == "backward":
        # X, U, W in, gX out; per pair: distance, k', U W^T both ways, W' X
        return {"bytes": 4.0 * (2 * N * d + 2 * R * N), "flops": _pairs(case) * (2 * d + 6 + 4 * R + 2 * (d + 1))}
    if op == "precond":
        k = case["rank"]
        return {"bytes": 4.0 * (N * d + N * k), "flops": N * (k * (2.0 * d + 4) + 2.0 * k * k)}
    k, J = case["rank"], case["iters"]
    mvm = _pairs(case) * (2 * d + 4 + 2 * R)
    if op == "solve":
        # per step: one MVM, the Woodbury apply, the projections on the earlier residuals
        return {"bytes": 4.0 * (N * d + N * k + 2 * R * N) + 4.0 * J * (N * k + (8 + J) * R * N),
                "flops": J * (mvm + 4.0 * N * k * R) + 2.0 * J * J * R * N}
    return {"bytes": 4.0 * (N * d + 2 * N * k + 4 * R * N) + 4.0 * J * (N * k + (8 + J) * R * N),
            "flops": J * (mvm + 4.0 * N * k * R) + _pairs(case) * (4 * d + 8 + 4 * R) + 2.0 * N * k * k}


# ---- plain FP64 ------------------------------------------------------------------------------------


def _unit(kernel: int, q: torch.Tensor):
    """k and dk/d(r^2) of the unit kernel at squared distances q."""
    if kernel == gpk.RBF:
        k = torch.exp(-0.5 * q)
        return k, -0.5 * k
    if kernel == gpk.MATERN32:
        u = torch.sqrt(3.0 * q)
        e = torch.exp(-u)
        return (1.0 + u) * e, -1.5 * e
    u = torch.sqrt(5.0 * q)
    e = torch.exp(-u)
    return (1.0 + u + u * u / 3.0) * e, -(5.0 / 6.0) * (1.0 + u) * e


def _sq(A: torch.Tensor, B: torch.Tensor) -> torch.Tensor:
    return ((A * A).sum(1)[:, None] + (B * B).sum(1)[None] - 2.0 * A @ B.T).clamp_(min=0.0)


def _kernel64(Xr, Xc, hyp) -> torch.Tensor:
    il = 1.0 / torch.tensor(hyp.lengthscale, dtype=torch.float64, device=Xr.device)
    return hyp.outputscale * _unit(hyp.kernel, _sq(Xr.double() * il, Xc.double() * il))[0]


def _mvm64(Xr, Xc, hyp, V) -> torch.Tensor:
    """K(Xr, Xc) V for V (R, Nc), by blocks of rows."""
    step = max(1, (1 << 28) // Xc.shape[0])
    return torch.cat([_kernel64(Xr[a:a + step], Xc, hyp) @ V.double().T for a in range(0, Xr.shape[0], step)]).T


def _factor(X: torch.Tensor, hyp, rank: int) -> gpk.Precond:
    """Rank-k pivoted Cholesky of K and its Woodbury core, in FP64 (a preconditioner that the caller holds)."""
    N = X.shape[0]
    L = torch.zeros((rank, N), dtype=torch.float64, device=X.device)
    diag = torch.full((N,), float(hyp.outputscale), dtype=torch.float64, device=X.device)
    piv = torch.zeros((rank,), dtype=torch.int64, device=X.device)
    for m in range(rank):
        p = torch.argmax(diag)
        piv[m] = p
        row = _kernel64(X[p][None], X, hyp)[0]
        l = (row - L[:m].T @ L[:m, p]) / torch.sqrt(diag[p])
        L[m] = l
        diag = (diag - l * l).index_fill(0, p[None], 0.0)
    L32 = L.float().contiguous()
    C = torch.eye(rank, dtype=torch.float64, device=X.device) + L32.double() @ L32.double().T / hyp.noise
    core = torch.linalg.cholesky(C).T.contiguous()    # column-major lower factor
    return gpk.Precond(L32, core, piv.int(), rank)


def _pcg64(K, B, L, noise: float, iters: int):
    """`iters` steps of preconditioned CG with K dense FP64; (solutions, alphas, betas, r_0^T P^-1 r_0) per column."""
    k = L.shape[0]
    C = torch.linalg.cholesky(torch.eye(k, dtype=K.dtype, device=K.device) + L @ L.T / noise)

    def P(w):   # rows are vectors
        return w / noise - (torch.cholesky_solve(L @ w.T, C).T @ L) / noise ** 2

    x, r = torch.zeros_like(B), B.clone()
    z = P(r)
    p, gam = z.clone(), (r * z).sum(1)
    rho, zeta, al, be, g0 = [], [], [], [], gam.clone()
    for _ in range(iters):
        rho.append(r / gam.sqrt()[:, None])
        zeta.append(z / gam.sqrt()[:, None])
        q = p @ K
        a = gam / (p * q).sum(1)
        x, r = x + a[:, None] * p, r - a[:, None] * q
        for _ in range(2):
            for u, v in zip(rho, zeta):
                r = r - (v * r).sum(1)[:, None] * u
        z = P(r)
        new = (r * z).sum(1)
        al.append(a)
        be.append(new / gam)
        p, gam = z + (new / gam)[:, None] * p, new
    return x, torch.stack(al), torch.stack(be), g0, C


def exact(case: dict, seed: int):
    s = prepare(case, seed)
    op, hyp, X = s["op"], s["hyp"], s["X"]
    if op == "mvm":
        return _mvm64(X, X, hyp, s["V"]) + hyp.noise * s["V"].double()
    if op == "mean":
        return _mvm64(s["Xt"], X, hyp, s["V"])
    if op == "backward":
        il = 1.0 / torch.tensor(hyp.lengthscale, dtype=torch.float64, device=X.device)
        gl, ga, gX = _vjp64(X.double(), il, hyp, s["U"].double(), s["W"].double())
        gs = (s["U"].double() * s["W"].double()).sum()
        return {"theta": torch.cat([gl, ga[None], gs[None]]), "X": gX}
    if op == "solve" and case["N"] <= 40_000:
        K = _mvm_dense(X, hyp)
        return _pcg64(K, s["V"].double(), s["precond"].L.double(), hyp.noise, case["iters"])[0]
    return None   # the pivots and the stopping of a training step are decided in FP32


def _mvm_dense(X, hyp) -> torch.Tensor:
    K = torch.empty((X.shape[0], X.shape[0]), dtype=torch.float64, device=X.device)
    for a in range(0, X.shape[0], 4096):
        K[a:a + 4096] = _kernel64(X[a:a + 4096], X, hyp)
    K.diagonal().add_(hyp.noise)
    return K


def _vjp64(X, il, hyp, U, W):
    """Gradients of sum_c u_c^T K w_c with respect to (l, a^2) and X."""
    A = X * il
    D = torch.zeros_like(A)
    ga = torch.zeros((), dtype=torch.float64, device=X.device)
    step = max(1, (1 << 27) // X.shape[0])
    for a in range(0, X.shape[0], step):
        k, dk = _unit(hyp.kernel, _sq(A[a:a + step], A))
        G = U[:, a:a + step].T @ W
        ga += (G * k).sum()
        H = hyp.outputscale * dk * (G + W[:, a:a + step].T @ U)
        D[a:a + step] = A[a:a + step] * H.sum(1, keepdim=True) - H @ A
    return -2.0 * il * (A * D).sum(0), ga, 2.0 * il * D
