"""Pivoted-Cholesky preconditioner (gp_pivchol_precond) and CG (gp_cg_solve,
Alg. 1 / Alg. 2) on the GPU against the FP64 oracle.

Solves are judged by their FP64-recomputed relative residual
||Ktilde U - B|| / ||B|| per column (the trajectory itself is not pinned)."""

import math

import numpy as np
import pytest

import oracle as O
from paper_2207_06856_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
KNAME = {0: "rbf", 1: "matern32", 2: "matern12", 3: "matern52"}


@pytest.fixture(scope="module")
def ctx():
    from paper_2207_06856_gb300 import gpk
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    c = gpk.Context(0)
    yield c
    c.close()


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda:0")


def _ohyp(w):
    return O.Hyp(KNAME[w.kernel], w.lengthscale, w.outputscale, w.noise)


def test_pivchol_invariants(ctx):
    from paper_2207_06856_gb300 import gpk
    X, _, kern, ls, a2, s2 = workloads.random_problem(1500, 5, 1, seed=21, kernel=1)
    hyp = gpk.Hyper(kern, ls, a2, s2)
    pc = gpk.pivchol(ctx, hyp, _dev(X), 30)
    ctx.check()
    assert pc.rank == 30
    L = pc.L.cpu().numpy().astype(np.float64).T          # N x k
    piv = pc.piv.cpu().numpy()
    oh = O.Hyp("matern32", ls, a2, s2)
    K = O.kernel_matrix(X, X, oh)
    assert piv[0] == 0 and len(set(piv.tolist())) == 30
    # interpolation: (L L^T)[p, :] = K[p, :] for the pivots (FP32 rows)
    assert np.max(np.abs((L @ L.T)[piv] - K[piv])) < 2e-4 * a2
    rem = np.diag(K) - np.sum(L * L, axis=1)
    assert rem.min() > -1e-4
    # the first pivots agree with the FP64 oracle (later ones may swap on near-ties)
    _, opiv = O.pivoted_cholesky(X, oh, 8)
    assert list(piv[:8]) == list(opiv[:8])
    # core: lower Cholesky factor of I + L^T L / sigma^2, in FP64
    Lc = pc.core.cpu().numpy().T
    C = np.eye(30) + (L.T @ L) / s2
    np.testing.assert_allclose(Lc @ Lc.T, C, rtol=1e-5, atol=1e-5 * np.abs(C).max())


@pytest.mark.parametrize("alg", ["stable", "standard"])
def test_plain_config_fp32(ctx, alg):
    """Plain workload: N = 2048, d = 8, RBF l = 0.5, sigma^2 = 0.01, rank 20,
    tol 1e-4, FP32 on the GPU vs the FP64 oracle."""
    from paper_2207_06856_gb300 import gpk
    w = workloads.plain()
    hyp = gpk.Hyper(w.kernel, w.lengthscale, w.outputscale, w.noise)
    X = _dev(w.X)
    pc = gpk.pivchol(ctx, hyp, X, w.rank)
    B = w.rhs()
    U, st, info = gpk.cg_solve(ctx, hyp, X, _dev(B), pc, tol=w.tol, max_iter=w.max_iter, precision="fp32",
                               algorithm=alg, reorth="pinv" if alg == "stable" else "none", restarts=4)
    ctx.check()
    assert st == gpk.GP_OK, info
    res = O.relative_residual(w.X, U.cpu().numpy().T, B.T, _ohyp(w))
    assert res.max() <= w.tol, res
    ref = O.cholesky_solve(w.X, _ohyp(w), B.T.astype(np.float64))
    err = np.linalg.norm(U.cpu().numpy().T - ref) / np.linalg.norm(ref)
    assert err < 1e-2


@pytest.mark.parametrize("prec", ["fp16", "bf16", "fp32"])
@pytest.mark.parametrize("kern", [0, 1])
def test_stable_cg_precision_workload_small(ctx, prec, kern):
    """The precision workload at N = 6000 (1 + 16 RHS, rank 100 preconditioner):
    the FP64 residual of every column is <= 1e-2."""
    from paper_2207_06856_gb300 import gpk
    w = workloads.precision(N=6000, kernel=kern)
    hyp = gpk.Hyper(w.kernel, w.lengthscale, w.outputscale, w.noise)
    X = _dev(w.X)
    pc = gpk.pivchol(ctx, hyp, X, w.rank)
    B = w.rhs()
    U, st, info = gpk.cg_solve(ctx, hyp, X, _dev(B), pc, tol=w.tol, max_iter=400, precision=prec)
    ctx.check()
    assert st == gpk.GP_OK, (info["col_iters"], info["rel_resid"])
    res = O.relative_residual(w.X, U.cpu().numpy().T, B.T, _ohyp(w))
    assert res.max() <= w.tol, res


def test_reorth_modes_and_standard_agree_on_small_problem(ctx):
    """All variants reach the same solution on a well-conditioned small problem."""
    from paper_2207_06856_gb300 import gpk
    X, V, kern, ls, a2, s2 = workloads.random_problem(900, 4, 3, seed=22, noise=0.1)
    hyp = gpk.Hyper(kern, ls, a2, s2)
    Xd, Bd = _dev(X), _dev(V)
    pc = gpk.pivchol(ctx, hyp, Xd, 10)
    ref = O.cholesky_solve(X, O.Hyp("rbf", ls, a2, s2), V.T.astype(np.float64))
    for alg, ro, pre in [("stable", "pinv", pc), ("stable", "euclid", None), ("stable", "none", pc),
                         ("standard", "none", pc), ("stable", "pinv", None)]:
        U, st, info = gpk.cg_solve(ctx, hyp, Xd, Bd, pre, tol=1e-6, max_iter=300, precision="fp32", algorithm=alg,
                                   reorth=ro, reorth_passes=2)
        ctx.check()
        assert st == gpk.GP_OK, (alg, ro, info["rel_resid"])
        err = np.linalg.norm(U.cpu().numpy().T - ref) / np.linalg.norm(ref)
        assert err < 1e-4, (alg, ro, err)


def test_cg_trajectory_matches_oracle_alg2(ctx):
    """Parity unpinned beyond the solution, but in FP32 the first step sizes of
    Alg. 2 follow the FP64 oracle's closely."""
    from paper_2207_06856_gb300 import gpk
    X, V, kern, ls, a2, s2 = workloads.random_problem(700, 3, 1, seed=23, noise=0.05)
    hyp = gpk.Hyper(kern, ls, a2, s2)
    Xd = _dev(X)
    pc = gpk.pivchol(ctx, hyp, Xd, 8)
    U, st, info = gpk.cg_solve(ctx, hyp, Xd, _dev(V), pc, tol=1e-5, max_iter=100, precision="fp32", restarts=0)
    oh = O.Hyp("rbf", ls, a2, s2)
    piv_np = pc.piv.cpu().numpy()
    L64, _ = O.pivoted_cholesky(X, oh, 8)
    Kt = O.ktilde_dense(X, oh)
    ores = O.cg_stable(lambda v: Kt @ v, V[0].astype(np.float64),
                       precond=lambda r: O.precond_apply(L64, s2, r), tol=1e-5, max_iter=100)
    assert list(piv_np) == list(O.pivoted_cholesky(X, oh, 8)[1])
    n = min(5, len(ores.alphas), info["alpha"].shape[0])
    np.testing.assert_allclose(info["alpha"][:n, 0], ores.alphas[:n], rtol=1e-3)
    np.testing.assert_allclose(info["beta"][:n, 0], ores.betas[:n], rtol=1e-2)
    assert abs(info["iters"] - ores.iters) <= 3
    assert abs(info["gamma0"][0] - ores.gamma0) < 1e-4 * ores.gamma0


def test_cg_edge_cases(ctx):
    from paper_2207_06856_gb300 import gpk
    # N = 1: Ktilde = a^2 + sigma^2, one step solves it
    hyp = gpk.Hyper(0, np.ones(2), 1.5, 0.5)
    X = _dev(np.zeros((1, 2), np.float32))
    B = _dev(np.array([[3.0]], np.float32))
    U, st, info = gpk.cg_solve(ctx, hyp, X, B, None, tol=1e-6, max_iter=5, precision="fp16")
    assert st == gpk.GP_OK
    assert abs(U.item() - 3.0 / 2.0) < 1e-5
    # zero right-hand side: nothing to do, U = 0
    Xn, V, kern, ls, a2, s2 = workloads.random_problem(500, 3, 2, seed=24)
    V[1] = 0.0
    hyp = gpk.Hyper(kern, ls, a2, s2)
    U, st, info = gpk.cg_solve(ctx, hyp, _dev(Xn), _dev(V), None, tol=1e-3, max_iter=100, precision="fp32")
    assert np.all(U.cpu().numpy()[1] == 0.0)
    # max_iter reached -> NOT_CONVERGED, iterate still returned
    U, st, info = gpk.cg_solve(ctx, hyp, _dev(Xn), _dev(V[:1]), None, tol=1e-12, max_iter=2, precision="fp32")
    assert st == gpk.GP_ERR_NOT_CONVERGED and info["iters"] == 2
    # warm start from the solution: converged before the first step
    ref = O.cholesky_solve(Xn, O.Hyp("rbf", ls, a2, s2), V[:1].T.astype(np.float64)).T.astype(np.float32)
    U0 = _dev(ref)
    U, st, info = gpk.cg_solve(ctx, hyp, _dev(Xn), _dev(V[:1]), None, tol=1e-4, max_iter=10, precision="fp32", U=U0)
    assert st == gpk.GP_OK and info["iters"] <= 1
    ctx.check()


STOP_MARGIN = 0.01   # the benchmark's margin under 1e-2 for the FP32 check's rounding


def test_precision_workload_full_size_fp16(ctx):
    """The benchmark solve: N = 65,536, d = 8, RBF, 1 + 16 RHS, rank-100
    preconditioner, FP16 tensor-core MVM, stable CG stopped at 0.99e-2 on its
    FP32 true-residual check.

    The residual ||Ktilde U - B|| / ||B|| is recomputed in FP64 over all
    65,536 rows (the oracle's multi-threaded matrix-free MVM) and must be
    <= 1e-2 for every column: the 1 % margin covers the FP32 check's rounding,
    about 2^-24 kappa / sqrt(N) = 3.4e-6 of ||b|| with kappa = || |K| |x| || /
    ||b|| ~ 1.5e4 (sum_j |k_ij x_j| rather than |(Ktilde x)_i| sets it)."""
    from oracle import cfp64 as C
    from paper_2207_06856_gb300 import gpk
    w = workloads.precision()
    hyp = gpk.Hyper(w.kernel, w.lengthscale, w.outputscale, w.noise)
    X = _dev(w.X)
    pc = gpk.pivchol(ctx, hyp, X, w.rank)
    B = w.rhs()
    U, st, info = gpk.cg_solve(ctx, hyp, X, _dev(B), pc, tol=w.tol * (1.0 - STOP_MARGIN), max_iter=w.max_iter,
                               precision="fp16")
    ctx.check()
    assert st == gpk.GP_OK, (info["col_iters"], info["rel_resid"])
    reported = np.asarray(info["rel_resid"])
    assert reported.max() <= w.tol * (1.0 - STOP_MARGIN), reported
    full = C.relative_residual(w.X, U.cpu().numpy().T, B.T, _ohyp(w))
    assert full.max() <= w.tol, full
    assert np.all(np.abs(full - reported) <= STOP_MARGIN * w.tol), (full, reported)


def test_breakdown_escalates_to_check_precision(ctx):
    """N = 20,000 points in d = 2, RBF l = 0.5, sigma^2 = 1e-4, single-term FP16
    inputs: the FP16 operator is not positive definite to the accuracy the solve
    needs, so CG breaks down; with escalation (the default) the restart continues
    with the FP32 check MVM and the solve converges by that MVM.  At this
    conditioning |x| ~ |y| / sigma^2, and the FP32 check's rounding (proportional
    to sum_j |k_ij x_j|) resolves the residual only to a few 1e-2: the FP64
    residual is checked against 5e-2."""
    from paper_2207_06856_gb300 import gpk
    rng = np.random.default_rng(0)
    N, d = 20000, 2
    X = rng.standard_normal((N, d)).astype(np.float32)
    y = (np.sin(2 * np.pi * X.mean(1)) + 0.1 * rng.standard_normal(N)).astype(np.float32)
    hyp = gpk.Hyper(gpk.RBF, np.full(d, 0.5, np.float32), 1.0, 1e-4)
    Xd, B = _dev(X), _dev(y[None])
    pc = gpk.pivchol(ctx, hyp, Xd, 20)
    _, st0, info0 = gpk.cg_solve(ctx, hyp, Xd, B, pc, tol=1e-2, max_iter=1000, precision="fp16",
                                 flags=gpk.MVM_NO_XSPLIT, escalate=False)
    assert st0 == gpk.GP_ERR_BREAKDOWN and info0["breakdowns"] >= 1
    U, st1, info1 = gpk.cg_solve(ctx, hyp, Xd, B, pc, tol=1e-2, max_iter=1000, precision="fp16",
                                 flags=gpk.MVM_NO_XSPLIT, escalate=True)
    assert st1 == gpk.GP_OK and info1["escalated"] == 1, info1["rel_resid"]
    rows = np.sort(np.random.default_rng(1).choice(N, 2048, replace=False))
    oh = O.Hyp("rbf", np.full(d, 0.5), 1.0, 1e-4)
    r = O.kmvm_rows(X, rows, U.cpu().numpy().T.astype(np.float64), oh)[:, 0] - y[rows]
    est = np.sqrt(N / len(rows) * np.sum(r * r)) / np.linalg.norm(y.astype(np.float64))
    assert est <= 5e-2, est


def test_split_fp16_solve_needs_fp32_iteration_count(ctx):
    """FP16 tensor-core MVM with the kernel tile and inputs carried as hi + lo:
    the stable CG needs at most 15 % more iterations than FP32 on the precision
    workload's distribution (N = 16,384), and its residual is verified in FP64."""
    from paper_2207_06856_gb300 import gpk
    w = workloads.precision(N=16384)
    hyp = gpk.Hyper(w.kernel, w.lengthscale, w.outputscale, w.noise)
    X, B = _dev(w.X), _dev(w.rhs())
    pc = gpk.pivchol(ctx, hyp, X, w.rank)
    _, st32, i32 = gpk.cg_solve(ctx, hyp, X, B, pc, tol=w.tol, max_iter=w.max_iter, precision="fp32")
    U, st16, i16 = gpk.cg_solve(ctx, hyp, X, B, pc, tol=w.tol, max_iter=w.max_iter, precision="fp16",
                                flags=gpk.MVM_PSPLIT | gpk.MVM_XSPLIT)
    assert st32 == gpk.GP_OK and st16 == gpk.GP_OK
    assert i16["iters"] <= 1.15 * i32["iters"], (i16["iters"], i32["iters"])
    rows = np.sort(np.random.default_rng(3).choice(w.N, 2048, replace=False))
    Bt = w.rhs().T.astype(np.float64)
    r = O.kmvm_rows(w.X, rows, U.cpu().numpy().T, _ohyp(w), add_noise=True) - Bt[rows]
    est = np.sqrt(w.N / len(rows) * np.sum(r * r, axis=0)) / np.linalg.norm(Bt, axis=0)
    assert est.max() <= 1.15 * w.tol, est


def test_precision_workload_full_size_relaxed_schedule(ctx):
    """The benchmark's solve with its relaxed MVM schedule: the FP16 MVM with the
    kernel tile and inputs as hi + lo until every column's recursive residual is
    <= 0.3 (30 x tol), the single-rounded FP16 MVM after.  The FP64 residual over
    all 65,536 rows must be <= 1e-2 for every column, and the schedule must need
    fewer iterations than the single-rounded MVM throughout (the accurate early
    MVMs keep the true residual close to the recursive one)."""
    from oracle import cfp64 as C
    from paper_2207_06856_gb300 import gpk
    w = workloads.precision()
    hyp = gpk.Hyper(w.kernel, w.lengthscale, w.outputscale, w.noise)
    X = _dev(w.X)
    pc = gpk.pivchol(ctx, hyp, X, w.rank)
    B = w.rhs()
    tol = w.tol * (1.0 - STOP_MARGIN)
    U, st, info = gpk.cg_solve(ctx, hyp, X, _dev(B), pc, tol=tol, max_iter=w.max_iter,
                               precision=gpk.FP16 | gpk.MVM_PSPLIT | gpk.MVM_XSPLIT, refine_precision="fp16",
                               refine_resid=30.0 * w.tol)
    _, st1, info1 = gpk.cg_solve(ctx, hyp, X, _dev(B), pc, tol=tol, max_iter=w.max_iter, precision="fp16")
    ctx.check()
    assert st == gpk.GP_OK and st1 == gpk.GP_OK
    assert info["iters"] < info1["iters"], (info["iters"], info1["iters"])
    full = C.relative_residual(w.X, U.cpu().numpy().T, B.T, _ohyp(w))
    assert full.max() <= w.tol, full


def test_refine_switch_points(ctx):
    """refine_resid above every residual switches before the first iteration,
    so the solve is bit-identical to one on the refine MVM alone; below every
    residual it never switches (bit-identical to the solve's own MVM); in
    between the trajectory starts like the first and differs later.  Invalid
    switch settings are refused."""
    from paper_2207_06856_gb300 import gpk
    w = workloads.precision(N=6000)
    hyp = gpk.Hyper(w.kernel, w.lengthscale, w.outputscale, w.noise)
    X, B = _dev(w.X), _dev(w.rhs())
    pc = gpk.pivchol(ctx, hyp, X, w.rank)
    split = gpk.FP16 | gpk.MVM_PSPLIT | gpk.MVM_XSPLIT
    kw = dict(tol=w.tol, max_iter=w.max_iter)
    Ua, _, ia = gpk.cg_solve(ctx, hyp, X, B, pc, precision=split, **kw)
    Ub, _, ib = gpk.cg_solve(ctx, hyp, X, B, pc, precision="fp16", **kw)
    Uhi, _, ihi = gpk.cg_solve(ctx, hyp, X, B, pc, precision=split, refine_precision="fp16", refine_resid=1e30, **kw)
    Ulo, _, ilo = gpk.cg_solve(ctx, hyp, X, B, pc, precision=split, refine_precision="fp16", refine_resid=1e-30,
                               **kw)
    Umid, _, imid = gpk.cg_solve(ctx, hyp, X, B, pc, precision=split, refine_precision="fp16", refine_resid=0.3,
                                 **kw)
    assert torch.equal(Uhi, Ub) and np.array_equal(ihi["alpha"], ib["alpha"])
    assert torch.equal(Ulo, Ua) and np.array_equal(ilo["alpha"], ia["alpha"])
    k = int(np.argmax(np.max(ia["resid_hist"], axis=1) <= 0.3))   # first iterate at or below the switch point
    assert k > 1
    assert np.array_equal(imid["alpha"][:k], ia["alpha"][:k])
    assert not np.array_equal(imid["alpha"], ia["alpha"][:len(imid["alpha"])])
    with pytest.raises(gpk.GPKError):
        gpk.cg_solve(ctx, hyp, X, B, pc, precision=split, refine_precision="fp16", refine_resid=-1.0, **kw)
    with pytest.raises(gpk.GPKError):
        gpk.cg_solve(ctx, hyp, X, B, pc, precision=split, refine_precision="fp16", refine_resid=0.0, restarts=0,
                     **kw)


@pytest.mark.parametrize("rank", [1, 31, 32, 33, 64, 100, 128, 129, 159, 160, 257, 300])
def test_core_factor_and_inverse_rank_edges(ctx, rank):
    """The FP64 core at the edges of its kernels (32-wide tiles of L^T L, rows per
    lane of the inverse, the factor in shared and in global memory).  Core: against
    I + L^T L / sigma^2 from the returned L; the sums run in FP32 over 64 rows, so
    each entry errs by at most 64 2^-24 of sum |l_a l_b| (4e-6 with the FP64
    factorisation's error far below).  Inverse: the first CG step
    from x_0 = 0 moves along P^{-1} b, so its direction is compared with the FP64 Woodbury
    apply: FP32 sums of at most 900 terms, 900 2^-24 = 5.4e-5, doubled."""
    from paper_2207_06856_gb300 import gpk
    X, V, kern, ls, a2, s2 = workloads.random_problem(900, 6, 2, seed=rank, kernel=1)
    hyp = gpk.Hyper(kern, ls, a2, s2)
    pc = gpk.pivchol(ctx, hyp, _dev(X), rank)
    assert pc.rank == rank
    L = pc.L.cpu().numpy().astype(np.float64)
    Lc = pc.core.cpu().numpy().T
    assert np.array_equal(np.triu(Lc, 1), np.zeros_like(Lc))
    C, bound = L @ L.T / s2, np.abs(L) @ np.abs(L).T / s2
    assert np.all(np.abs(Lc @ Lc.T - np.eye(rank) - C) <= 4e-6 * bound + 1e-12)
    U, _, _ = gpk.cg_solve(ctx, hyp, _dev(X), _dev(V), pc, tol=1e-4, max_iter=1, precision="fp32", restarts=0)
    ctx.check()
    B = V.astype(np.float64)
    C = np.eye(rank) + C
    Z = (B - (np.linalg.solve(C, L @ B.T).T @ L) / s2) / s2
    U = U.cpu().numpy().astype(np.float64)
    unit = lambda A: A / np.linalg.norm(A, axis=1, keepdims=True)
    assert np.abs(unit(U) - unit(Z)).max() <= 1e-4


# rows at the edges of 1,024 threads (1 to 8 elements each), of a warp, and of the one-launch
# path (8,192 rows; N (rank + 32) = 600,000: rank 41 in, 42 out at N = 8,192)
TAIL_CASES = [(1, 0, 1, "none", 1, "fp32"), (31, 5, 2, "pinv", 1, "fp32"), (33, 20, 3, "euclid", 2, "fp32"),
              (1023, 100, 1, "pinv", 1, "fp32"), (1024, 33, 4, "pinv", 2, "fp32"), (1025, 0, 17, "euclid", 1, "fp32"),
              (2047, 20, 2, "none", 1, "fp32"), (2049, 100, 1, "pinv", 1, "fp32_pv"),
              (2049, 20, 5, "pinv", 1, "hilo"), (4097, 64, 2, "pinv", 1, "hilo"), (8191, 40, 1, "pinv", 1, "fp32"),
              (8192, 41, 2, "pinv", 1, "fp32"), (8192, 42, 1, "pinv", 1, "fp32"), (8193, 20, 2, "pinv", 1, "fp32")]


@pytest.mark.parametrize("N,rank,R,reorth,passes,prec", TAIL_CASES)
def test_one_launch_iteration_edges(ctx, N, rank, R, reorth, passes, prec):
    """Small systems, where one launch follows each MVM: the FP64 residual of a solve
    that reports convergence.  The solver accepts by an FP32 MVM, whose sums of at most
    512 + 32 terms (a column range, then the ranges) err by at most 544 2^-24 of
    |Ktilde| |u|; the bound is tol plus that.  Euclidean re-orthogonalisation with a
    preconditioner (whose residuals are P^{-1}-orthogonal, not orthogonal) uses up its
    four checks here and is then accepted on the recurrence's estimate, on the general
    path too: no FP64 bound follows from that status, and that case only has to end
    as reported (its iterates are compared with the general path's below)."""
    from paper_2207_06856_gb300 import gpk
    X, V, kern, ls, a2, s2 = workloads.random_problem(N, 4, R, seed=N + R, noise=0.1)
    hyp = gpk.Hyper(kern, ls, a2, s2)
    flags = {"fp32": gpk.PRECISIONS["fp32"], "hilo": gpk.FP16 | gpk.MVM_PSPLIT | gpk.MVM_XSPLIT,
             "fp32_pv": gpk.FP16 | gpk.MVM_XSPLIT | gpk.MVM_FP32_PV}[prec]
    pc = gpk.pivchol(ctx, hyp, _dev(X), rank) if rank else None
    U, st, info = gpk.cg_solve(ctx, hyp, _dev(X), _dev(V), pc, tol=1e-3, max_iter=500, precision=flags, reorth=reorth,
                               reorth_passes=passes)
    ctx.check()
    assert st == gpk.GP_OK
    if info["restarts"] == 4:
        assert reorth == "euclid" and rank > 0 and np.all(np.asarray(info["rel_resid"]) <= 1e-3)
        return
    Kt = O.ktilde_dense(X.astype(np.float64), O.Hyp("rbf", ls, a2, s2))
    U = U.cpu().numpy().astype(np.float64).T
    B = V.T.astype(np.float64)
    bnorm = np.linalg.norm(B, axis=0)
    bound = 1e-3 + 544 * 2.0 ** -24 * np.linalg.norm(Kt @ np.abs(U), axis=0) / bnorm   # Ktilde >= 0
    assert np.all(np.linalg.norm(Kt @ U - B, axis=0) / bnorm <= bound)


@pytest.mark.parametrize("alg,reorth,passes", [("stable", "pinv", 1), ("stable", "pinv", 2), ("stable", "euclid", 2),
                                               ("stable", "none", 1), ("standard", "none", 1)])
@pytest.mark.parametrize("precond", [False, True])
def test_one_launch_iteration_matches_general_path(ctx, alg, reorth, passes, precond):
    """8,192 rows (one launch after each MVM) against the same system with one more point
    whose kernel value with every other is exactly 0 and whose right-hand side is 0
    (8,193 rows, the general path; the factor spends one more column on it): in exact
    arithmetic the same iterates.  Six steps in FP32: dots over 8,192 terms summed in
    blocks and the two MVMs differ by some 1e-6, with a factor 100 for the steps."""
    from paper_2207_06856_gb300 import gpk
    X, V, kern, ls, a2, s2 = workloads.random_problem(8192, 4, 2, seed=5, noise=0.1)
    X1 = np.vstack([np.full((1, 4), 1e3, np.float32), X])   # first: also the first pivot
    V1 = np.hstack([np.zeros((2, 1), np.float32), V])
    hyp = gpk.Hyper(kern, ls, a2, s2)
    out = []
    for x, v, k in ((X, V, 20), (X1, V1, 21)):
        pc = gpk.pivchol(ctx, hyp, _dev(x), k) if precond else None
        U, st, info = gpk.cg_solve(ctx, hyp, _dev(x), _dev(v), pc, tol=1e-9, max_iter=6, precision="fp32",
                                   algorithm=alg, reorth=reorth, reorth_passes=passes, restarts=0)
        ctx.check()
        assert st == gpk.GP_ERR_NOT_CONVERGED and info["iters"] == 6
        out.append((U.cpu().numpy()[:, -8192:].astype(np.float64), info["alpha"][:6], info["beta"][:5]))
    for a, b in zip(*out):
        assert np.linalg.norm(a - b) <= 1e-4 * np.linalg.norm(b)


def _padded(pc, rank):
    """The same preconditioner with columns of zeros appended to L (and 1 on the diagonal of the
    core): the same sums with zeros added, and a rank that the one-launch iteration leaves to
    the general path."""
    from paper_2207_06856_gb300 import gpk
    N, k = pc.L.shape[1], pc.rank
    L = torch.zeros((rank, N), dtype=torch.float32, device="cuda:0")
    L[:k] = pc.L
    core = torch.eye(rank, dtype=torch.float64, device="cuda:0")
    core[:k, :k] = pc.core
    return gpk.Precond(L, core, pc.piv, rank)


def _tail_problem(N, R, seed):
    """A slowly converging system (Matern-1/2 in 3 dimensions, noise 1e-3): hundreds of steps."""
    from paper_2207_06856_gb300 import gpk
    r = np.random.default_rng(seed)
    X, V = r.standard_normal((N, 3)).astype(np.float32), r.standard_normal((R, N)).astype(np.float32)
    return gpk.Hyper(2, np.ones(3, np.float32), 1.0, 1e-3), _dev(X), _dev(V)


def _tail_flags(prec):
    from paper_2207_06856_gb300 import gpk
    return {"fp32": gpk.FP32, "fp16": gpk.FP16, "bf16": gpk.BF16, "hilo": gpk.FP16 | gpk.MVM_PSPLIT | gpk.MVM_XSPLIT,
            "fp32_pv": gpk.FP16 | gpk.MVM_XSPLIT | gpk.MVM_FP32_PV}[prec]


# one to four dot chunks of 2,048 rows, and their edges; the last two cross over to the general
# path on the way, at N = 8,000 near 70 bases
TAIL_BITS = [(300, 4, "fp32_pv", 20, "pinv", 1, 12), (700, 1, "fp32", 20, "pinv", 1, 12),
             (2048, 3, "hilo", 31, "pinv", 2, 12), (2049, 1, "fp32_pv", 20, "pinv", 1, 12),
             (2500, 17, "fp16", 1, "euclid", 2, 12), (4096, 5, "bf16", 20, "pinv", 1, 12),
             (5000, 2, "fp32_pv", 33, "none", 1, 12), (8191, 33, "hilo", 7, "pinv", 1, 12),
             (8192, 2, "hilo", 20, "pinv", 1, 40), (8000, 2, "fp32_pv", 20, "pinv", 1, 130),
             (6001, 3, "hilo", 20, "pinv", 2, 100)]


@pytest.mark.parametrize("N,R,prec,rank,reorth,passes,iters", TAIL_BITS)
def test_one_launch_iteration_bit_identical(ctx, N, R, prec, rank, reorth, passes, iters):
    """One launch after each MVM (its own sum of the MVM's partial results, its own FP32 copy of
    the next direction) against the general path on the same system, bit for bit."""
    from paper_2207_06856_gb300 import gpk
    if torch.cuda.get_device_properties(0).multi_processor_count < 128:
        pytest.skip("the Woodbury apply sums other blocks of rows on fewer than 128 SMs")
    hyp, X, V = _tail_problem(N, R, N + R)
    pc = gpk.pivchol_precond(ctx, hyp, X, rank)
    out = []
    for p in (pc, _padded(pc, 512)):
        n0 = ctx.launches
        U, _, info = gpk.cg_solve(ctx, hyp, X, V, p, tol=0.0, min_iter=iters, max_iter=iters, restarts=0, reorth=reorth,
                                  reorth_passes=passes, precision=_tail_flags(prec), escalate=False)
        ctx.check()
        out.append((ctx.launches - n0, U.cpu().numpy(), info["alpha"], info["beta"][:-1], info["resid_hist"]))
    assert out[1][0] - out[0][0] >= 8 * min(iters, 30)   # they did take different paths
    for a, b in zip(out[0][1:], out[1][1:]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("N,R,passes", [(8000, 1, 1), (8000, 17, 1), (6000, 17, 2)])
def test_one_launch_iteration_ends_with_many_bases(ctx, N, R, passes):
    """One CTA per column reads all stored bases: beyond some number of them the general path,
    which spreads that read over the GPU, is the faster one and is taken. Steps are counted by
    their launches, 8 or more fewer on the one-launch path."""
    from paper_2207_06856_gb300 import gpk
    hyp, X, V = _tail_problem(N, R, 3)
    pc = gpk.pivchol_precond(ctx, hyp, X, 20)
    n = []
    for iters in (1, 11, 150, 160):
        n0 = ctx.launches
        gpk.cg_solve(ctx, hyp, X, V, pc, tol=0.0, min_iter=iters, max_iter=iters, restarts=0, reorth_passes=passes,
                     precision=_tail_flags("fp32_pv" if R == 1 else "hilo"), escalate=False)
        ctx.check()
        n.append(ctx.launches - n0)
    assert n[3] - n[2] >= (n[1] - n[0]) + 10 * 8
