"""Backward of the kernel MVM (gp_kmvm_vjp) and the loss / gradient
(gp_mll_and_grad, Eq. loss / approx) against the FP64 oracle.

Tolerances: the FP32 backward against the FP64 bilinear-form gradient 1e-4
(relative, vector norm); gradients from solves <= 1e-2 relative against the
same-probe FP64 estimator (exact solves); the loss value <= 1e-3 relative
against the same-probe FP64 SLQ estimate."""

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
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to("cuda:0")


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a) - np.asarray(b)) / np.linalg.norm(np.asarray(b)))


@pytest.mark.parametrize("kern", [0, 1, 2, 3])
@pytest.mark.parametrize("shape", [(300, 3, 2), (1000, 8, 17), (777, 18, 5)])
def test_vjp_matches_oracle(ctx, kern, shape):
    from paper_2207_06856_gb300 import gpk
    N, d, R = shape
    X, V, _, ls, a2, s2 = workloads.random_problem(N, d, R, seed=N + d, kernel=kern)
    U = np.random.default_rng(N).standard_normal((R, N)).astype(np.float32)
    hyp = gpk.Hyper(kern, ls, a2, s2)
    g, gX = gpk.kmvm_vjp(ctx, hyp, _dev(X), _dev(U), _dev(V), want_X=True)
    ref, refX = O.quad_form_grad(X, O.Hyp(KNAME[kern], ls, a2, s2), U.T, V.T, wrt_X=True)
    assert _rel(g, ref) <= 1e-4, (g, ref)
    assert _rel(gX.cpu().numpy(), refX) <= 1e-4


def _problem(N=1500, d=5, M=8, seed=3, kernel=0):
    rng = np.random.default_rng(seed)
    X = rng.standard_normal((N, d)).astype(np.float32)
    y = (np.sin(X.sum(axis=1)) + 0.1 * rng.standard_normal(N)).astype(np.float32)
    ls = np.full(d, 1.2, np.float32)
    return X, y, ls, 1.1, 0.05, M, kernel


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-6), ("fp16", 1e-3)])
def test_gradient_matches_same_probe_estimator(ctx, prec, tol):
    """Rademacher probes (E[zz^T] = I), no preconditioner: the library's
    gradient against Eq. approx evaluated in FP64 with exact solves."""
    from paper_2207_06856_gb300 import gpk
    X, y, ls, a2, s2, M, kern = _problem()
    Z = workloads.rademacher(np.random.default_rng(9), M, X.shape[0])
    hyp = gpk.Hyper(kern, ls, a2, s2)
    mll, g, _, U, info = gpk.mll_and_grad(ctx, hyp, _dev(X), _dev(y), _dev(Z), tol=tol, max_iter=500,
                                          precision=prec, want_logdet=True, return_U=True)
    oh = O.Hyp("rbf", ls, a2, s2)
    B = np.column_stack([y, Z.T]).astype(np.float64)
    Uex = O.cholesky_solve(X, oh, B)
    ref = O.pseudo_loss_grad(X, oh, Uex, Z.T.astype(np.float64))
    assert _rel(g, ref) <= 1e-2, (g, ref)
    # the same-probe estimator approximates the exact gradient (Hutchinson variance)
    exact = O.mll_grad_exact(X, y, oh)
    assert _rel(ref, exact) < 0.5


def test_mll_value_with_preconditioner_probes(ctx):
    """P-distributed probes z = L e + sigma z~, SLQ log-determinant plus log|P|:
    the loss against the same-probe FP64 SLQ estimate (1e-3) and the exact
    loss (within the estimator's spread)."""
    from paper_2207_06856_gb300 import gpk
    X, y, ls, a2, s2, M, kern = _problem(N=1200, M=16, seed=4)
    rank = 20
    rng = np.random.default_rng(11)
    Zt = rng.standard_normal((M, X.shape[0])).astype(np.float32)
    E = rng.standard_normal((M, rank)).astype(np.float32)
    hyp = gpk.Hyper(kern, ls, a2, s2)
    Xd = _dev(X)
    pc = gpk.pivchol(ctx, hyp, Xd, rank)
    mll, g, _, U, info = gpk.mll_and_grad(ctx, hyp, Xd, _dev(y), _dev(Zt), precond=pc, E=_dev(E),
                                          precond_probes=True, want_logdet=True, tol=1e-6, max_iter=400,
                                          precision="fp32", return_U=True, restarts=0)
    oh = O.Hyp("rbf", ls, a2, s2)
    # the oracle builds the same probes from the GPU's L (FP32 factor, pivots as chosen)
    L = pc.L.cpu().numpy().astype(np.float64).T
    Zp = (L @ E.T.astype(np.float64) + math.sqrt(s2) * Zt.T.astype(np.float64))   # N x M
    Kt = O.ktilde_dense(X, oh)
    pre = lambda r: O.precond_apply(L, s2, r)  # noqa: E731
    est = []
    for j in range(M):
        res = O.cg_stable(lambda v: Kt @ v, Zp[:, j], precond=pre, tol=1e-10, max_iter=X.shape[0])
        est.append(O.slq_quadrature(O.lanczos_tridiagonal(res.alphas, res.betas), res.gamma0))
    logdet_slq = O.precond_logdet(L, s2) + float(np.mean(est))
    alpha = np.linalg.solve(Kt, y.astype(np.float64))
    ref = 0.5 * logdet_slq + 0.5 * float(y @ alpha) + 0.5 * X.shape[0] * math.log(2 * math.pi)
    assert abs(mll - ref) <= 1e-3 * abs(ref), (mll, ref)
    exact = O.mll_exact(X, y, oh)
    spread = 0.5 * float(np.std(est)) / math.sqrt(M)
    assert abs(mll - exact) <= 5 * spread + 1e-3 * abs(exact), (mll, exact, spread)
    # gradient with P-probes against the same-probe FP64 estimator (u_j paired with P^{-1} z_j)
    B = np.column_stack([y.astype(np.float64), Zp])
    Uex = np.linalg.solve(Kt, B)
    refg = O.pseudo_loss_grad(X, oh, Uex, Zp, W=pre(Zp))
    assert _rel(g, refg) <= 1e-2, (g, refg)


def test_autograd_fit_moves_toward_better_loss(ctx):
    """A few Adam steps of the training loop on a small problem lower the exact loss."""
    from paper_2207_06856_gb300 import autograd, gpk
    X, y, ls, a2, s2, M, kern = _problem(N=1000, d=3, M=8, seed=5)
    oh0 = O.Hyp("rbf", np.full(3, 2.5), 1.0, 0.3)
    hist = autograd.fit(ctx, _dev(X), _dev(y), gpk.RBF, np.full(3, 2.5), 1.0, 0.3, steps=15, lr=0.1, M=8,
                        rank=20, tol=1e-2, max_iter=200, precision="fp16")
    l, a, s = hist[-1][1], hist[-1][2], hist[-1][3]
    assert O.mll_exact(X, y, O.Hyp("rbf", l, a, s)) < O.mll_exact(X, y, oh0)


@pytest.mark.parametrize("name", ["differentiation", "scale"])
def test_workload_distributions_gradient(ctx, name):
    """The differentiation (d = 18, ARD RBF, Gaussian mixture) and scale (d = 11,
    Matern-3/2, anisotropic mixture) workloads' input distributions at a size the
    oracle solves exactly: the FP16 gradient of Eq. approx against the same-probe
    FP64 estimator (1e-2), with solves to 1e-3 (FP32 true-residual restarts)."""
    from paper_2207_06856_gb300 import gpk
    w = getattr(workloads, name)(N=1500)
    X, y = w.X, w.y
    N, d = X.shape
    ls = np.random.default_rng(5).uniform(0.7, 1.5, size=d).astype(np.float32)   # ARD
    M = 8
    Z = workloads.rademacher(np.random.default_rng(13), M, N)
    hyp = gpk.Hyper(w.kernel, ls, w.outputscale, max(w.noise, 0.02))
    mll, g, _, U, info = gpk.mll_and_grad(ctx, hyp, _dev(X), _dev(y), _dev(Z), tol=1e-3, max_iter=600,
                                          precision="fp16", want_logdet=True, return_U=True)
    oh = O.Hyp(KNAME[w.kernel], ls.astype(np.float64), w.outputscale, max(w.noise, 0.02))
    B = np.column_stack([y, Z.T]).astype(np.float64)
    Uex = O.cholesky_solve(X, oh, B)
    ref = O.pseudo_loss_grad(X, oh, Uex, Z.T.astype(np.float64))
    assert _rel(g, ref) <= 1e-2, (g, ref)


def test_mll_fp16_differentiation_inputs_n16384(ctx):
    """The differentiation inputs (d = 18, ARD RBF, 8-component Gaussian
    mixture, random-feature targets) at N = 16,384, where the dense FP64
    oracle fits: the FP16 loss of gp_mll_and_grad (P-distributed probes,
    rank-100 preconditioner, SLQ log-determinant, solves to 1e-3) within 1e-3
    of the same-probe FP64 estimate, and its gradient within 1e-2 of the
    same-probe FP64 estimator (Eq. approx) with converged FP64 solves."""
    from oracle import cfp64 as C
    from paper_2207_06856_gb300 import gpk
    w = workloads.differentiation(N=16384)
    X, y = w.X, w.y
    N, d = X.shape
    M, rank = 16, 100
    rng = np.random.default_rng(17)
    Zt = rng.standard_normal((M, N)).astype(np.float32)
    E = rng.standard_normal((M, rank)).astype(np.float32)
    hyp = gpk.Hyper(w.kernel, w.lengthscale, w.outputscale, w.noise)
    Xd = _dev(X)
    pc = gpk.pivchol(ctx, hyp, Xd, rank)
    mll, g, _, U, info = gpk.mll_and_grad(ctx, hyp, Xd, _dev(y), _dev(Zt), precond=pc, E=_dev(E),
                                          precond_probes=True, want_logdet=True, tol=1e-3, max_iter=1000,
                                          precision="fp16", return_U=True)
    ctx.check()
    oh = O.Hyp("rbf", w.lengthscale.astype(np.float64), w.outputscale, w.noise)
    L = pc.L.cpu().numpy().astype(np.float64).T                                  # the GPU's factor
    s2 = w.noise
    Zp = L @ E.T.astype(np.float64) + math.sqrt(s2) * Zt.T.astype(np.float64)   # N x M, E[zz^T] = P
    pre = lambda r: O.precond_apply(L, s2, r)  # noqa: E731
    Kt = O.ktilde_dense(X, oh)
    res = O.cg_mbcg(lambda V: Kt @ V, np.column_stack([y.astype(np.float64), Zp]), precond=pre, tol=1e-9,
                    max_iter=3000)
    del Kt
    est = [O.slq_quadrature(O.lanczos_tridiagonal(r.alphas, r.betas), r.gamma0) for r in res[1:]]
    logdet = O.precond_logdet(L, s2) + float(np.mean(est))
    ref = 0.5 * logdet + 0.5 * float(y.astype(np.float64) @ res[0].x) + 0.5 * N * math.log(2 * math.pi)
    assert abs(mll - ref) <= 1e-3 * abs(ref), (mll, ref)
    Uex = np.column_stack([r.x for r in res])
    refg = C.pseudo_loss_grad(X, oh, Uex, Zp, W=pre(Zp))
    assert _rel(g, refg) <= 1e-2, (g, refg)


def test_mll_loss_depth_is_decoupled_from_tolerance(ctx):
    """At the training tolerance (1.0, iteration floor 10) the solve stops after
    10 iterations, too few Lanczos steps for the loss value; with
    GP_MLL_SLQ_MIN_ITER(n) every column runs n iterations and the loss agrees
    with the loss of converged solves (tol 1e-4) to 1e-3."""
    from paper_2207_06856_gb300 import gpk
    w = workloads.differentiation(N=4000)
    N = w.X.shape[0]
    M, rank = 16, 100
    rng = np.random.default_rng(19)
    Zt = _dev(rng.standard_normal((M, N)))
    E = _dev(rng.standard_normal((M, rank)))
    hyp = gpk.Hyper(w.kernel, w.lengthscale, w.outputscale, w.noise)
    Xd, yd = _dev(w.X), _dev(w.y)
    pc = gpk.pivchol(ctx, hyp, Xd, rank)
    kw = dict(precond=pc, E=E, precond_probes=True, want_logdet=True, max_iter=400, precision="fp32")
    conv, *_ = gpk.mll_and_grad(ctx, hyp, Xd, yd, Zt, tol=1e-4, **kw)
    loose, _, _, _, i_loose = gpk.mll_and_grad(ctx, hyp, Xd, yd, Zt, tol=1.0, min_iter=10, **kw)
    deep, _, _, _, i_deep = gpk.mll_and_grad(ctx, hyp, Xd, yd, Zt, tol=1.0, min_iter=10, loss_depth=200, **kw)
    ctx.check()
    assert np.all(i_deep["col_iters"] >= 200) and np.max(i_loose["col_iters"]) < 200
    assert abs(deep - conv) <= 1e-3 * abs(conv), (deep, conv, loose)


def test_kmvm_differentiation_workload_sampled_rows(ctx):
    """The differentiation workload's MVM (N = 262,144, d = 18, ARD RBF, FP16
    with the inputs carried as hi + lo): 64 sampled rows against exact FP64 rows."""
    from oracle import cfp64 as C
    from paper_2207_06856_gb300 import gpk
    w = workloads.differentiation()
    dev = torch.device("cuda:0")
    V = np.random.default_rng(21).standard_normal((5, w.X.shape[0])).astype(np.float32)
    hyp = gpk.Hyper(w.kernel, w.lengthscale, w.outputscale, w.noise)
    out = gpk.kmvm(ctx, hyp, torch.from_numpy(w.X).to(dev), torch.from_numpy(V).to(dev), precision="fp16",
                   add_noise=True)
    ctx.check()
    rows = np.sort(np.random.default_rng(22).choice(w.X.shape[0], 64, replace=False))
    got = out[:, torch.from_numpy(rows).to(dev)].cpu().numpy().astype(np.float64)
    oh = O.Hyp("rbf", w.lengthscale.astype(np.float64), w.outputscale, w.noise)
    ref = C.kmvm(w.X, V.T.astype(np.float64), oh, rows=rows).T
    err = np.max(np.linalg.norm(got - ref, axis=1) / np.linalg.norm(ref, axis=1))
    assert err <= 2e-3, err


VJP_TC_SHAPES = [(300, 3, 2), (1000, 8, 17), (777, 18, 5), (4097, 8, 17), (2000, 12, 32), (129, 20, 1)]


@pytest.mark.parametrize("kern", [0, 1, 3])
@pytest.mark.parametrize("shape", VJP_TC_SHAPES)
def test_vjp_tensor_core_matches_oracle(ctx, kern, shape):
    """The tensor-core backward (FP16 S, H = [u|w][w|u]^T and W' = a^2 k' H,
    FP32 accumulation) against the FP64 bilinear-form gradient: <= 1e-2
    relative, the gradient tolerance, for the hyperparameters and for X."""
    from paper_2207_06856_gb300 import gpk
    N, d, R = shape
    X, V, _, ls, a2, s2 = workloads.random_problem(N, d, R, seed=N + 7 * d, kernel=kern)
    U = np.random.default_rng(N + 1).standard_normal((R, N)).astype(np.float32)
    hyp = gpk.Hyper(kern, ls, a2, s2)
    g, gX = gpk.kmvm_vjp(ctx, hyp, _dev(X), _dev(U), _dev(V), want_X=True, precision="fp16")
    ctx.check()
    ref, refX = O.quad_form_grad(X, O.Hyp(KNAME[kern], ls, a2, s2), U.T, V.T, wrt_X=True)
    assert _rel(g, ref) <= 1e-2, (g, ref)
    assert _rel(gX.cpu().numpy(), refX) <= 1e-2


def test_vjp_tensor_core_refuses_matern12(ctx):
    from paper_2207_06856_gb300 import gpk
    X, V, _, ls, a2, s2 = workloads.random_problem(300, 3, 2, seed=3, kernel=2)
    with pytest.raises(gpk.GPKError):
        gpk.kmvm_vjp(ctx, gpk.Hyper(2, ls, a2, s2), _dev(X), _dev(V), _dev(V), precision="fp16")


def test_vjp_tensor_core_differentiation_inputs_n16384(ctx):
    """The differentiation inputs (d = 18: inputs as hi + lo, k_pad 64) at
    N = 16,384 with the 17 columns of the pseudo-loss: against the oracle's
    matrix-free FP64 gradient, hyperparameters and X."""
    from oracle import cfp64 as C
    from paper_2207_06856_gb300 import gpk
    w = workloads.differentiation(N=16384)
    N = w.X.shape[0]
    rng = np.random.default_rng(23)
    U = rng.standard_normal((17, N)).astype(np.float32)
    V = rng.standard_normal((17, N)).astype(np.float32)
    hyp = gpk.Hyper(w.kernel, w.lengthscale, w.outputscale, w.noise)
    g, gX = gpk.kmvm_vjp(ctx, hyp, _dev(w.X), _dev(U), _dev(V), want_X=True, precision="fp16")
    ctx.check()
    oh = O.Hyp("rbf", w.lengthscale.astype(np.float64), w.outputscale, w.noise)
    ref, refX = C.quad_form_grad(w.X, oh, U.T, V.T, wrt_X=True)
    assert _rel(g, ref) <= 1e-2, (g, ref)
    assert _rel(gX.cpu().numpy(), refX) <= 1e-2


@pytest.mark.parametrize("kern", [0, 3])
@pytest.mark.parametrize("shape", [(2, 1, 1), (127, 7, 2), (128, 8, 16), (129, 15, 17), (257, 16, 16), (255, 20, 31)])
def test_vjp_tensor_core_tile_edges(ctx, kern, shape):
    """Rows at the edges of the 128-row tiles and 64-column slots, 2 (d + 1) output columns
    at the edges of their groups of 16, right-hand sides at the edges of 16.  Operands and
    W' rounded to FP16 (2^-11 each, four roundings): <= 1e-2 relative in the vector norm,
    as for the other shapes."""
    from paper_2207_06856_gb300 import gpk
    N, d, R = shape
    X, V, _, ls, a2, s2 = workloads.random_problem(N, d, R, seed=N + 7 * d, kernel=kern)
    U = np.random.default_rng(N + 1).standard_normal((R, N)).astype(np.float32)
    hyp = gpk.Hyper(kern, ls, a2, s2)
    g, gX = gpk.kmvm_vjp(ctx, hyp, _dev(X), _dev(U), _dev(V), want_X=True, precision="fp16")
    ctx.check()
    ref, refX = O.quad_form_grad(X, O.Hyp(KNAME[kern], ls, a2, s2), U.T, V.T, wrt_X=True)
    assert _rel(g, ref) <= 1e-2, (g, ref)
    assert _rel(gX.cpu().numpy(), refX) <= 1e-2
