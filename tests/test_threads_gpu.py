"""Calls from several threads, each with its own context and stream."""

import ctypes
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _calls(gpk, what, size):
    """The C call alone (prepared once, so that the threads spend their time in the library)."""
    P = ctypes.POINTER
    ctx = gpk.Context(0, 64 << 20)
    s = torch.cuda.Stream()
    g = torch.Generator(device="cuda").manual_seed(size)
    N, d = 256, {"mvm": 18 if size % 2 else 4, "one_tile": 18 if size % 2 else 4, "vjp": 20 if size % 2 else 2}.get(what, 4)
    X = torch.randn((N, d), generator=g, device="cuda")
    V = torch.randn((17, N), generator=g, device="cuda")
    hyp = gpk.Hyper("matern32", np.full(d, 0.4, np.float32), 1.0, 0.1)
    h, st, lib, out = hyp.c(), int(s.cuda_stream), gpk.lib(), torch.empty_like(V)
    keep = [ctx, s, X, V, hyp, h, out]
    if what in ("mvm", "one_tile"):
        fl = gpk.FP16 | (gpk.MVM_ONE_TILE if what == "one_tile" else 0)
        args = (ctx.ptr, ctypes.byref(h), X.data_ptr(), N, X.data_ptr(), N, V.data_ptr(), 17, out.data_ptr(), fl, st)
        return keep, lambda: lib.gp_kmvm(*args)
    if what == "vjp":
        gpk.kmvm_vjp(ctx, hyp, X, V, V, precision="fp16")   # sizes the workspace, declares the call
        gt = np.zeros(d + 2, np.float64)
        args = (ctx.ptr, ctypes.byref(h), X.data_ptr(), N, V.data_ptr(), V.data_ptr(), 17, gpk.FP16,
                gt.ctypes.data_as(P(ctypes.c_double)), None, st)
        return keep + [gt], lambda: lib.gp_kmvm_vjp_prec(*args)
    rank = 80 + 8 * size
    pc = gpk.pivchol_precond(ctx, hyp, X, rank)
    assert pc.rank == rank
    if what == "factor":
        rk = ctypes.c_int(0)
        args = (ctx.ptr, ctypes.byref(h), X.data_ptr(), N, rank, pc.L.data_ptr(), pc.piv.data_ptr(), pc.core.data_ptr(),
                ctypes.byref(rk), st)
        return keep + [pc, rk], lambda: lib.gp_pivchol_precond(*args)
    o = gpk._CgOpts(1e-8, 1, 0, gpk.FP32, 0, 0, 1, 0, 0, gpk.FP32, 0, 0, 0.0)
    stats, c = gpk._CgStats(), pc.c()
    ctx.reserve(64 << 20)
    args = (ctx.ptr, ctypes.byref(h), X.data_ptr(), N, V.data_ptr(), 1, out.data_ptr(), ctypes.byref(c), ctypes.byref(o),
            ctypes.byref(stats), st)
    return keep + [pc, o, stats, c], lambda: lib.gp_cg_solve(*args)


@pytest.mark.parametrize("what,calls", [("mvm", 2000), ("one_tile", 2000), ("vjp", 500), ("factor", 60), ("solve", 1000)])
def test_launches_of_one_kernel_with_different_shared_memory(what, calls):
    """A kernel's shared-memory limit is state of the function: threads that launch it with more
    and with less (other dimensions, other ranks) do not refuse each other's launches."""
    from paper_2207_06856_gb300 import gpk
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    work = [_calls(gpk, what, i) for i in range(6)]
    torch.cuda.synchronize()
    bad = [0] * len(work)

    def go(i):
        for _ in range(calls):
            if work[i][1]() not in (gpk.GP_OK, gpk.GP_ERR_NOT_CONVERGED):
                bad[i] += 1
        work[i][0][1].synchronize()

    threads = [threading.Thread(target=go, args=(i,)) for i in range(len(work))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for w in work:
        w[0][0].check()
    assert bad == [0] * len(work)
