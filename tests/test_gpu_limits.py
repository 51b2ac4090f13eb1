"""Calls at the limits of the number formats and of memory, against the oracle at
the tolerance of the quantity's own parity test."""
import numpy as np
import pytest

import wlgen
from oracle import graph, walks

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def WL(g, **kw):
    from paper_2601_11338_gb300.api import WalkLaplacian
    return WalkLaplacian(g.row_ptr.astype(np.int32), g.col_idx, g.n, **kw)


@pytest.mark.parametrize("shift", [0.0, 1.0])
@pytest.mark.parametrize("prec,tol,bound", [("fp64", 1e-13, 1e-9), ("refined", 1e-12, 1e-8)])
def test_diffusion_does_not_depend_on_the_scale_of_its_columns(prec, tol, bound, shift):
    """exp(-tau L) is linear and the basis is normalised in FP64: columns whose
    norms FP32 cannot hold come out like any other, each to its own scale."""
    g = wlgen.erdos_renyi(400, 6.0, 9)
    A = graph.dense_adjacency(g.row_ptr, g.col_idx, g.n)
    w = WL(g, variant="nbt", alpha_rel=0.5, prec=prec, tol=tol, outer_tol=1e-11, shift=shift)
    lam, Q = np.linalg.eigh(walks.walk_laplacian(walks.phi_resolvent_closed(A, 1.0, w.info["alpha"])))
    U = np.random.default_rng(3).standard_normal((g.n, 6))
    scale = np.array([1e-60, 1e-44, 1e-35, 1.0, 1e37, 1e60])
    taus = [0.0, 0.3, 2.0]
    got = w.expmv(torch.as_tensor(U * scale, device="cuda"), taus).cpu().numpy().reshape(3, g.n, 6) / scale
    for t, tau in enumerate(taus):
        want = Q @ (np.exp(-tau * lam)[:, None] * (Q.T @ U))
        err = np.linalg.norm(got[t] - want, axis=0) / np.linalg.norm(want, axis=0)
        assert (err <= bound).all(), (tau, err)
    w.close()


@pytest.mark.parametrize("prec", ["fp64", "refined"])
@pytest.mark.parametrize("f", ["resolvent", "identity", "exp"])
def test_statistics_count_the_columns_of_the_caller(prec, f):
    """nnz_rhs_iters sums nnz times columns over the operator's applications, and
    bytes_alg the bytes of these columns, also where a block of 13 is worked on as 16."""
    g = wlgen.erdos_renyi(2000, 8.0, 5)
    kw = dict(alpha_rel=0.5) if f == "resolvent" else {}
    w = WL(g, variant="nbt", f=f, prec=prec, tol=1e-10, **kw)
    w.degrees()
    v = torch.as_tensor(np.random.default_rng(1).standard_normal((g.n, 1)), device="cuda")
    calls = [lambda V: w.apply(V)]
    if f != "exp":
        calls.append(lambda V: w.expmv(V, [0.2]))
    if f != "exp":
        calls.append(lambda V: w.markov(V.abs(), [1, 3]))
    for call in calls:
        times = {}
        for k in (16, 13, 1):
            call(v.repeat(1, k).contiguous())
            times[k] = w.last.nnz_rhs_iters / (g.nnz * k)  # applications to one column
            assert times[k] == round(times[k]) > 0, (k, w.last.nnz_rhs_iters)
            if f == "resolvent":
                per = 4.0 * g.nnz + 4.0 * (g.n + 1) + 6.0 * g.n * k * (8 if prec == "fp64" else 4)
                assert w.last.bytes_alg == w.last.k_cg_iters * per
        # equal columns: the same work each, up to a step of the stopping rule in every solve
        assert abs(times[13] - times[16]) <= 0.1 * times[16], times
    w.close()


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_an_overflowing_gradient_is_infinite(sign):
    """One tile whose gradient of b3 and W3 passes FP32's range (6e38 and 4.6e38):
    infinities, as plain FP32 sums give them, and no NaN. W3 = 0 keeps the other
    gradients at zero."""
    from paper_2601_11338_gb300 import wl
    p = np.zeros(4553, dtype=np.float32)
    p[4:8] = 1.0
    p[4424:4488] = 1.0  # b2: h2 = tanh(1)
    F = np.random.default_rng(2).normal(size=(128, 4)).astype(np.float32)
    T = np.full(128, -3e38 * sign, dtype=np.float32)
    grad = np.zeros(4553, dtype=np.float32)
    loss = wl.wl_mlp_loss_grad(p, F, T, 128, grad)
    assert loss == np.inf
    assert (grad[4488:] == sign * np.inf).all(), grad[4488:]
    assert not grad[:4488].any()


# Rows beyond the SMs' shared memory for 16 columns: the phase kernels
def _large(prec):
    g = wlgen.erdos_renyi(200003, 6.0, 3)
    return g, WL(g, variant="nbt", alpha_rel=0.5, prec=prec, tol=1e-10)


def _free():
    from paper_2601_11338_gb300 import wl
    import gc
    gc.collect()
    wl.wl_pool_release()
    return wl.wl_selftest_pool_live()


@pytest.mark.parametrize("prec", ["fp64", "refined"])
def test_a_solve_needs_no_kept_residuals(monkeypatch, prec):
    """With room for the vectors of conjugate gradients in place and no more, an
    apply gives the result that it gives with all the memory."""
    from paper_2601_11338_gb300 import wl
    k, MB = 16, 1 << 20
    g, w = _large(prec)
    V = torch.as_tensor(np.random.default_rng(5).standard_normal((g.n, k)), device="cuda")
    want = w.apply(V)
    w.close()
    _free()
    g, w = _large(prec)
    w.degrees()
    # V, X, b in FP64; then r, p, q (FP64), or b, x, r as two terms each, d, r, p, q (FP32); lists of long rows
    # and 2 MB to round each of some twenty blocks up
    need = (3 + 3) * 8 * g.n * k if prec == "fp64" else (3 * 8 + 10 * 4) * g.n * k
    monkeypatch.setenv("WL_FAULT", f"budget:{wl.wl_selftest_pool_live() + need + 40 * g.n + 28 * MB}")
    got = w.apply(V)
    monkeypatch.delenv("WL_FAULT")
    assert float((got - want).abs().max()) <= 1e-8 * float(want.abs().max())
    w.close()


@pytest.mark.parametrize("prec", ["fp64", "refined"])
def test_kept_residuals_are_given_back(monkeypatch, prec):
    """An outer basis that fits only where the residuals of an earlier apply stood."""
    from paper_2601_11338_gb300 import wl
    k, MB = 16, 1 << 20
    _free()
    g, w = _large(prec)
    V = torch.as_tensor(np.random.default_rng(6).standard_normal((g.n, k)), device="cuda")
    w.set(max_outer=12)
    want = w.expmv(V, [0.05], allow=(wl.WL_ERR_NO_CONVERGENCE,))
    w.close()
    _free()
    g, w = _large(prec)
    w.set(max_outer=12)
    w.apply(V)
    hist = 17 * (8 if prec == "fp64" else 4) * g.n * k
    basis = 13 * 8 * g.n * k
    # the basis, D_f as two terms, the coefficients; half of the residuals stay out
    monkeypatch.setenv("WL_FAULT", f"budget:{wl.wl_selftest_pool_live() + basis + 16 * g.n + 40 * MB - hist // 2}")
    got = w.expmv(V, [0.05], allow=(wl.WL_ERR_NO_CONVERGENCE,))
    monkeypatch.delenv("WL_FAULT")
    assert float((got - want).abs().max()) <= 1e-8 * float(want.abs().max())
    w.close()


@pytest.mark.parametrize("prec", ["fp64", "refined"])
def test_a_padded_block_that_does_not_fit_is_done_unpadded(monkeypatch, prec):
    """13 columns are worked on as 16 where there is room for the basis of 16, and
    as 8, 4 and 1 where there is not."""
    from paper_2601_11338_gb300 import wl
    k, MB = 13, 1 << 20
    g = wlgen.erdos_renyi(20011, 12.0, 3)
    assert wl.wl_selftest_column_blocks(k, g.n, g.nnz, prec == "fp64") == [(16, 13)]

    def make():
        _free()
        w = WL(g, variant="nbt", alpha_rel=0.5, prec=prec, tol=1e-11, outer_tol=1e-9, max_outer=150)
        w.degrees()
        return w
    U = torch.as_tensor(np.random.default_rng(7).standard_normal((g.n, k)), device="cuda")
    w = make()
    want, W = w.expmv(U, [0.4]), w.apply(U)
    w.close()
    w = make()
    basis = 151 * 8 * 8 * g.n  # of eight columns: 194 MB, of 16: 387 MB; some 20 vectors of 16 columns beside it
    monkeypatch.setenv("WL_FAULT", f"budget:{wl.wl_selftest_pool_live() + basis + 20 * 8 * 16 * g.n + 40 * MB}")
    got = w.expmv(U, [0.4])
    work = w.last.nnz_rhs_iters
    got_apply = w.apply(U)
    monkeypatch.delenv("WL_FAULT")
    assert work % g.nnz == 0
    assert float((got - want).abs().max()) <= 1e-8 * float(want.abs().max())
    assert float((got_apply - W).abs().max()) <= 1e-8 * float(W.abs().max())
    w.close()
