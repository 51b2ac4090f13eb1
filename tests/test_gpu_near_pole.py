"""Solves near the pole alpha = 1 / rho, and shifted ones with a small shift: the
kernels that keep residuals take delta from (r, q), which rounding makes wrong there.
The iterations are held to those with delta = (p, q), simulated here in the
precision of the kernels, or to the FP64 form's."""
import numpy as np
import pytest

import wlgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _csr(g):
    import scipy.sparse as sp
    return sp.csr_matrix((np.ones(g.nnz), g.col_idx, g.row_ptr.astype(np.int64)), shape=(g.n, g.n))


def _cg(M, b, tol, dtype):
    """Iterations to |r| <= tol |b| by the recurrences of the kernels, dot
    products in FP64."""
    def dot(u, v):
        return float(np.dot(u.astype(np.float64), v.astype(np.float64)))
    M, r = M.astype(dtype), b.astype(dtype)
    x = np.zeros_like(r)
    g0 = g = dot(r, r)
    p = q = None
    for it in range(1, 2000):
        w = M @ r
        p, q = (r.copy(), w) if p is None else (r + dtype(be) * p, w + dtype(be) * q)
        al = g / dot(p, q)
        x += dtype(al) * p
        r = r - dtype(al) * q
        g, be = dot(r, r), dot(r, r) / g
        if g <= tol * tol * g0:
            break
    return it, x


# Rows beyond what the SMs' shared memory holds: the phase kernels; the FP64 form is
# the reference.
@pytest.mark.parametrize("rel,shift", [(0.5, 2.0), (0.994, 2.0), (0.999, 2.0)])
def test_shifted_solves_near_the_pole(rel, shift):
    from paper_2601_11338_gb300.api import WalkLaplacian
    g = wlgen.erdos_renyi(200003, 8.0, 3)
    U0 = torch.zeros((g.n, 16), dtype=torch.float64, device="cuda")
    U0[torch.arange(16) * 1000 + 7, torch.arange(16)] = 1.0
    U, its = {}, {}
    for prec in ("fp64", "refined"):
        w = WalkLaplacian(g.row_ptr.astype(np.int32), g.col_idx, g.n, variant="allwalk", alpha_rel=rel, prec=prec,
                          tol=1e-10, outer_tol=1e-9, shift=shift)
        w.degrees()
        U[prec] = w.expmv(U0, [1.0])
        its[prec] = w.last.k_cg_iters / w.last.outer_iters
        w.close()
    err = (U["refined"] - U["fp64"]).norm(dim=1) / U["fp64"].norm(dim=1)
    # residuals of 1e-10 over a condition of some 1e4 near the pole
    assert float(err.max()) <= (1e-8 if rel == 0.5 else 1e-6), err.max()
    # FP32 corrections restart the Krylov space for every 5 digits: three times the iterations at the most
    assert its["refined"] <= 3.0 * its["fp64"], its


@pytest.mark.parametrize("rel,shift", [(0.999, 0.1), (0.9999, 2.0)])
def test_shifted_solves_end_very_near_the_pole(rel, shift):
    """M stays positive definite: no solve may meet a non-positive (p, M p)."""
    from paper_2601_11338_gb300.api import WalkLaplacian
    g = wlgen.erdos_renyi(200003, 8.0, 3)
    U0 = torch.zeros((g.n, 16), dtype=torch.float64, device="cuda")
    U0[torch.arange(16) * 1000 + 7, torch.arange(16)] = 1.0
    w = WalkLaplacian(g.row_ptr.astype(np.int32), g.col_idx, g.n, variant="allwalk", alpha_rel=rel, prec="refined",
                      tol=1e-10, outer_tol=1e-8, shift=shift, max_outer=24)
    w.degrees()
    assert bool(torch.isfinite(w.expmv(U0, [1.0])).all())
    w.close()


@pytest.mark.parametrize("rel", [0.5, 0.97, 0.999])
def test_iterations_of_the_batch(rel):
    import scipy.sparse as sp
    from paper_2601_11338_gb300 import wl
    gs = [wlgen.erdos_renyi(20000, 10.0, 2), wlgen.chung_lu(20000)]
    graphs = [(g.row_ptr.astype(np.int32), g.col_idx, g.n, g.nnz) for g in gs]
    p = wl.make_params(f=wl.WL_F_RESOLVENT, alpha_rel=rel, prec=wl.WL_REFINED, tol=1e-10,
                       stream=torch.cuda.current_stream().cuda_stream)
    b = wl.wl_batch_build(graphs, [0.0], p)
    n = sum(g.n for g in gs)
    V = torch.ones((n, 2), dtype=torch.float64, device="cuda")
    D = torch.zeros((1, n), dtype=torch.float64, device="cuda")
    W = torch.zeros((1, n, 2), dtype=torch.float64, device="cuda")
    wl.wl_batch_run(b, V, 2, D, W)
    row = 0
    for i, g in enumerate(gs):
        info = wl.wl_batch_info(b, i, 0)
        M = (sp.eye(g.n) - info["alpha"] * _csr(g)).tocsr()
        r, total, x = np.ones(g.n), 0, np.zeros(g.n)
        while np.linalg.norm(r) > 1e-10 * np.sqrt(g.n):  # every correction to 5e-6
            it, d = _cg(M, r, 5e-6, np.float32)
            total += it
            x += d
            r = 1.0 - M @ x
        assert info["status"] == wl.WL_OK
        assert info["iters_df"] <= 1.1 * total + 2, (i, info["iters_df"], total)
        assert info["iters_v"] <= 1.1 * total + 2, (i, info["iters_v"], total)
        # both residuals are below 1e-10 |b|: D_f differs by at most their sum over 1 - alpha rho
        dd = np.linalg.norm(D[0, row:row + g.n].cpu().numpy() - x)
        assert dd <= 2e-10 / (1 - rel) * np.sqrt(g.n)
        row += g.n
    b.destroy()
