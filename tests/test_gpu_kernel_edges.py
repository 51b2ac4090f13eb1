"""Kernels at the sizes where their work split changes: tile edges, remainders,
and the smallest and largest members of each range. Every result is compared
with the oracle, or with a closed form where the graph has one, at the
tolerance of the quantity's own parity test."""
import numpy as np
import pytest

import wlgen
from oracle import features, graph, mlp, philox, walks, xnys

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def WL(g, **kw):
    from paper_2601_11338_gb300.api import WalkLaplacian
    return WalkLaplacian(g.row_ptr.astype(np.int32), g.col_idx, g.n, **kw)


# FP64 Gram: 4 x 4 tiles (M = 3, 4, 5), many copies of the tile set in a CTA
# (M = 2), the last M with two copies and the first with one (M = 48, 52), all
# tiles (M = 64); row counts below, at and above a 32-row stage
@pytest.mark.parametrize("M,n", [(2, 97), (3, 97), (4, 128), (5, 97), (31, 300), (48, 700), (52, 704), (61, 700),
                                 (64, 801)])
def test_trace_fp64_gram_tiles(M, n):
    g = wlgen.erdos_renyi(n, 8, 4)
    w = WL(g, variant="nbt", alpha_rel=0.5, tol=1e-13, prec="fp64")
    A = graph.dense_adjacency(g.row_ptr, g.col_idx, g.n)
    phi = walks.phi_resolvent_closed(A, 1.0, w.info["alpha"])
    est, err = w.trace(M, 900 + M)
    Om, _ = philox.gaussian_sketch(g.n, M, 900 + M)
    e_o, r_o, _ = xnys.xnystrace(phi, Om)
    assert abs(est - e_o) <= 1e-10 * abs(e_o), (est, e_o)
    assert abs(err - r_o) <= 1e-6 * r_o, (err, r_o)
    w.close()
# Triangles: lists for one warp (up to 128 higher-ranked neighbours), for a CTA
# (more), in pieces of 1024, and rows read by a whole CTA (more than 512 entries)
@pytest.mark.parametrize("reorder", [0, 1, 2])
@pytest.mark.parametrize("n", [3, 129, 130, 514, 1026, 1300])
def test_triangles_of_complete_graphs(n, reorder):
    from paper_2601_11338_gb300.api import mlp_features
    g = wlgen.complete(n)
    w = WL(g, variant="nbt", alpha=0.2 / n, reorder=reorder)
    F, _ = mlp_features(w)
    t = (n - 1) * (n - 2) // 2
    want = np.log1p([n - 1.0, (n - 1.0) ** 2, float(t), (n - 1.0) * (n - 2.0)])
    # log1p in FP64 rounded to FP32: half a unit in the last place
    assert np.abs(F.cpu().numpy() / want - 1.0).max() <= 1.2e-7
    w.close()


@pytest.mark.parametrize("seed", [1, 2])
def test_triangles_of_a_skewed_graph(seed):
    """R-MAT scale 11: hubs beyond 512 entries beside nodes of degree 0 and 1."""
    from paper_2601_11338_gb300.api import mlp_features
    g = wlgen.rmat(11, 24, seed=seed)
    w = WL(g, variant="nbt", alpha_rel=0.5)
    F, _ = mlp_features(w)
    tri = features.triangles_by_intersection(g.row_ptr, g.col_idx, g.n)
    assert np.abs(F[:, 2].cpu().numpy().astype(np.float64) - np.log1p(tri)).max() <= 1.2e-7 * np.log1p(tri.max())
    w.close()


# Network: tiles of 128 rows, one tile a CTA up to 304 tiles, then several
@pytest.mark.parametrize("rows", [1, 127, 128, 129, 304 * 128, 304 * 128 + 1, 3 * 304 * 128 + 77])
def test_network_gradient_and_prediction_tiles(rows):
    from paper_2601_11338_gb300 import wl
    rng = np.random.default_rng(rows)
    p = mlp.init_params(64, 4, seed=5)
    for k in ("b1", "b2", "b3"):
        p[k] = 0.1 * rng.standard_normal(p[k].shape)
    v = np.concatenate([rng.normal(size=4), rng.uniform(0.5, 2, 4)] +
                       [p[k].ravel() for k in ("W1", "b1", "W2", "b2", "W3", "b3")]).astype(np.float32)
    F = rng.normal(size=(rows, 4)).astype(np.float32)
    T = rng.normal(size=rows).astype(np.float32)
    xan = rng.uniform(1, 2, rows)
    w = v.astype(np.float64)
    X = (F.astype(np.float64) - w[0:4]) / w[4:8]
    q = {"W1": w[8:264].reshape(64, 4), "b1": w[264:328], "W2": w[328:4424].reshape(64, 64), "b2": w[4424:4488],
         "W3": w[4488:4552].reshape(1, 64), "b3": w[4552:]}
    g = mlp.backward(q, X, T.astype(np.float64))
    want = np.concatenate([g[k].ravel() for k in ("W1", "b1", "W2", "b2", "W3", "b3")])
    grad = np.zeros(v.size, dtype=np.float32)
    loss = wl.wl_mlp_loss_grad(v, F, T, rows, grad)
    assert np.linalg.norm(grad[8:] - want) <= 1e-5 * np.linalg.norm(want)
    assert not grad[:8].any()
    y, _ = mlp.forward(q, X)
    assert abs(loss - np.mean((y - T) ** 2)) <= 1e-5 * np.mean((y - T) ** 2)
    out = torch.full((rows,), float("nan"), dtype=torch.float64, device="cuda")
    wl.wl_mlp_predict(torch.as_tensor(v).cuda(), torch.as_tensor(F).cuda(), rows, torch.as_tensor(xan).cuda(), out)
    assert np.abs(out.cpu().numpy() / (xan * np.exp(y)) - 1.0).max() <= 1e-5


# Cooperative CG: one row, rows below and above a pass of the CTAs, K on both
# sides of every lane width, long hub rows (a whole CTA), hub and mid rows (a
# warp), against the oracle's dense phi at the form's parity tolerance
def _solve_graphs():
    yield wlgen.path(2)
    yield wlgen.erdos_renyi(257, 6.0, 7)
    yield wlgen.star(2500)                      # one hub of 2500 entries
    yield wlgen.barabasi_albert(1500, 20, 3)    # mid and hub rows
    yield wlgen.erdos_renyi(1900, 90.0, 5)      # only mid rows


@pytest.mark.parametrize("reorder", [0, 1])
@pytest.mark.parametrize("prec,tol,bound", [("fp64", 1e-13, 1e-10), ("refined", 1e-12, 1e-8)])
def test_small_solves(prec, tol, bound, reorder):
    for g in _solve_graphs():
        A = graph.dense_adjacency(g.row_ptr, g.col_idx, g.n)
        w = WL(g, variant="btdw", mu=0.4, alpha_rel=0.5, prec=prec, tol=tol, reorder=reorder)
        phi = walks.phi_resolvent_closed(A, 0.4, w.info["alpha"])
        D = walks.walk_degrees(phi)
        L = walks.walk_laplacian(phi)
        Df = w.degrees().cpu().numpy()
        assert np.abs(Df - D).max() <= bound * np.abs(D).max(), g.name
        for k in (1, 2, 3, 4, 8, 16, 32, 64):
            V = np.random.default_rng(k).standard_normal((g.n, k))
            V[:, k // 2] = 0.0 if k > 1 else V[:, 0]  # a zero column takes no part
            W = w.apply(torch.as_tensor(V, device="cuda")).cpu().numpy()
            want = L @ V
            assert np.abs(W - want).max() <= bound * np.abs(want).max(), (g.name, k)
        # a warm start away from the solution
        x0 = D * (1.0 + 0.3 * np.cos(np.arange(g.n)))
        w.warm_start(torch.as_tensor(x0, device="cuda"))
        Df = w.degrees().cpu().numpy()
        assert np.abs(Df - D).max() <= bound * np.abs(D).max(), g.name
        w.close()


def test_fp64_neighbour_sums_of_uneven_magnitude():
    """FP64 solve of a graph too large for the cooperative kernel (the phase
    kernels' integer-aligned neighbour sums): right-hand sides whose entries
    spread over 18 decades with mixed signs, and rows of 0 to 200 entries,
    against scipy's FP64 CG."""
    from oracle import krylov
    e = wlgen.erdos_renyi(70001, 8.0, 3)
    src = np.repeat(np.arange(e.n), e.degrees)
    hub = np.arange(5, 70001, 350)  # node 3 joins 200 others
    g = wlgen.csr_from_edges(e.n, np.concatenate([src, np.full(hub.size, 3)]), np.concatenate([e.col_idx, hub]))
    w = WL(g, variant="nbt", alpha_rel=0.5, prec="fp64", tol=1e-13)
    L = krylov.ResolventLaplacian(krylov.adjacency(g.row_ptr, g.col_idx, g.n), 1.0, w.info["alpha"], tol=1e-14)
    rng = np.random.default_rng(11)
    V = rng.standard_normal((g.n, 16)) * 10.0 ** rng.uniform(-9, 9, (g.n, 1))
    V[:, 3] = 0.0
    V[:, 4] *= 1e-120
    W = w.apply(torch.as_tensor(V, device="cuda")).cpu().numpy()
    want = L.apply(V)
    scale = np.abs(want).max(0)
    assert (np.abs(W - want).max(0) <= 1e-10 * scale).all()
    w.close()


# Column counts that end in a padded block, and leading dimensions beyond k:
# the columns after the block's own keep what the caller has there
@pytest.mark.parametrize("prec,tol,bound", [("fp64", 1e-13, 1e-10), ("refined", 1e-12, 1e-8)])
@pytest.mark.parametrize("reorder", [0, 1])
def test_padded_column_blocks(prec, tol, bound, reorder):
    from paper_2601_11338_gb300 import wl
    g = wlgen.erdos_renyi(411, 7.0, 9)
    A = graph.dense_adjacency(g.row_ptr, g.col_idx, g.n)
    w = WL(g, variant="nbt", alpha_rel=0.5, prec=prec, tol=tol, outer_tol=tol, reorder=reorder)
    phi = walks.phi_resolvent_closed(A, 1.0, w.info["alpha"])
    L, D = walks.walk_laplacian(phi), walks.walk_degrees(phi)
    for k in (3, 5, 13, 33, 63, 67, 100):
        ld = k + 3
        V = torch.as_tensor(np.random.default_rng(k).standard_normal((g.n, ld)), device="cuda")
        W = torch.full((g.n, ld), 7.25, dtype=torch.float64, device="cuda")
        assert wl.wl_apply(w.h, V, ld, k, W, ld) == wl.WL_OK
        want = L @ V.cpu().numpy()[:, :k]
        got = W.cpu().numpy()
        assert (got[:, k:] == 7.25).all()
        assert np.abs(got[:, :k] - want).max() <= bound * np.abs(want).max(), k
    k = 5
    U = torch.full((2, g.n, 8), 7.25, dtype=torch.float64, device="cuda")
    for shift in ((0.0, 2.0) if prec == "refined" else (0.0,)):
        w.set(shift=shift)
        assert wl.wl_expmv(w.h, V, ld, k, [0.5, 2.0], U, 8) == wl.WL_OK
        want = walks.diffusion(L, V.cpu().numpy()[:, :k], [0.5, 2.0])
        got = U.cpu().numpy()
        assert (got[:, :, k:] == 7.25).all()
        for t in range(2):
            assert np.abs(got[t, :, :k] - want[t]).max() <= bound * np.abs(want[t]).max()
    w.set(shift=0.0)
    P0 = torch.rand((g.n, ld), dtype=torch.float64, device="cuda")
    assert wl.wl_markov(w.h, P0, ld, k, [1, 3], U, 8) == wl.WL_OK
    got, p = U.cpu().numpy(), P0.cpu().numpy()[:, :k]
    for t, steps in ((0, 1), (1, 2)):
        for _ in range(steps):
            p = phi @ (p / D[:, None])
        assert np.abs(got[t, :, :k] - p).max() <= bound * np.abs(p).max()
    assert (got[:, :, k:] == 7.25).all()
    w.close()


def test_small_refined_solves_scale_with_their_columns():
    """The cooperative FP32 corrections scale each column by a power of two:
    columns of very different size give the same solutions, scaled (to the
    parity tolerance; squares of 2^+-40 stay inside FP32's range)."""
    for g in (wlgen.erdos_renyi(700, 8.0, 2), wlgen.barabasi_albert(9001, 10, 4)):
        w = WL(g, variant="nbt", alpha_rel=0.5, prec="refined", tol=1e-12)
        V = torch.as_tensor(np.random.default_rng(4).standard_normal((g.n, 8)), device="cuda")
        e = torch.tensor([0, 40, -40, 13, -27, 1, 31, -38], device="cuda")
        s = torch.pow(torch.tensor(2.0, dtype=torch.float64, device="cuda"), e)
        want = w.apply(V)
        got = w.apply(V * s) / s
        assert (got - want).abs().max() <= 1e-8 * want.abs().max(), g.name
        one = torch.stack([w.apply(V[:, :1] * c)[:, 0] / c for c in s], 1)
        assert (one - want[:, :1]).abs().max() <= 1e-8 * want.abs().max(), g.name
        w.close()


# Phase kernels: x from the residuals kept over more iterations than are kept at
# a time (near the pole), a warm start added to, several widths, and the final
# residual that the FP64 shifted solves hand on; against scipy's FP64 CG
@pytest.mark.parametrize("prec,tol,bound", [("fp64", 1e-13, 1e-10), ("refined", 1e-12, 1e-8)])
def test_solves_by_kept_residuals(prec, tol, bound):
    from oracle import krylov
    g = wlgen.erdos_renyi(220001, 6.0, 8)
    A = krylov.adjacency(g.row_ptr, g.col_idx, g.n)
    for rel in (0.3, 0.97):
        w = WL(g, variant="nbt", alpha_rel=rel, prec=prec, tol=tol)
        L = krylov.ResolventLaplacian(A, 1.0, w.info["alpha"], tol=1e-14)
        for k in (8, 16, 32) if rel < 0.5 else (16,):
            V = np.random.default_rng(k).standard_normal((g.n, k))
            V[:, 5] = 0.0
            W = w.apply(torch.as_tensor(V, device="cuda")).cpu().numpy()
            want = L.apply(V[:, :4])
            assert np.abs(W[:, :4] - want).max() <= bound * np.abs(want).max(), (rel, k)
            assert (W[:, 5] == 0.0).all()
        x0 = L.Df * (1.0 + 0.3 * np.cos(np.arange(g.n)))
        w.warm_start(torch.as_tensor(x0, device="cuda"))
        Df = w.degrees().cpu().numpy()
        assert np.abs(Df - L.Df).max() <= bound * np.abs(L.Df).max()
        if rel < 0.5:  # plain and shifted Lanczos on 16 sources agree
            w.set(outer_tol=1e-11)
            V = torch.zeros((g.n, 16), dtype=torch.float64, device="cuda")
            V[torch.arange(16) * 999, torch.arange(16)] = 1.0
            U = w.expmv(V, [0.5, 2.0])
            w.set(shift=2.0)
            S = w.expmv(V, [0.5, 2.0])
            for t in range(2):
                assert (S[t] - U[t]).abs().max() <= bound * U[t].abs().max()
        w.close()


# One column, vectors streamed: rows by the CTA (one of 70000 entries), by a warp
# and by eight lanes, groups of rows with and without one of them between, a
# last group that isn't whole, with and without the nodes ordered; against
# scipy's FP64 CG, and the spectral scale against its Lanczos solver
@pytest.mark.parametrize("reorder", [0, 1])
def test_one_column_of_many_rows(reorder):
    from scipy.sparse.linalg import eigsh
    from oracle import krylov
    n = 600037
    e = wlgen.erdos_renyi(n, 3.0, 12)
    src = np.repeat(np.arange(n), e.degrees)
    rng = np.random.default_rng(5)
    deg = {17: 70000, 5000: 3000, 299999: 4096, 300000: 4097, 450001: 257, 450002: 256, 600036: 31}
    hs = np.concatenate([np.full(d, v) for v, d in deg.items()])
    hd = np.concatenate([rng.choice(n, d, replace=False) for d in deg.values()])
    keep = hs != hd
    g = wlgen.csr_from_edges(n, np.concatenate([src, hs[keep]]), np.concatenate([e.col_idx, hd[keep]]))
    A = krylov.adjacency(g.row_ptr, g.col_idx, g.n)
    lmax = eigsh(A, k=1, which="LA", return_eigenvectors=False)[0]
    for prec, tol, bound in (("fp64", 1e-13, 1e-10), ("refined", 1e-12, 1e-8)):
        w = WL(g, variant="nbt", alpha_rel=0.5, prec=prec, tol=tol, reorder=reorder)
        assert abs(w.info["lambda_max"] - lmax) <= 1e-9 * lmax
        D = krylov.ResolventLaplacian(A, 1.0, w.info["alpha"], tol=1e-14).Df
        Df = w.degrees().cpu().numpy()
        assert np.abs(Df - D).max() <= bound * np.abs(D).max()
        w.warm_start(torch.as_tensor(D * (1.0 + 0.3 * np.cos(np.arange(n))), device="cuda"))
        Df = w.degrees().cpu().numpy()
        assert np.abs(Df - D).max() <= bound * np.abs(D).max()
        w.close()


# Batched corrections whose residuals are kept: near the pole (tens of
# iterations, so x and p are formed several times), far from it (fewer than are
# kept), an odd number of rows (unaligned halves of the buffers, one column) and
# a hub row, against the oracle's dense phi
@pytest.mark.parametrize("rel", [0.02, 0.5, 0.97])
@pytest.mark.parametrize("k", [1, 2, 4, 32])
def test_batched_corrections_by_kept_residuals(rel, k):
    from paper_2601_11338_gb300 import wl
    gs = [wlgen.erdos_renyi(301, 6.0, 4), wlgen.path(3), wlgen.star(701), wlgen.grid2d(9, 11)]
    mus = [0.25, 0.0]
    n = sum(g.n for g in gs)
    assert n % 2 == 1
    p = wl.make_params(f=wl.WL_F_RESOLVENT, alpha_rel=rel, prec=wl.WL_REFINED, tol=1e-11,
                       stream=torch.cuda.current_stream().cuda_stream)
    b = wl.wl_batch_build([(g.row_ptr.astype(np.int32), g.col_idx, g.n, g.nnz) for g in gs], mus, p)
    V = np.random.default_rng(k).standard_normal((n, k))
    V[:301, k - 1] = 0.0 if k > 1 else V[:301, 0]  # a zero column of the first graph
    Df = torch.empty((2, n), dtype=torch.float64, device="cuda")
    W = torch.empty((2, n, k), dtype=torch.float64, device="cuda")
    st = wl.wl_stats()
    assert wl.wl_batch_run(b, torch.as_tensor(V, device="cuda"), k, Df, W, 0, st, ()) == wl.WL_OK
    lo = 0
    for i, g in enumerate(gs):
        A = graph.dense_adjacency(g.row_ptr, g.col_idx, g.n)
        for s, mu in enumerate(mus):
            phi = walks.phi_resolvent_closed(A, mu, wl.wl_batch_info(b, i, s)["alpha"])
            D, L = walks.walk_degrees(phi), walks.walk_laplacian(phi)
            got, w = Df[s, lo:lo + g.n].cpu().numpy(), W[s, lo:lo + g.n].cpu().numpy()
            want = L @ V[lo:lo + g.n]
            assert np.abs(got - D).max() <= 1e-8 * np.abs(D).max(), (g.name, mu)
            assert np.abs(w - want).max() <= 1e-8 * np.abs(want).max(), (g.name, mu)
        lo += g.n
    b.destroy()


# Symmetry of the stored pattern: one entry without its mirror image at either
# end of a hub row or between equal rows, two that keep the counts equal, in
# groups of 32 rows with and without empty rows; and the sound graphs
def test_every_one_sided_entry_is_found():
    from paper_2601_11338_gb300 import wl
    rng = np.random.default_rng(3)
    n = 1301
    e = wlgen.erdos_renyi(n, 3.0, 6)
    src = np.repeat(np.arange(n), e.degrees)
    hub = rng.choice(np.arange(200, n - 100), 700, replace=False)
    g = wlgen.csr_from_edges(n, np.concatenate([src, np.full(700, 77)]), np.concatenate([e.col_idx, hub]))
    rows = np.repeat(np.arange(n), np.diff(g.row_ptr))
    cols = g.col_idx.astype(np.int64)

    def built(drop):
        keep = np.ones(cols.size, bool)
        keep[list(drop)] = False
        rp = np.concatenate([[0], np.cumsum(np.bincount(rows[keep], minlength=n))]).astype(np.int32)
        try:
            w = WL(wlgen.CSR(n, rp.astype(np.int64), cols[keep].astype(np.int32)), variant="nbt", alpha_rel=0.5)
            w.close()
            return wl.WL_OK
        except wl.WLError as err:
            return err.status

    assert built(()) == wl.WL_OK
    assert built(np.flatnonzero((rows == 77) | (cols == 77))) == wl.WL_OK  # row 77 empty, both sides gone
    hubrow, hubcol = np.flatnonzero(rows == 77), np.flatnonzero(cols == 77)
    small = np.flatnonzero((rows != 77) & (cols != 77))
    for i in (hubrow[0], hubrow[-1], hubcol[0], hubcol[-1], *rng.choice(small, 6, replace=False)):
        assert built((i,)) == wl.WL_ERR_NOT_SYMMETRIC, i
    for a, b in ((hubrow[3], hubcol[5]), (hubrow[0], hubrow[1]), (small[0], small[-1]), (hubcol[0], small[5])):
        if not (rows[a] == cols[b] and cols[a] == rows[b]):
            assert built((a, b)) == wl.WL_ERR_NOT_SYMMETRIC, (a, b)


def test_right_hand_sides_outside_the_integer_split():
    """Refined solves split their right-hand sides by integer instructions for
    values from 2^-63 to 2^127, by conversions elsewhere: entries spread over 30
    decades with both signs and zeros, values halfway between two FP32 ones,
    against the FP64 form (at the refined form's parity tolerance)."""
    g = wlgen.erdos_renyi(1500, 8.0, 2)
    rng = np.random.default_rng(8)
    V = rng.standard_normal((g.n, 4)) * 10.0 ** rng.uniform(-30, 0, (g.n, 4))
    V[::7] = 0.0
    V[1::7, 1] = np.float64(np.float32(V[1::7, 1])) * (1 + 2.0 ** -24)
    V[3::7, 1] = np.nextafter(np.float32(2.0), np.float32(0)) * (1 + 2.0 ** -24.5)
    out = []
    for prec, tol in (("fp64", 1e-13), ("refined", 1e-12)):
        w = WL(g, variant="nbt", alpha_rel=0.5, prec=prec, tol=tol)
        out.append(w.apply(torch.as_tensor(V, device="cuda")).cpu().numpy())
        w.close()
    assert (np.abs(out[1] - out[0]).max(0) <= 1e-8 * np.abs(out[0]).max(0)).all()


# Phase kernels with rows on both sides of every way a row is taken (a lane
# group up to 30 entries, a warp up to 1400, a CTA beyond), and with no row between
# 31 and 1400, against scipy's FP64 CG
@pytest.mark.parametrize("degs", [{7: 31, 99: 256, 1000: 257, 70000: 1400, 150001: 1401, 220000: 5000},
                                  {3: 1500, 219999: 3000}])
@pytest.mark.parametrize("prec,tol,bound", [("fp64", 1e-13, 1e-10), ("refined", 1e-12, 1e-8)])
def test_long_rows_of_the_phase_kernels(prec, tol, bound, degs):
    from oracle import krylov
    n = 220001
    e = wlgen.erdos_renyi(n, 4.0, 8)
    src = np.repeat(np.arange(n), e.degrees)
    rng = np.random.default_rng(6)
    hs = np.concatenate([np.full(d, v) for v, d in degs.items()])
    hd = np.concatenate([rng.choice(n, d, replace=False) for d in degs.values()])
    keep = hs != hd
    g = wlgen.csr_from_edges(n, np.concatenate([src, hs[keep]]), np.concatenate([e.col_idx, hd[keep]]))
    A = krylov.adjacency(g.row_ptr, g.col_idx, g.n)
    w = WL(g, variant="nbt", alpha_rel=0.5, prec=prec, tol=tol)
    L = krylov.ResolventLaplacian(A, 1.0, w.info["alpha"], tol=1e-14)
    for k in (8, 16, 64):
        V = np.random.default_rng(k).standard_normal((n, k))
        W = w.apply(torch.as_tensor(V, device="cuda")).cpu().numpy()
        want = L.apply(V[:, :2])
        assert np.abs(W[:, :2] - want).max() <= bound * np.abs(want).max(), k
    w.close()
