"""The library as it runs where the device places no thread-block clusters
(WL_FAULT=nocluster takes the placement away, on the host)."""
import numpy as np
import pytest

import wlgen
from oracle import graph, walks

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# bounds: those of the parity tests of each form
@pytest.mark.parametrize("prec,tol,bound", [("fp64", 1e-13, 1e-10), ("refined", 1e-12, 1e-8)])
@pytest.mark.parametrize("n,k", [(2, 1), (40, 2), (300, 5), (1023, 1), (1900, 16)])
def test_small_solves_without_clusters(monkeypatch, prec, tol, bound, n, k):
    from paper_2601_11338_gb300.api import WalkLaplacian
    monkeypatch.setenv("WL_FAULT", "nocluster")
    g = wlgen.erdos_renyi(n, 6.0, 11) if n > 2 else wlgen.path(2)
    A = graph.dense_adjacency(g.row_ptr, g.col_idx, g.n)
    w = WalkLaplacian(g.row_ptr.astype(np.int32), g.col_idx, g.n, variant="btdw", mu=0.4, alpha_rel=0.5, prec=prec,
                      tol=tol)
    phi = walks.phi_resolvent_closed(A, 0.4, w.info["alpha"])
    D = walks.walk_degrees(phi)
    assert np.abs(w.degrees().cpu().numpy() - D).max() <= bound * np.abs(D).max()
    V = np.random.default_rng(n).standard_normal((g.n, k))
    want = walks.walk_laplacian(phi) @ V
    W = w.apply(torch.as_tensor(V, device="cuda")).cpu().numpy()
    assert np.abs(W - want).max() <= bound * np.abs(want).max()
    w.close()
