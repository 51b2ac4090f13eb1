"""An expired device-side wait of any kernel comes back as WL_ERR_TIMEOUT, at once
and whatever follows that kernel on the stream, and the handle works again
afterwards. The wait is made to have expired on the host (WL_FAULT=timeout: every
barrier starts in the gave-up state)."""
import time

import numpy as np
import pytest

import wlgen
from oracle import graph, walks

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture
def fault(monkeypatch):
    def set_mode(mode):
        monkeypatch.setenv("WL_FAULT", mode)
    yield set_mode
    monkeypatch.delenv("WL_FAULT", raising=False)


def WL(g, **kw):
    from paper_2601_11338_gb300.api import WalkLaplacian
    return WalkLaplacian(g.row_ptr.astype(np.int32), g.col_idx, g.n, **kw)


def times_out(fault, w, call):
    from paper_2601_11338_gb300 import wl
    fault("timeout")
    t0 = time.perf_counter()
    call((wl.WL_ERR_TIMEOUT,))
    assert w.last.status == wl.WL_ERR_TIMEOUT
    assert time.perf_counter() - t0 < 1.5  # no 2 s wait
    fault("")


# one cluster (300 rows), one grid (20000 rows)
@pytest.mark.parametrize("n", [300, 20000])
@pytest.mark.parametrize("shift", [0.0, 1.0])
def test_refined_cooperative_solve(fault, n, shift):
    g = wlgen.erdos_renyi(n, 6, 4)
    w = WL(g, variant="nbt", alpha_rel=0.5, tol=1e-12, prec="refined", shift=shift)
    times_out(fault, w, lambda allow: w.degrees(allow=allow))
    V = torch.as_tensor(np.random.default_rng(0).standard_normal((g.n, 4)), device="cuda")
    want = w.degrees().clone()
    U = w.expmv(V, [0.5]).clone()
    times_out(fault, w, lambda allow: w.apply(V, allow=allow))
    times_out(fault, w, lambda allow: w.expmv(V, [0.5], allow=allow))
    assert torch.equal(w.degrees(), want) and torch.equal(w.expmv(V, [0.5]), U)
    if n <= 300:
        A = graph.dense_adjacency(g.row_ptr, g.col_idx, g.n)
        D = walks.walk_degrees(walks.phi_resolvent_closed(A, 1.0, w.info["alpha"]))
        assert np.abs(want.cpu().numpy() - D).max() <= 1e-8 * np.abs(D).max()
    w.close()


def test_refined_streamed_solve_of_one_column(fault):
    g = wlgen.erdos_renyi(520000, 3, 4)  # beyond the rows that stay in shared memory
    w = WL(g, variant="nbt", alpha_rel=0.5, tol=1e-12, prec="refined")
    times_out(fault, w, lambda allow: w.degrees(allow=allow))
    want = w.degrees().clone()
    times_out(fault, w, lambda allow: w.degrees(allow=allow))
    assert torch.equal(w.degrees(), want)
    w.close()
