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


@pytest.mark.parametrize("n", [300, 20000])
def test_fp64_cooperative_solve(fault, n):
    g = wlgen.erdos_renyi(n, 6, 4)
    w = WL(g, variant="nbt", alpha_rel=0.5, tol=1e-12, prec="fp64")
    times_out(fault, w, lambda allow: w.degrees(allow=allow))
    want = w.degrees().clone()
    times_out(fault, w, lambda allow: w.degrees(allow=allow))
    assert torch.equal(w.degrees(), want)
    w.close()


def test_fp64_streamed_solve_of_one_column(fault):
    # more than half of the entries in long rows: hubs worth keeping in shared memory
    g = wlgen.star(620000)
    w = WL(g, variant="nbt", alpha=1e-4, tol=1e-12, prec="fp64")
    times_out(fault, w, lambda allow: w.degrees(allow=allow))
    want = w.degrees().clone()
    assert torch.equal(w.degrees(), want)
    w.close()


def test_sketch_solve(fault):
    from paper_2601_11338_gb300 import wl
    g = wlgen.erdos_renyi(3000, 6, 4)
    w = WL(g, variant="nbt", alpha_rel=0.5, prec="sketch")
    want = w.trace(16, 5)
    fault("timeout")
    with pytest.raises(wl.WLError) as e:
        w.trace(16, 5)
    assert e.value.status == wl.WL_ERR_TIMEOUT
    fault("")
    assert w.trace(16, 5) == want
    w.close()


@pytest.mark.parametrize("n", [300, 260000])  # vectors in shared memory, and streamed
def test_spectral_search(fault, n):
    from paper_2601_11338_gb300 import wl
    g = wlgen.erdos_renyi(n, 4, 4)
    fault("timeout")
    with pytest.raises(wl.WLError) as e:
        WL(g, variant="nbt", alpha_rel=0.5)
    assert e.value.status == wl.WL_ERR_TIMEOUT
    fault("")
    w = WL(g, variant="nbt", alpha_rel=0.5)
    assert w.info["rho"] > 1.0
    w.close()


def test_outer_lanczos_step_fp64(fault):
    """f = identity makes no solve: the first kernel that waits is the Lanczos step."""
    g = wlgen.erdos_renyi(300, 6, 4)
    w = WL(g, f="identity", prec="fp64")
    U0 = torch.zeros((g.n, 2), dtype=torch.float64, device="cuda")
    U0[0, 0] = U0[7, 1] = 1.0
    want = w.expmv(U0, [1.0]).clone()
    times_out(fault, w, lambda allow: w.expmv(U0, [1.0], allow=allow))
    assert torch.equal(w.expmv(U0, [1.0]), want)
    w.close()


def test_outer_lanczos_step_refined(fault):
    """Solves by the phase kernels (16 columns, more rows than the SMs hold) wait for
    nothing; a Lanczos run of one step is checked after it."""
    from paper_2601_11338_gb300 import wl
    g = wlgen.erdos_renyi(200003, 6, 3)
    w = WL(g, variant="nbt", alpha_rel=0.5, tol=1e-10, prec="refined", max_outer=1)
    U0 = torch.as_tensor(np.random.default_rng(0).standard_normal((g.n, 16)), device="cuda")
    w.degrees()
    capped = (wl.WL_ERR_NO_CONVERGENCE,)
    want = w.expmv(U0, [0.5], allow=capped).clone()
    times_out(fault, w, lambda allow: w.expmv(U0, [0.5], allow=allow + capped))
    assert torch.equal(w.expmv(U0, [0.5], allow=capped), want)
    w.close()
