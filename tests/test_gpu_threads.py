"""Handles in different host threads: nearly every solve is one kernel over the
whole chip whose CTAs wait for one another, so the handles' kernels take turns. Each
gives the results that it gives alone."""
import gc
import threading

import numpy as np
import pytest

import wlgen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class Job:
    def __init__(self, g, k, calls, **kw):
        from paper_2601_11338_gb300.api import WalkLaplacian
        self.stream = torch.cuda.Stream()
        self.w = WalkLaplacian(g.row_ptr.astype(np.int32), g.col_idx, g.n, variant="nbt", alpha_rel=0.5,
                               stream=self.stream.cuda_stream, **kw)
        self.V = torch.as_tensor(np.random.default_rng(k).standard_normal((g.n, k)), device="cuda")
        self.calls, self.n, self.k = calls, g.n, k
        self.D = torch.zeros(g.n, dtype=torch.float64, device="cuda")
        self.W = torch.zeros((g.n, k), dtype=torch.float64, device="cuda")
        self.U = torch.zeros((1, g.n, k), dtype=torch.float64, device="cuda")
        self.error = None
        torch.cuda.synchronize()

    def once(self):
        self.w.degrees(out=self.D)
        self.w.apply(self.V, out=self.W)
        self.w.expmv(self.V, [0.3], out=self.U)

    def run(self, want):
        try:
            for _ in range(self.calls):
                self.once()
                for got, exp in zip((self.D, self.W, self.U), want):
                    assert torch.equal(got, exp)
        except BaseException as e:  # handed to the main thread
            self.error = e


@pytest.fixture
def collected():
    yield
    gc.collect()  # the jobs' tensors go here, and not during a later test that watches the memory in use


def test_two_handles_in_two_threads(collected):
    """One cluster, one grid of few CTAs, and grids over all SMs, side by side."""
    jobs = [Job(wlgen.erdos_renyi(300, 6, 4), 1, 12, prec="fp64", tol=1e-11),
            Job(wlgen.erdos_renyi(20011, 10, 5), 13, 8, prec="refined", tol=1e-10),
            Job(wlgen.chung_lu(60000), 8, 4, prec="refined", tol=1e-10, shift=1.0),
            Job(wlgen.barabasi_albert(5000, 6, 3), 4, 8, prec="fp64", tol=1e-11)]
    wants = []
    for j in jobs:
        j.once()
        wants.append([t.clone() for t in (j.D, j.W, j.U)])
    for pair in ((0, 1), (1, 2), (3, 2), (0, 3)):
        ts = [threading.Thread(target=jobs[i].run, args=(wants[i],)) for i in pair]
        for t in ts:
            t.start()
        for t in ts:
            t.join()
        for i in pair:
            if jobs[i].error is not None:
                raise jobs[i].error
    for j in jobs:
        j.w.close()
