"""Performance cases of the walk-Laplacian library: what a user has it do,
through the public entry points, over the range of sizes it is used at.

A case names one operation on one seeded synthetic graph:

  op      what one pass runs (see `run`)
  graph   er (Erdos-Renyi, mean degree 8), chunglu (power law 2.5, mean degree
          12), rmat (edge factor 16, or `ef`), grid (2D 4-neighbour) or mix (uneven
          sizes of ER, Barabasi-Albert and grids, for the batched executor)
  n       nodes (rmat: the scale is log2 n; mix: the largest graph)
  variant allwalk, nbt or btdw (with its mu); f = resolvent throughout, alpha
          = 0.5 / rho(Z_mu), or 0.25 on grids (near the pole there)
  prec    fp64 (the plain form, the default of the API) or refined
  k       columns: right-hand sides, sources or test vectors

The graph, the right-hand sides and the handle are made in `prepare`; what
depends on the call alone (walk degrees, solves, Lanczos steps) in `run`.
`exact` gives the same results by plain FP64 torch: conjugate gradients and
Lanczos with full reorthogonalisation on a sparse CSR product.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import wlgen
from paper_2601_11338_gb300 import wl
from paper_2601_11338_gb300.api import WalkLaplacian, csr_to_device, mlp_features
from paper_2601_11338_gb300.warmstart import initial_params

MUS = (0.0, 0.25, 0.5, 0.75, 1.0)  # backtrack weights of the batched sweep


def listed():
    return [
        # One small network, the size of the paper's examples and of the unit
        # tests: walk degrees and four columns in the default FP64 form. Bound
        # by launches and waits.
        dict(name="er2k_degrees_apply", op="degrees_apply", graph="er", n=2000, variant="allwalk", mu=0.0, prec="fp64",
             k=4, tol=1e-12),
        # Diffusion from one node of that network (the smallest exp(-tau L) u).
        dict(name="er2k_diffusion", op="expmv", graph="er", n=2000, variant="allwalk", mu=0.0, prec="fp64", k=1,
             tol=1e-12, outer_tol=1e-10, shift=0.0),
        # A mid-size network and a column count that is no power of two, with
        # partial backtrack weighting, in the refined form.
        dict(name="er20k_apply_ragged", op="apply", graph="er", n=20011, variant="btdw", mu=0.5, prec="refined", k=13,
             tol=1e-10),
        # A user with a new power-law graph: validation, relabelling, spectral
        # scale, then its walk degrees.
        dict(name="chunglu400k_new_graph", op="build", graph="chunglu", n=400003, variant="nbt", mu=1.0,
             prec="refined", k=1, tol=1e-10),
        # The plain FP64 Krylov form on a block of 16 vectors.
        dict(name="chunglu300k_apply_fp64", op="apply", graph="chunglu", n=300000, variant="nbt", mu=1.0, prec="fp64",
             k=16, tol=1e-12),
        # The benchmark workload: diffusion of 16 point sources at three times
        # by shift-and-invert Lanczos, refined form. The largest case.
        dict(name="chunglu1m_diffusion", op="expmv", graph="chunglu", n=1000000, variant="nbt", mu=1.0,
             prec="refined", k=16, tol=1e-10, outer_tol=1e-8, shift=2.0),
        # Walk degrees of a graph with heavy hubs (one right-hand side, the
        # gather's worst locality).
        dict(name="rmat20_degrees", op="degrees", graph="rmat", n=1 << 20, variant="allwalk", mu=0.0, prec="refined",
             k=1, tol=1e-10),
        # XNysTrace with 64 test vectors in the accurate mixed form (the widest
        # block).
        dict(name="rmat17_trace", op="trace", graph="rmat", n=1 << 17, variant="allwalk", mu=0.0, prec="refined",
             k=64, tol=1e-10),
        # Node features of the learned warm start (triangle counts above all).
        dict(name="rmat18_features", op="features", graph="rmat", n=1 << 18, variant="nbt", mu=1.0, prec="refined",
             k=1, tol=1e-10),
        # One training step of the warm-start network and its prediction, on
        # the rows of a few graphs.
        dict(name="mlp_step_200k", op="mlp", graph="rows", n=200003, variant="", mu=0.0, prec="", k=1, tol=0.0),
        # Many graphs of uneven size, five backtrack weights, 32 columns, in
        # one captured launch.
        dict(name="batch24_run", op="batch", graph="mix", n=20000, variant="btdw", mu=0.0, prec="refined", k=32,
             tol=1e-10),
        # Average return probability on a road-like grid, near the pole.
        dict(name="grid250_return_prob", op="return_prob", graph="grid", n=62500, variant="nbt", mu=1.0,
             prec="refined", k=30, tol=1e-12, outer_tol=1e-10, shift=1.0),
    ]


# Drawn cases: (weight, op, graph, n range, k range, precisions). No drawn case
# costs more than chunglu1m_diffusion.
_RANGES = [
    (3, "degrees_apply", "er", (300, 60000), (1, 32), ("fp64", "refined")),
    (2, "expmv", "er", (300, 20000), (1, 16), ("fp64", "refined")),
    (2, "apply", "er", (2000, 200000), (1, 64), ("refined",)),
    (2, "build", "chunglu", (5000, 500000), (1, 1), ("fp64", "refined")),
    (3, "apply", "chunglu", (5000, 300000), (1, 32), ("fp64", "refined")),
    (2, "expmv", "chunglu", (20000, 500000), (1, 16), ("refined",)),
    (2, "degrees", "rmat", (1 << 13, 1 << 20), (1, 1), ("fp64", "refined")),
    (1, "trace", "rmat", (1 << 12, 1 << 17), (8, 64), ("refined",)),
    (2, "features", "rmat", (1 << 13, 1 << 18), (1, 1), ("refined",)),
    (1, "mlp", "rows", (1000, 200000), (1, 1), ("",)),
    (1, "batch", "mix", (3000, 20000), (32, 32), ("refined",)),
    (1, "return_prob", "grid", (900, 40000), (8, 30), ("refined",)),
]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    w = [r[0] for r in _RANGES]
    _, op, graph, nr, kr, precs = rng.choices(_RANGES, weights=w)[0]
    n = _spread(rng, *nr)
    k = _spread(rng, *kr)
    if graph == "rmat":
        n = 1 << max(int(round(math.log2(n))), 12)
    if graph == "grid":
        n = max(int(round(math.sqrt(n))), 2) ** 2
    variant, mu = rng.choice((("allwalk", 0.0), ("nbt", 1.0), ("btdw", round(rng.uniform(0.05, 0.95), 3))))
    prec = rng.choice(precs)
    if op == "batch":
        k = rng.choice((1, 2, 4, 8, 16, 32))
        variant, mu = "btdw", 0.0
    if op == "mlp":
        variant, mu = "", 0.0
    if graph == "grid":
        variant, mu = "nbt", 1.0  # alpha = 0.25 is below 1 / rho there
    c = dict(op=op, graph=graph, n=n, variant=variant, mu=mu, prec=prec, k=k,
             tol=0.0 if op == "mlp" else 1e-12 if prec == "fp64" else 1e-10)
    if graph == "rmat":
        c["ef"] = rng.randint(6, 16)
    if op in ("expmv", "return_prob"):
        c["tol"] = 1e-12 if graph != "chunglu" else 1e-10
        c["outer_tol"] = 1e-10 if graph != "chunglu" else 1e-8
        c["shift"] = {"er": 0.0, "chunglu": rng.choice((0.0, 2.0)), "grid": 1.0}[graph]
    return c


# ---------------------------------------------------------------- inputs
def _graph(case, seed):
    kind, n = case["graph"], case["n"]
    if kind == "er":
        return wlgen.erdos_renyi(n, 8.0, seed)
    if kind == "chunglu":
        return wlgen.chung_lu(n, 2.5, 12.0, seed)
    if kind == "rmat":
        return wlgen.rmat(n.bit_length() - 1, case.get("ef", 16), 0.57, 0.19, 0.19, seed)
    r = int(round(math.sqrt(n)))
    return wlgen.grid2d(r, r)


def _mix(case, seed):
    """24 graphs with sizes spread over [1000, n], the kinds of wlgen.batch_graphs in turn."""
    out = []
    for i in range(24):
        size = int(1000 * (case["n"] / 1000) ** ((7 * i % 24) / 23))
        r = int(round(math.sqrt(size)))
        if i % 3 == 0:
            out.append(wlgen.erdos_renyi(size, 10.0, seed * 1000 + i))
        elif i % 3 == 1:
            out.append(wlgen.barabasi_albert(size, 3, seed * 1000 + i))
        else:
            out.append(wlgen.grid2d(r, size // r))
    return out


def _scale(case):
    return dict(alpha=0.25) if case["graph"] == "grid" else dict(alpha_rel=0.5)


def _sources(case, g, seed):
    """Right-hand sides: point sources for a diffusion, Gaussian columns for an apply."""
    if case["op"] == "expmv":
        return wlgen.unit_block(g.n, wlgen.point_sources(g, case["k"], seed))
    return wlgen.gaussian_block(g.n, case["k"], seed)


def _rows(case, seed):
    """Feature rows as the generated graphs give them (standardised scale), targets near them, x_an."""
    rng = np.random.default_rng(seed)
    n = case["n"]
    d = np.floor(np.exp(rng.gamma(2.0, 0.9, n))) + 1.0
    ad = d * np.exp(1.5 + 0.5 * rng.standard_normal(n))
    t = np.floor(0.02 * d * d * rng.uniform(0, 1, n))
    F = np.log1p(np.stack([d, ad, t, np.maximum(ad - d, 0.0)], 1)).astype(np.float32)
    T = (0.05 * np.tanh(F[:, 0] - 1.0) + 0.02 * F[:, 2] / (1 + F[:, 1])).astype(np.float32)
    p = initial_params(seed)
    p[0:4], p[4:8] = F.mean(0), F.std(0)
    return F, T, p, np.exp(0.1 * F[:, 0].astype(np.float64))


def _times():
    return np.linspace(0.0, 100.0, 24)


TAUS = {"er": [1.0], "chunglu": [0.1, 1.0, 10.0]}


def prepare(case, seed):
    s = {"case": case, "seed": seed}
    op = case["op"]
    if op == "mlp":
        F, T, p, xan = _rows(case, seed)
        s.update(F=torch.as_tensor(F).cuda(), T=torch.as_tensor(T).cuda(), p=torch.as_tensor(p).cuda(),
                 xan=torch.as_tensor(xan).cuda())
        s["grad"] = torch.empty_like(s["p"])
        s["out"] = torch.empty_like(s["xan"])
        return s
    if op == "batch":
        gs = _mix(case, seed)
        par = wl.make_params(alpha_rel=0.5, prec=wl.WL_REFINED, tol=case["tol"],
                             stream=torch.cuda.current_stream().cuda_stream)
        s["b"] = wl.wl_batch_build([(g.row_ptr.astype(np.int32), g.col_idx, g.n, g.nnz) for g in gs], MUS, par)
        n = sum(g.n for g in gs)
        s["V"] = torch.as_tensor(wlgen.gaussian_block(n, case["k"], seed)).cuda()
        s["Df"] = torch.empty((len(MUS), n), dtype=torch.float64, device="cuda")
        s["W"] = torch.empty((len(MUS), n, case["k"]), dtype=torch.float64, device="cuda")
        return s
    g = _graph(case, seed)
    rp, ci = csr_to_device(g.row_ptr, g.col_idx)
    kw = dict(variant=case["variant"], mu=case["mu"], prec=case["prec"], tol=case["tol"],
              outer_tol=case.get("outer_tol", 0.0), shift=case.get("shift", 0.0), **_scale(case))
    if op == "build":
        s.update(rp=rp, ci=ci, n=g.n, kw=kw)
        return s
    s["w"] = WalkLaplacian(rp, ci, g.n, **kw)
    if op in ("degrees_apply", "apply", "expmv"):
        s["V"] = torch.as_tensor(_sources(case, g, seed)).cuda()
    if op == "apply":
        s["w"].degrees()  # a program that applies L has its walk degrees already
    return s


def run(s):
    c = s["case"]
    op = c["op"]
    if op == "degrees_apply":
        return s["w"].degrees(), s["w"].apply(s["V"])
    if op == "apply":
        return s["w"].apply(s["V"])
    if op == "expmv":
        return s["w"].expmv(s["V"], TAUS[c["graph"]])
    if op == "degrees":
        return s["w"].degrees()
    if op == "build":
        w = WalkLaplacian(s["rp"], s["ci"], s["n"], **s["kw"])
        info = w.info
        D = w.degrees()
        w.close()
        return D, info["rho"], info["lambda_max"], info["alpha"]
    if op == "trace":
        return s["w"].trace(c["k"], s["seed"])
    if op == "features":
        return mlp_features(s["w"])
    if op == "mlp":
        st = torch.cuda.current_stream().cuda_stream
        loss = wl.wl_mlp_loss_grad(s["p"], s["F"], s["T"], c["n"], s["grad"], st)
        wl.wl_mlp_predict(s["p"], s["F"], c["n"], s["xan"], s["out"], st)
        return s["grad"], s["out"], loss
    if op == "batch":
        wl.wl_batch_run(s["b"], s["V"], c["k"], s["Df"], s["W"])
        return s["Df"], s["W"]
    if op == "return_prob":
        return s["w"].return_prob(c["k"], s["seed"], _times())
    raise ValueError(op)


# ---------------------------------------------------------------- work of a pass
def work(case):
    """Bytes: the graph, inputs and outputs once. Operations: the additions of
    the operator products that a Krylov method needs at these tolerances, about
    12 a solve at alpha = 0.5 / rho (30 on the grid, near its pole), one solve
    per Lanczos step, about 20 steps."""
    op, n, k = case["op"], case["n"], case["k"]
    deg = {"er": 8, "chunglu": 12, "rmat": 1.9 * case.get("ef", 16), "grid": 4, "mix": 7, "rows": 0}[case["graph"]]
    if op == "mlp":
        fwd = 2 * (4 * 64 + 64 * 64 + 64)
        return {"bytes": n * (16 + 4 + 8 + 8), "flops": n * fwd * 4}
    if op == "batch":
        n = int(24 * (n - 1000) / math.log(n / 1000))  # mean of the log-uniform sizes
        nnz = n * deg
        return {"bytes": 4 * (n + nnz) + n * k * 8 + 5 * (n * 8 + n * k * 8), "flops": 5 * 12 * 2 * nnz * (k + 1)}
    nnz = n * deg
    csr = 4 * (n + 1) + 4 * nnz
    if op == "degrees":
        return {"bytes": csr + 8 * n, "flops": 12 * 2 * nnz}
    if op == "degrees_apply":
        return {"bytes": csr + 8 * n + 16 * n * k, "flops": 12 * 2 * nnz * (k + 1)}
    if op == "apply":
        return {"bytes": csr + 8 * n + 16 * n * k, "flops": 12 * 2 * nnz * k}
    if op == "build":
        return {"bytes": csr + 8 * n, "flops": 60 * 2 * nnz}
    if op == "expmv":
        nt = len(TAUS[case["graph"]])
        return {"bytes": csr + 8 * n * k * (1 + nt), "flops": 20 * 12 * 2 * nnz * k}
    if op == "trace":
        return {"bytes": csr, "flops": 12 * 2 * nnz * k + 4 * n * k * k}
    if op == "features":
        return {"bytes": csr + 24 * n, "flops": 8 * nnz}
    return {"bytes": csr, "flops": 20 * 30 * 2 * nnz * k}


# ---------------------------------------------------------------- the same results in plain FP64
class _Op:
    """A as a sparse FP64 CSR tensor, its degrees, and M_mu(alpha)."""

    def __init__(self, g):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        self.n = g.n
        self.A = torch.sparse_csr_tensor(torch.as_tensor(g.row_ptr), torch.as_tensor(g.col_idx.astype(np.int64)),
                                         torch.ones(g.nnz, dtype=torch.float64), size=(g.n, g.n)).to(dev)
        self.d = torch.as_tensor(g.degrees.astype(np.float64), device=dev)
        self.dev = dev

    def largest(self, diag, u=None):
        """Largest eigenvalue (and vector) of A + diag by Lanczos with full reorthogonalisation."""
        gen = torch.Generator(device="cpu").manual_seed(7)
        v = u if u is not None else torch.rand(self.n, dtype=torch.float64, generator=gen).to(self.dev) + 0.5
        m = min(self.n, 120)
        for _ in range(30):
            Q = torch.zeros((m + 1, self.n), dtype=torch.float64, device=self.dev)
            Q[0] = v / v.norm()
            al, be, cut = [], [], m
            for j in range(m):
                w = self.A @ Q[j] + diag * Q[j]
                for _r in range(2):
                    h = Q[: j + 1] @ w
                    w = w - h @ Q[: j + 1]
                    if _r == 0:
                        al.append(float(h[j]))
                b = float(w.norm())
                be.append(b)
                if b <= 1e-13 * max(1.0, abs(al[0])):
                    cut = j + 1
                    break
                Q[j + 1] = w / b
                if j % 10 == 9:
                    T = np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1)
                    e, z = np.linalg.eigh(T)
                    if abs(b * z[-1, -1]) <= 1e-9 * abs(e[-1]):
                        cut = j + 1
                        break
            T = np.diag(al) + np.diag(be[: cut - 1], 1) + np.diag(be[: cut - 1], -1)
            e, z = np.linalg.eigh(T)
            v = torch.as_tensor(z[:, -1].copy(), device=self.dev) @ Q[:cut]
            if cut < m or be[cut - 1] * abs(z[-1, -1]) <= 1e-9 * abs(e[-1]):
                break
        return float(e[-1]), v

    def rho(self, mu):
        """rho(Z_mu): the root of lambda_max(A - (mu/lambda)(D - mu I)) = lambda."""
        lmax, u = self.largest(torch.zeros_like(self.d))
        if mu == 0.0:
            return lmax, lmax
        lam = lmax
        for _ in range(60):
            # Rayleigh functional of the last vector, then a new vector there
            t, u = self.largest(-(mu / lam) * (self.d - mu), u)
            u = u / u.norm()
            q = float(u @ (self.d * u))
            uAu = float(u @ (self.A @ u))
            c = mu * (q - mu)
            new = 0.5 * (uAu + math.sqrt(max(uAu * uAu - 4 * c, 0.0)))
            if abs(new - lam) <= 1e-14 * lam:
                lam = new
                break
            lam = new
        return lam, lmax

    def setup(self, mu, alpha=None):
        self.rho_z, self.lmax = (None, None) if alpha is not None else self.rho(mu)
        self.mu = mu
        self.alpha = alpha if alpha is not None else 0.5 / self.rho_z
        a = self.alpha
        self.a = 1.0 - mu * mu * a * a
        self.md = self.a + a * a * mu * self.d
        return self

    def phi(self, B):
        """(1 - mu^2 alpha^2) M^{-1} B by CG to 1e-15."""
        B = self.a * B
        X = torch.zeros_like(B)
        R, P = B.clone(), B.clone()
        g = (R * R).sum(0)
        g0 = g.clone().clamp_min(1e-300)
        for _ in range(200):
            Q = self.md[:, None] * P - self.alpha * (self.A @ P)
            al = g / (P * Q).sum(0).clamp_min(1e-300)
            X += al * P
            R -= al * Q
            gn = (R * R).sum(0)
            if bool((gn <= 1e-30 * g0).all()):
                break
            P = R + (gn / g.clamp_min(1e-300)) * P
            g = gn
        return X

    def degrees(self):
        return self.phi(torch.ones((self.n, 1), dtype=torch.float64, device=self.dev))[:, 0]

    def diffusion(self, U0, taus):
        """exp(-tau L) U0 by Lanczos on L, all columns side by side."""
        D = self.degrees()[:, None]
        nrm = U0.norm(dim=0)
        Q = [U0 / nrm]
        al, be, prev = [], [], None
        for j in range(160):
            w = D * Q[j] - self.phi(Q[j])
            if j:
                w = w - be[j - 1] * Q[j - 1]
            a = (w * Q[j]).sum(0)
            w = w - a * Q[j]
            for q in Q:
                w = w - (q * w).sum(0) * q
            b = w.norm(dim=0)
            al.append(a)
            be.append(b)
            Q.append(w / b.clamp_min(1e-300))
            if j % 4 == 3:
                A_, B_ = torch.stack(al).cpu().numpy(), torch.stack(be).cpu().numpy()
                Y = np.zeros((len(taus), j + 1, U0.shape[1]))
                for c in range(U0.shape[1]):
                    e, z = np.linalg.eigh(np.diag(A_[:, c]) + np.diag(B_[:-1, c], 1) + np.diag(B_[:-1, c], -1))
                    for t, tau in enumerate(taus):
                        Y[t, :, c] = z @ (np.exp(-tau * e) * z[0])
                if prev is not None and np.abs(Y[:, : prev.shape[1]] - prev).max() < 1e-14 and np.abs(
                        Y[:, prev.shape[1]:]).max() < 1e-14:
                    break
                prev = Y
        Yd = torch.as_tensor(Y, device=self.dev)
        out = torch.zeros((len(taus), self.n, U0.shape[1]), dtype=torch.float64, device=self.dev)
        for i in range(Yd.shape[1]):
            out += Yd[:, i][:, None, :] * (Q[i] * nrm)
        return out


def _triangles(g):
    """Triangles through every node: wedges of the degree-ordered orientation looked up among its edges."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    n = g.n
    deg = torch.as_tensor(g.degrees, device=dev)
    rank = torch.empty(n, dtype=torch.int64, device=dev)
    rank[torch.argsort(deg, stable=True)] = torch.arange(n, device=dev)
    src = torch.repeat_interleave(torch.arange(n, device=dev), deg)
    dst = torch.as_tensor(g.col_idx.astype(np.int64), device=dev)
    a, b = rank[src], rank[dst]
    a, b = a[a < b], b[a < b]
    key, _ = torch.sort(a * n + b)
    a, b = key // n, key % n
    out = torch.bincount(a, minlength=n)
    start = torch.cumsum(out, 0) - out
    t = torch.zeros(n, dtype=torch.int64, device=dev)
    wedges = out[b]
    ends = torch.cumsum(wedges, 0)
    total = int(ends[-1]) if ends.numel() else 0
    if total > 4_000_000_000:
        return None
    e0, step = 0, 1 << 26
    while e0 < a.numel():
        base = int(ends[e0 - 1]) if e0 else 0
        e1 = max(e0 + 1, int(torch.searchsorted(ends, base + step)))
        w = wedges[e0:e1]
        u, v = torch.repeat_interleave(a[e0:e1], w), torch.repeat_interleave(b[e0:e1], w)
        off = torch.arange(u.numel(), device=dev) - torch.repeat_interleave(torch.cumsum(w, 0) - w, w)
        x = b[start[v] + off]
        q = u * n + x
        pos = torch.searchsorted(key, q).clamp_max(key.numel() - 1)
        hit = key[pos] == q
        for z in (u, v, x):
            t += torch.bincount(z[hit], minlength=n)
        e0 = e1
    return t[rank]


def exact(case, seed):
    op = case["op"]
    if op in ("batch", "trace", "return_prob"):
        return None  # as many eigenproblems, or this library's own random draws
    if op == "mlp":
        F, T, p, xan = _rows(case, seed)
        q = torch.as_tensor(p.astype(np.float64)).requires_grad_(True)
        F, T = torch.as_tensor(F.astype(np.float64)), torch.as_tensor(T.astype(np.float64))
        s = (F - q[0:4].detach()) / q[4:8].detach()
        W1, b1, W2, b2 = q[8:264].view(64, 4), q[264:328], q[328:4424].view(64, 64), q[4424:4488]
        W3, b3 = q[4488:4552], q[4552]
        y = torch.tanh(torch.tanh(s @ W1.T + b1) @ W2.T + b2) @ W3 + b3
        loss = ((y - T) ** 2).mean()
        loss.backward()
        return q.grad, torch.as_tensor(xan) * torch.exp(y.detach()), float(loss)
    g = _graph(case, seed)
    o = _Op(g).setup(case["mu"], _scale(case).get("alpha"))
    if op == "degrees":
        return o.degrees()
    if op == "build":
        return o.degrees(), o.rho_z, o.lmax, o.alpha
    if op == "features":
        d = o.d
        ad = o.A @ d
        a, mu, al = o.a, o.mu, o.alpha
        c1 = (al - al * al * mu) / a
        xan = 1.0 + c1 * d + c1 * (al * ad - al * al * mu * d * d) / a
        t = _triangles(g)
        if t is None:
            return None, xan
        return torch.log1p(torch.stack([d, ad, t.double(), ad - d], 1)), xan
    V = torch.as_tensor(_sources(case, g, seed), device=o.dev)
    if op == "expmv":
        return o.diffusion(V, TAUS[case["graph"]])
    D = o.degrees()
    W = D[:, None] * V - o.phi(V)
    return (D, W) if op == "degrees_apply" else W
