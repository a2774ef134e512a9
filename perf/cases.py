"""Performance cases of the M-RA library: the calls its users make, over their range.

A case is one call through the package's public entry points on one problem:

* ``loglik``   -- the log-likelihood at a parameter vector (one step of any
  likelihood-based inference), in each of the three precision forms;
* ``grad``     -- log-likelihood and gradient (one step of a maximum-likelihood
  fit), through ``torch.autograd`` or ``Handle.loglik_grad``;
* ``predict``  -- kriging means and variances from a fitted handle;
* ``refresh``  -- new locations and data of the same size on a kept handle
  (host arrays, as they arrive), then the log-likelihood;
* ``batch``    -- many datasets of uneven size in one call.

Problems are seeded draws shaped like the paper's data: locations uniform on
the unit square or in satellite-style swaths, a random-Fourier-feature draw of
the field plus measurement noise.  ``exact`` evaluates the same quantities in
FP64 with batched torch linear algebra, written from the recursions of Sec. 3
in block-Cholesky form; it shares no code with the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1507_04789_gb300 import autograd, mra

DEV = "cuda"


# ---- the cases -----------------------------------------------------------------
def listed():
    return [
        # a small field (a county, a test site) on the default FP64 form: launch latency
        dict(name="loglik_4k_fp64", op="loglik", precision="fp64", n=4096, M=3, r=16, family="exp", layout="uniform"),
        # a mid-sized field, few regions a level: latency of the tensor-core form
        dict(name="loglik_16k_emu", op="loglik", precision="emu", n=16384, M=4, r=64, family="matern15",
             layout="uniform"),
        # a million observations, 64 knots: the library's main workload
        dict(name="loglik_1M_emu", op="loglik", precision="emu", n=1 << 20, M=7, r=64, family="matern15",
             layout="uniform"),
        # the default form at a quarter of a million observations
        dict(name="loglik_256k_fp64", op="loglik", precision="fp64", n=1 << 18, M=6, r=64, family="matern15",
             layout="uniform"),
        # the 3xTF32 form, an odd number of observations and the 7 x 7 knot grid of Sec. 4.2
        dict(name="loglik_100k_mixed", op="loglik", precision="mixed", n=100003, M=6, r=49, family="exp",
             layout="uniform"),
        # one step of a maximum-likelihood fit through torch.autograd
        dict(name="grad_256k_emu", op="grad", precision="emu", n=1 << 18, M=6, r=64, family="matern15",
             layout="uniform", torch=True),
        # the same on the default form, a small field
        dict(name="grad_16k_fp64", op="grad", precision="fp64", n=16384, M=4, r=64, family="matern15",
             layout="uniform", torch=False),
        # the map of a fitted model: a 512 x 512 grid
        dict(name="predict_256k_emu", op="predict", precision="emu", n=1 << 18, M=6, r=64, family="matern15",
             layout="uniform", points=1 << 18, host=False),
        # predictions at a list of sites, host arrays
        dict(name="predict_1k_fp64", op="predict", precision="fp64", n=4096, M=3, r=16, family="exp",
             layout="uniform", points=1024, host=True),
        # a day's swaths replace yesterday's: sparse and empty leaves, nonstationary variance
        dict(name="refresh_150k_swath_emu", op="refresh", precision="emu", n=150001, M=7, r=32, family="exp",
             layout="swath"),
        # many datasets (one a day, one a sensor) of uneven size in swaths, pruned trees
        dict(name="batch_16_swath_emu", op="batch", precision="emu", ndata=16, n=10000, n_max=200000, r=32,
             family="exp", layout="swath"),
    ]


def _levels(n: int, per_leaf: float = 64.0) -> int:
    """Quadtree levels with at most about ``per_leaf`` observations per leaf on average."""
    return max(1, math.ceil(math.log(n / per_leaf) / math.log(4.0) - 1e-9))


def _log_uniform(rng, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["loglik", "loglik", "loglik", "grad", "predict", "refresh", "batch"])
    r = rng.choice([16, 25, 32, 36, 48, 49, 64, 64])
    family = rng.choice(["exp", "matern15"])
    if op == "loglik":
        precision = rng.choice(["fp64", "emu", "emu", "mixed"])
        n = _log_uniform(rng, 4096, {"fp64": 200000, "emu": 700000, "mixed": 300000}[precision])
        return dict(op=op, precision=precision, n=n, M=_levels(n), r=r, family=family, layout="uniform")
    if op == "grad":
        precision = rng.choice(["fp64", "emu", "emu"])
        n = _log_uniform(rng, 4096, {"fp64": 30000, "emu": 200000}[precision])
        return dict(op=op, precision=precision, n=n, M=_levels(n), r=r, family=family, layout="uniform",
                    torch=rng.random() < 0.5)
    if op == "predict":
        n = _log_uniform(rng, 4096, 200000)
        return dict(op=op, precision=rng.choice(["fp64", "emu"]), n=n, M=_levels(n), r=r, family=family,
                    layout="uniform", points=_log_uniform(rng, 512, 200000), host=rng.random() < 0.5)
    if op == "refresh":
        n = _log_uniform(rng, 10000, 200000)
        return dict(op=op, precision="emu", n=n, M=_levels(n, 32.0) + 1, r=rng.choice([16, 25, 32]), family="exp",
                    layout="swath")
    n = _log_uniform(rng, 5000, 20000)
    return dict(op=op, precision=rng.choice(["emu", "emu", "fp64"]), ndata=rng.randint(4, 12), n=n,
                n_max=rng.randint(2 * n, 120000), r=rng.choice([16, 25, 32]), family="exp", layout="swath")


# ---- inputs --------------------------------------------------------------------
def _generator(seed: int) -> torch.Generator:
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _swath_locations(g, n: int) -> torch.Tensor:
    """n points on 24 parallel strips of width 0.02 at a common angle, 30 % of the strips dropped."""
    th = float(_rand(g, 1)) * math.pi
    u = torch.tensor([math.cos(th), math.sin(th)], device=DEV, dtype=torch.float64)
    v = torch.tensor([-math.sin(th), math.cos(th)], device=DEV, dtype=torch.float64)
    lo = min(0.0, float(v[0])) + min(0.0, float(v[1]))
    hi = max(0.0, float(v[0])) + max(0.0, float(v[1]))
    centres = lo + (hi - lo) * (torch.arange(24, device=DEV) + 0.2 + 0.6 * _rand(g, 24)) / 24
    order = torch.argsort(_rand(g, 24))
    centres = centres[order[:17]]
    # strips weighted by the length of their centre line inside the square
    t = torch.linspace(-1.5, 1.5, 3001, device=DEV, dtype=torch.float64)
    line = centres[:, None, None] * v + t[None, :, None] * u
    length = ((line >= 0) & (line <= 1)).all(2).double().sum(1) + 1e-9
    parts, have = [], 0
    while have < n:
        k = 6 * (n - have) + 1024
        c = centres[torch.multinomial(length, k, replacement=True, generator=g)]
        p = (c + 0.02 * (_rand(g, k) - 0.5))[:, None] * v + (3.0 * _rand(g, k) - 1.5)[:, None] * u
        p = p[((p >= 0) & (p <= 1)).all(1)]
        parts.append(p)
        have += p.shape[0]
    return torch.cat(parts)[:n].contiguous()


def _field(g, locs: torch.Tensor, nu: float, kappa: float, features: int = 256) -> torch.Tensor:
    """Random-Fourier-feature draw of the unit-variance Matern-nu field (2 nu an odd integer)."""
    z = torch.randn(features, 2, generator=g, device=DEV, dtype=torch.float64)
    chi = torch.randn(features, int(2 * nu), generator=g, device=DEV, dtype=torch.float64).square().sum(1)
    w = z / (kappa * torch.sqrt(chi / (2.0 * nu)))[:, None]
    b = 2.0 * math.pi * _rand(g, features)
    out = torch.empty(locs.shape[0], device=DEV, dtype=torch.float64)
    for i in range(0, locs.shape[0], 1 << 18):
        out[i:i + (1 << 18)] = torch.cos(locs[i:i + (1 << 18)] @ w.T + b).sum(1)
    return out * math.sqrt(2.0 / features)


def _dataset(n: int, family: str, layout: str, g, kappa: float, tau2: float, nonstat: bool):
    locs = _rand(g, n, 2) if layout == "uniform" else _swath_locations(g, n)
    f = _field(g, locs, 0.5 if family == "exp" else 1.5, kappa)
    if nonstat:
        f = f * torch.sqrt(1.0 + 0.5 * torch.sin(4.0 * math.pi * locs[:, 0]))
    y = f + math.sqrt(tau2) * torch.randn(n, generator=g, device=DEV, dtype=torch.float64)
    return locs.contiguous(), y.contiguous()


def _theta(g, family: str):
    """(sigma2, range, tau2): the values an optimiser passes through near the truth."""
    base = (1.0, 0.05, 0.05) if family == "exp" else (1.0, 0.1, 0.01)
    u = _rand(g, 3).cpu().numpy()
    return tuple(b * float(1.0 + 0.1 * (x - 0.5)) for b, x in zip(base, u))


def _inputs(case: dict, seed: int) -> dict:
    """Everything a case is computed from, made from the seed alone."""
    g = _generator(seed)
    fam, layout = case["family"], case["layout"]
    nonstat = case["op"] == "refresh"
    kappa, tau2 = (0.05, 0.05) if fam == "exp" else (0.1, 0.01)
    if case["op"] == "batch":
        sets = []
        for k in range(case["ndata"]):
            # sizes spread evenly over the logarithm, so that the work does not hang on the seed
            n = int(case["n"] * (case["n_max"] / case["n"]) ** (k / max(1, case["ndata"] - 1)))
            kap = 0.02 + 0.28 * float(_rand(g, 1))
            locs, y = _dataset(n, fam, layout, g, kap, tau2, False)
            sets.append(dict(locs=locs, y=y, theta=(1.0, kap, tau2), M=_fit_levels(locs)))
        return dict(sets=sets)
    locs, y = _dataset(case["n"], fam, layout, g, kappa, tau2, nonstat)
    out = dict(locs=locs, y=y, theta=_theta(g, fam), nonstat=nonstat)
    if case["op"] == "predict":
        side = math.isqrt(case["points"])
        if side * side == case["points"]:        # a square number of points: the cell-centred grid of a map
            c = (torch.arange(side, device=DEV, dtype=torch.float64) + 0.5) / side
            yy, xx = torch.meshgrid(c, c, indexing="ij")
            out["points"] = torch.stack([xx.reshape(-1), yy.reshape(-1)], 1).contiguous()
        else:
            out["points"] = _rand(g, case["points"], 2)
    return out


def _cells(locs: torch.Tensor, M: int) -> torch.Tensor:
    """Morton ids of the level-M quadtree cells (child digit b_x + 2 b_y)."""
    ij = torch.clamp((locs * (1 << M)).floor().long(), 0, (1 << M) - 1)
    out = torch.zeros(locs.shape[0], dtype=torch.long, device=locs.device)
    for b in range(M):
        out |= ((ij[:, 0] >> b) & 1) << (2 * b)
        out |= ((ij[:, 1] >> b) & 1) << (2 * b + 1)
    return out


def _fit_levels(locs: torch.Tensor, most: int = 64) -> int:
    """The fewest quadtree levels whose leaves hold at most ``most`` observations."""
    for M in range(1, 11):
        if int(torch.bincount(_cells(locs, M)).max()) <= most:
            return M
    raise ValueError("no quadtree of at most 10 levels fits")


# ---- prepare and run -----------------------------------------------------------
def prepare(case: dict, seed: int) -> dict:
    x = _inputs(case, seed)
    op = case["op"]
    if op == "batch":
        sets = [dict(locs=s["locs"].cpu().numpy(), y=s["y"].cpu().numpy(), M=s["M"], family=case["family"])
                for s in x["sets"]]
        b = mra.Batch(sets, r=case["r"], precision=case["precision"])
        thetas = [s["theta"] for s in x["sets"]]
        b.loglik(thetas)                         # a user's first call tunes the tiles and captures the launches
        return dict(op=op, handle=b, theta=thetas)
    kw = dict(M=case["M"], r=case["r"], family=case["family"], precision=case["precision"], nonstat=x["nonstat"])
    st = dict(op=op, theta=x["theta"])
    if op == "refresh":
        # the kept handle was built on the same swaths' earlier pass; today's data arrive on the host
        st["locs"], st["y"] = x["locs"].cpu().numpy(), x["y"].cpu().numpy()
        st["handle"] = mra.Handle(x["locs"], x["y"], prune=True, **kw)
        return st
    st["handle"] = mra.Handle(x["locs"], x["y"], **kw)
    if op == "grad":
        st["torch"] = case["torch"]
    if op == "predict":
        st["handle"].loglik(x["theta"])          # the fit the predictions condition on
        st["points"] = x["points"].cpu().numpy() if case["host"] else x["points"]
    return st


def run(state: dict):
    h, op = state["handle"], state["op"]
    if op == "batch":
        return h.loglik(state["theta"])
    if op == "loglik":
        return np.float64(h.loglik(state["theta"]))      # (all 64 bits of the Python float)
    if op == "refresh":
        h.update(state["locs"], state["y"])
        return np.float64(h.loglik(state["theta"]))
    if op == "predict":
        return h.predict(state["theta"], state["points"])
    if state["torch"]:
        theta = torch.tensor(state["theta"], dtype=torch.float64, requires_grad=True)
        ll = autograd.loglik(h, theta)
        ll.backward()
        return ll.detach(), theta.grad
    ll, grad = h.loglik_grad(state["theta"])
    return np.float64(ll), grad


# ---- the work a case cannot do without -----------------------------------------
def _tree_counts(case: dict, locs, M: int):
    """Regions with data per level (complete trees: all of them) and the leaves' occupancies."""
    occ = torch.bincount(_cells(locs, M), minlength=4 ** M).double()
    pruned = case["op"] in ("refresh", "batch")
    nreg = []
    for m in range(M + 1):
        per = occ.reshape(4 ** m, -1).sum(1)
        nreg.append(int((per > 0).sum()) if pruned else 4 ** m)
    return nreg, occ


def _forward_flops(nreg, occ, M: int, r: int) -> float:
    """Multiply-adds (2) of one evaluation; symmetric and triangular products once."""
    f = 0.0
    for m in range(M):
        prior = sum(2.0 * r * r * l * r + r * r * (r + 1) for l in range(m)) + r * (r + 1) * m * r + 2.0 * r ** 3 / 3
        post = 2.0 * r ** 3 / 3 + m * r * r * (r + 1) + r * (r + 1)
        f += nreg[m] * (prior + post)
        if m > 0:
            f += nreg[m] * (m * r) * (m * r + 1) * r + 2.0 * m * r * r * nreg[m]
    c1, c2, c3 = (float(occ.pow(k).sum()) for k in (1, 2, 3))
    Mr = M * r
    chain = sum(2.0 * r * l * r + r * (r + 1) for l in range(M))
    f += c1 * (chain + Mr * (Mr + 1) + 2.0 * Mr) + (c2 + c1) * 2.0 * Mr + 2.0 * c3 / 3 + c2
    return f


def work(case: dict) -> dict:
    x = _inputs(case, 0)
    if case["op"] == "batch":
        flops = size = 0.0
        for s in x["sets"]:
            nreg, occ = _tree_counts(case, s["locs"], s["M"])
            flops += _forward_flops(nreg, occ, s["M"], case["r"])
            size += 24.0 * s["locs"].shape[0] + 8.0
        return dict(bytes=size, flops=flops)
    M, r, n = case["M"], case["r"], case["n"]
    nreg, occ = _tree_counts(case, x["locs"], M)
    fwd = _forward_flops(nreg, occ, M, r)
    if case["op"] == "grad":                     # the adjoint of a product is two products
        return dict(bytes=24.0 * n + 32.0, flops=3.0 * fwd)
    if case["op"] == "predict":
        p = case["points"]
        c = n / 4.0 ** M                         # chain, leaf covariance row and its solve, posterior recursion
        per = sum(2.0 * r * l * r + r * (r + 1) for l in range(M)) + 4.0 * c * M * r + c * c
        per += sum(r * (r + 1) + 2.0 * m * r * r for m in range(M)) + 4.0 * M * r
        # the factors are read from where the fit left them: V, L^{-1}, Lt^{-1}, G of every level, H and L_Sigma^{-1}
        factors = sum(nreg[m] * (2.0 * m * r * r + 2.0 * r * r) for m in range(M)) + n * (M * r + 1.0) + \
            float(occ.pow(2).sum())
        return dict(bytes=8.0 * (4.0 * p + factors), flops=p * per)
    return dict(bytes=24.0 * n + 8.0, flops=fwd)


# ---- the same quantities in plain FP64 torch -----------------------------------
def _cov(theta, family: str, nonstat: bool, a: torch.Tensor, b: torch.Tensor) -> torch.Tensor:
    """C0 between batches of points (..., p, 2) and (..., q, 2)."""
    s2, kappa = theta[0], theta[1]
    d2 = (a[..., :, None, :] - b[..., None, :, :]).square().sum(-1)
    same = d2 == 0
    h = torch.where(same, torch.zeros_like(d2), torch.sqrt(torch.where(same, torch.ones_like(d2), d2)))
    if family == "exp":
        c = s2 * torch.exp(-h / kappa)
    else:
        t = math.sqrt(3.0) * h / kappa
        c = s2 * (1.0 + t) * torch.exp(-t)
    if nonstat:
        va = torch.sqrt(1.0 + 0.5 * torch.sin(4.0 * math.pi * a[..., 0]))
        vb = torch.sqrt(1.0 + 0.5 * torch.sin(4.0 * math.pi * b[..., 0]))
        c = c * va[..., :, None] * vb[..., None, :]
    return c


def _knots(ids: torch.Tensor, m: int, r: int) -> torch.Tensor:
    """The cell-centred gx x gy knots of the level-m regions ``ids`` (gx the smallest divisor of r with gx^2 >= r)."""
    gx = next(d for d in range(1, r + 1) if r % d == 0 and d * d >= r)
    gy = r // gx
    ix, iy = torch.zeros_like(ids), torch.zeros_like(ids)
    for b in range(m):
        ix |= ((ids >> (2 * b)) & 1) << b
        iy |= ((ids >> (2 * b + 1)) & 1) << b
    w = 0.5 ** m
    q = torch.arange(r, device=ids.device)
    x = (ix[:, None] + ((q % gx).double() + 0.5) / gx) * w
    y = (iy[:, None] + ((q // gx).double() + 0.5) / gy) * w
    return torch.stack([x, y], 2)


def _rows(key: torch.Tensor, ids: torch.Tensor):
    """Items grouped by their region: (regions, most) indexes into the items, and which of them are real."""
    order = torch.argsort(key, stable=True)
    counts = torch.bincount(torch.searchsorted(ids, key), minlength=len(ids))
    most = max(1, int(counts.max()))
    start = torch.cumsum(counts, 0) - counts
    k = torch.arange(most, device=key.device)
    real = k[None, :] < counts[:, None]
    at = torch.where(real, start[:, None] + k[None, :], torch.zeros_like(start)[:, None])
    return order[at], real


class _Exact:
    """Sec. 3's recursions in block-Cholesky form over the quadtree's regions, level by level."""

    def __init__(self, locs, M, r, family, nonstat, complete):
        self.locs, self.M, self.r, self.family, self.nonstat = locs, M, r, family, nonstat
        leaf = _cells(locs, M)
        self.ids = []
        for m in range(M + 1):
            if complete:
                self.ids.append(torch.arange(4 ** m, device=DEV))
            else:
                self.ids.append(torch.unique(leaf >> (2 * (M - m))))
        self.par = [None] + [torch.searchsorted(self.ids[m - 1], self.ids[m] >> 2) for m in range(1, M + 1)]
        self.rows, self.real = _rows(leaf, self.ids[M])

    def _up(self, m, at, l):
        for t in range(m, l, -1):
            at = self.par[t][at]
        return at

    def _chain(self, theta, pts, m, at):
        """[V^0 .. V^{m-1}] of batches of points whose level-m regions are ``at``."""
        blocks = []
        for l in range(m):
            a = self._up(m, at, l)
            x = _cov(theta, self.family, self.nonstat, pts, self.Q[l][a])
            if l:
                x = x - torch.cat(blocks, 2) @ self.V[l][a].transpose(1, 2)
            blocks.append(torch.linalg.solve_triangular(self.L[l][a], x.transpose(1, 2), upper=False).transpose(1, 2))
        return torch.cat(blocks, 2) if blocks else pts.new_zeros(pts.shape[0], pts.shape[1], 0)

    def prior(self, theta):
        self.Q = [_knots(self.ids[m], m, self.r) for m in range(self.M)]
        self.V, self.L = [], []
        for m in range(self.M):
            at = torch.arange(len(self.ids[m]), device=DEV)
            v = self._chain(theta, self.Q[m], m, at)
            w = _cov(theta, self.family, self.nonstat, self.Q[m], self.Q[m]) - v @ v.transpose(1, 2)
            self.V.append(v)
            self.L.append(torch.linalg.cholesky(w))

    def _leaf(self, theta, y, at):
        """Leaves ``at``: V_F, the factor of Sigma_F, L_Sigma^{-1} V_F, L_Sigma^{-1} y, points, mask (padded rows zero)."""
        most = max(1, int(self.real[at].sum(1).max()))
        rows, real = self.rows[at][:, :most], self.real[at][:, :most]
        pts, mask = self.locs[rows], real.double()
        v = self._chain(theta, pts, self.M, at) * mask[:, :, None]
        s = _cov(theta, self.family, self.nonstat, pts, pts) * (mask[:, :, None] * mask[:, None, :])
        s = s - v @ v.transpose(1, 2) + torch.diag_embed(theta[2] * mask + (1.0 - mask))
        ls = torch.linalg.cholesky(s)
        hz = torch.linalg.solve_triangular(ls, torch.cat([v, (y[rows] * mask)[:, :, None]], 2), upper=False)
        return v, ls, hz[:, :, :-1], hz[:, :, -1:], pts, mask

    def loglik(self, theta, y, chunk: int = 1 << 30):
        M, r = self.M, self.r
        self.prior(theta)
        npar = len(self.ids[M - 1])
        A = torch.zeros(npar, M * r, M * r, device=DEV, dtype=torch.float64)
        om = torch.zeros(npar, M * r, 1, device=DEV, dtype=torch.float64)
        d = u = torch.zeros((), device=DEV, dtype=torch.float64)
        for c0 in range(0, len(self.ids[M]), chunk):
            at = torch.arange(c0, min(len(self.ids[M]), c0 + chunk), device=DEV)
            _, ls, h, z, _, mask = self._leaf(theta, y, at)
            d = d + 2.0 * (torch.log(torch.diagonal(ls, dim1=1, dim2=2)) * mask).sum()
            u = u + z.square().sum()
            ht = h.transpose(1, 2)
            A = A.index_add(0, self.par[M][at], ht @ h) if theta.requires_grad else \
                A.index_add_(0, self.par[M][at], ht @ h)
            om = om.index_add(0, self.par[M][at], ht @ z)
        self.Lt, self.G, self.g = [None] * M, [None] * M, [None] * M
        eye = torch.eye(r, device=DEV, dtype=torch.float64)
        for m in range(M - 1, -1, -1):
            k = m * r
            lt = torch.linalg.cholesky(A[:, k:, k:] + eye)
            gg = torch.linalg.solve_triangular(lt, torch.cat([A[:, k:, :k], om[:, k:]], 2), upper=False)
            G, g = gg[:, :, :k], gg[:, :, k:]
            self.Lt[m], self.G[m], self.g[m] = lt, G, g
            d = d + 2.0 * torch.log(torch.diagonal(lt, dim1=1, dim2=2)).sum()
            u = u - g.square().sum()
            if m:
                up = len(self.ids[m - 1])
                Gt = G.transpose(1, 2)
                A2 = torch.zeros(up, k, k, device=DEV, dtype=torch.float64)
                A = A2.index_add(0, self.par[m], A[:, :k, :k] - Gt @ G)
                o2 = torch.zeros(up, k, 1, device=DEV, dtype=torch.float64)
                om = o2.index_add(0, self.par[m], om[:, :k] - Gt @ g)
        return -0.5 * (d + u) - 0.5 * self.locs.shape[0] * math.log(2.0 * math.pi)

    def predict(self, theta, y, plocs, chunk: int):
        """Kriging means and variances after ``loglik`` at the same theta (Prop. 2)."""
        M, r = self.M, self.r
        prow, preal = _rows(_cells(plocs, M), self.ids[M])
        mean, var = torch.empty(len(plocs), device=DEV).double(), torch.empty(len(plocs), device=DEV).double()
        for c0 in range(0, len(self.ids[M]), chunk):
            at = torch.arange(c0, min(len(self.ids[M]), c0 + chunk), device=DEV)
            v, ls, h, z, pts, mask = self._leaf(theta, y, at)
            most = int(preal[at].sum(1).max())
            if most == 0:
                continue
            pr, real = prow[at][:, :most], preal[at][:, :most]
            pp = plocs[pr]
            b = self._chain(theta, pp, M, at)
            cross = (_cov(theta, self.family, self.nonstat, pp, pts) - b @ v.transpose(1, 2)) * mask[:, None, :]
            p = torch.linalg.solve_triangular(ls, cross.transpose(1, 2), upper=False).transpose(1, 2)
            own = theta[0] * torch.ones_like(pp[..., 0])
            if self.nonstat:
                own = own * (1.0 + 0.5 * torch.sin(4.0 * math.pi * pp[..., 0]))
            var_c = own - b.square().sum(2) - p.square().sum(2)
            mean_c = (p @ z)[..., 0]
            b = b - p @ h
            for m in range(M - 1, -1, -1):
                a = self._up(M, at, m)
                w = torch.linalg.solve_triangular(self.Lt[m][a], b[:, :, m * r:].transpose(1, 2), upper=False)
                w = w.transpose(1, 2)
                mean_c = mean_c + (w @ self.g[m][a])[..., 0]
                var_c = var_c + w.square().sum(2)
                b = b[:, :, :m * r] - w @ self.G[m][a]
            mean[pr[real]], var[pr[real]] = mean_c[real], var_c[real]
        return mean, var


def exact(case: dict, seed: int):
    x = _inputs(case, seed)
    op, fam = case["op"], case["family"]
    if op == "batch":
        out = []
        for s in x["sets"]:
            e = _Exact(s["locs"], s["M"], case["r"], fam, False, complete=False)
            th = torch.tensor(s["theta"], dtype=torch.float64, device=DEV)
            out.append(float(e.loglik(th, s["y"], chunk=8192)))
            del e
            torch.cuda.empty_cache()
        return np.array(out)
    e = _Exact(x["locs"], case["M"], case["r"], fam, x["nonstat"], complete=op == "predict")
    th = torch.tensor(x["theta"], dtype=torch.float64, device=DEV)
    if op == "grad":
        th.requires_grad_(True)
        ll = e.loglik(th, x["y"])
        ll.backward()
        if case["torch"]:
            return ll.detach().cpu(), th.grad.cpu()
        return np.float64(ll.detach().cpu()), th.grad.cpu().numpy()
    ll = np.float64(e.loglik(th, x["y"], chunk=4096).cpu())
    if op != "predict":
        return ll
    mean, var = e.predict(th, x["y"], x["points"], chunk=2048)
    return (mean.cpu().numpy(), var.cpu().numpy()) if case["host"] else (mean, var)
