"""The work that a user of this library has it do, as cases to measure.

A case is one pass through the public entry points of
paper_2508_13986_gb300.gbees, from new inputs on the host to results on the
host, in one of three forms:

  filter  an estimation run: the prior as a Gaussian, propagation over one or
          more segments, a measurement update at the end of each (or none),
          then the moments and the density of the result
  tick    one period of a loop that keeps its density as a cell list: load the
          cells, propagate a few time steps, update with a measurement, read
          the moments and the cells back
  batch   independent grids in one launch, each with its own prior and target
          time, then the moments and the density of every grid

A density is read into buffers that the caller keeps (room for as many cells as
half the pool may hold; rows past the count stay 0), as a C program reads it.
The sizes are those of the named workloads (workloads.py) and of the tests:
Lorenz '63 with h = 0.25 and 0.5, the paper's own Lorenz '63 case, Lorenz '96 in
4 and 6 dimensions, linear drift in 1 to 5 dimensions, both storage precisions.
A density is read in sorted order (the default of read_cells), except those of
millions of cells, which end with an update and are read in storage order: the
update's prune leaves a pool of that size in key order.
"""
import math

import numpy as np
import torch

from paper_2508_13986_gb300 import gbees

L63 = (10.0, 28.0, 8.0 / 3.0)
DYN = {"constant": gbees.GBEES_DYN_CONSTANT, "linear": gbees.GBEES_DYN_LINEAR, "l63": gbees.GBEES_DYN_LORENZ63,
       "l63s": gbees.GBEES_DYN_LORENZ63_SHIFTED, "l96": gbees.GBEES_DYN_LORENZ96}


def case(form, dyn, n, h, sigma, t_end, thr, cap, f32=False, segments=1, measured=0, r=0.25, cfl=0.9, corr=0.0,
         grids=1, whole_order=True):
    """measured: components seen by each update (0: no update); r: variance of a
    measurement; corr: largest correlation of the prior; cap: pool capacity;
    whole_order: read the density sorted."""
    return {"form": form, "dyn": dyn, "n": n, "h": h, "sigma": sigma, "t_end": t_end, "thr": thr, "cap": cap,
            "f32": f32, "segments": segments, "measured": measured, "r": r, "cfl": cfl, "corr": corr,
            "grids": grids, "sorted": whole_order}


def listed():
    named = [
        # the smallest calls: a real-time loop's period on about 10^3 cells, a few time steps
        ("tick_l63", case("tick", "l63", 3, 0.5, 0.5, 0.02, 1e-3, 1 << 14, measured=1)),
        # lorenz63_h0.5: one prediction of about 10^4 cells, no measurement
        ("l63_h0.5", case("filter", "l63", 3, 0.5, 1.0, 0.5, 1e-7, 1 << 17)),
        # lorenz63_h0.25: the filter with full-state measurements every 0.25, in both precisions
        ("l63_h0.25_filter", case("filter", "l63", 3, 0.25, 1.0, 1.0, 1e-7, 1 << 19, segments=4, measured=3)),
        ("l63_h0.25_filter_f32", case("filter", "l63", 3, 0.25, 1.0, 1.0, 1e-7, 1 << 19, f32=True, segments=4,
                                      measured=3)),
        # the paper's Lorenz '63 case: shifted form, one component measured in the middle and at the end
        ("paper_e1", case("filter", "l63s", 3, 0.5, 1.0, 2.0, 1e-3, 1 << 17, segments=2, measured=1, r=1.0, cfl=1.0)),
        # a linear model of two states on a fine grid with a correlated prior
        ("linear_2d", case("filter", "linear", 2, 0.01, 0.25, 0.2, 1e-6, 1 << 19, segments=2, measured=1, r=0.04,
                           corr=0.4)),
        # Lorenz '96 in four dimensions: the pool outgrows the small-grid launch mode on the way
        ("l96_4d", case("filter", "l96", 4, 0.25, 0.5, 0.3, 1e-6, 1 << 22, segments=2, measured=2, corr=0.3)),
        # a served 6-D request: the serving stream's width, horizon and corrections
        ("l96_6d_h0.5", case("filter", "l96", 6, 0.5, 0.5, 0.3, 1e-6, 1 << 23, segments=2, measured=6)),
        # the paper's 6-D case (threshold 1e-4, h = half the standard deviation), its first stretch, in both precisions
        ("paper_e2_start_f32", case("filter", "l96", 6, 0.1, 0.2, 0.1, 1e-4, 1 << 24, f32=True, measured=3, r=0.04,
                                    cfl=1.0, whole_order=False)),
        # the benchmark's 6-D grid of 7 * 10^6 cells: one cycle of prediction and update
        ("l96_6d_h0.25", case("filter", "l96", 6, 0.25, 0.5, 0.2, 1e-6, 1 << 25, measured=3, whole_order=False)),
        # ragged Lorenz '63 grids in one launch, as a server's round or an ensemble study runs them
        ("batch_l63_f32", case("batch", "l63", 3, 0.5, 1.0, 0.2, 1e-5, 1 << 17, f32=True, grids=96)),
        ("batch_l63", case("batch", "l63", 3, 0.5, 1.0, 0.2, 1e-5, 1 << 17, grids=24)),
    ]
    return [dict(c, name=name) for name, c in named]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["tick", "l63", "l63", "linear", "l96", "l96", "large", "batch"])
    f32 = rng.random() < 0.4
    if kind == "tick":
        return case("tick", "l63", 3, _log(rng, 0.3, 0.6), rng.uniform(0.4, 0.7), _log(rng, 0.005, 0.05),
                    _log(rng, 1e-4, 1e-2), 1 << 16, f32, measured=rng.randint(1, 3))
    if kind == "l63":
        segments = rng.randint(1, 4)
        shifted = rng.random() < 0.3
        return case("filter", "l63s" if shifted else "l63", 3, _log(rng, 0.25, 0.6), rng.uniform(0.7, 1.1),
                    _log(rng, 0.1, 1.0), _log(rng, 1e-7, 1e-3), 1 << 20, f32, segments,
                    rng.randint(1, 3) if segments > 1 else rng.choice([0, 1]), cfl=rng.choice([0.9, 1.0]),
                    corr=rng.choice([0.0, 0.3]))
    if kind == "linear":
        n = rng.choice([1, 2, 2, 3, 4, 5])
        # cells per standard deviation: 10^3 to 3 * 10^5 cells in the ellipsoid of the prior
        thr = _log(rng, 1e-6, 1e-3)
        per = (_log(rng, 1e3, 3e5) / _ball(n, thr)) ** (1.0 / n)
        per = min(max(per, 2.0), 400.0)
        return case("filter", "linear", n, 0.25 / per, 0.25, min(0.5, _log(rng, 20, 150) * 0.25 / per / n), thr,
                    1 << 21, f32, rng.randint(1, 2), rng.randint(1, n), r=0.04, corr=rng.choice([0.0, 0.4]))
    if kind == "l96":
        n = rng.choice([4, 5, 6])
        h = {4: _log(rng, 0.2, 0.5), 5: _log(rng, 0.35, 0.6), 6: _log(rng, 0.45, 0.6)}[n]
        return case("filter", "l96", n, h, rng.uniform(0.45, 0.55), _log(rng, 0.05, 0.3), 1e-6, 1 << 23, f32,
                    rng.randint(1, 3), rng.randint(1, n), corr=rng.choice([0.0, 0.3]))
    if kind == "large":
        sigma = rng.uniform(0.46, 0.5)
        return case("filter", "l96", 6, _log(rng, 0.25, 0.32), sigma, _log(rng, 0.02, 0.2), 1e-6, 1 << 25, f32,
                    1, rng.randint(1, 6), whole_order=False)
    return case("batch", "l63", 3, _log(rng, 0.45, 0.6), rng.uniform(0.7, 1.0), _log(rng, 0.05, 0.2),
                _log(rng, 1e-5, 1e-3), 1 << 17, f32, grids=int(round(_log(rng, 4, 96))))


# ------------------------------------------------------------------ inputs


def _mean(c, g):
    """A prior mean: the workloads' means, moved by the seed."""
    if c["dyn"] in ("l63", "l63s"):
        if c["form"] == "batch":
            return np.array([g.uniform(-15, 15), g.uniform(-20, 20), g.uniform(5, 40)])
        return np.array([-11.5, -10.0, 9.5]) + g.uniform(-0.25, 0.25, 3)
    if c["dyn"] == "l96":
        m = np.full(c["n"], 4.0)
        m[0] += 0.5 if c["h"] <= 0.1 else 0.01
        return m + g.uniform(-0.02, 0.02, c["n"])
    return g.uniform(-1.0, 1.0, c["n"])


def _cov(c, g):
    n = c["n"]
    s = c["sigma"] * (g.uniform(0.8, 1.2, n) if c["form"] == "batch" else g.uniform(0.97, 1.03, n))
    C = np.eye(n)
    if c["corr"] > 0.0 and n > 1:
        a = g.uniform(-1.0, 1.0, n)
        a *= math.sqrt(c["corr"]) / np.max(np.abs(a))
        C = np.outer(a, a)
        np.fill_diagonal(C, 1.0)
    return C * np.outer(s, s)


def _params(c, g):
    n = c["n"]
    if c["dyn"] == "l63":
        return np.array(L63)
    if c["dyn"] == "l63s":
        return np.array([4.0, 1.0, 48.0])
    if c["dyn"] == "l96":
        return np.array([4.0])
    # a rotating, slowly contracting flow with a constant term
    A = g.uniform(-1.0, 1.0, (n, n))
    A = 0.5 * (A - A.T) * 2.0 - 0.1 * np.eye(n)
    return np.concatenate([A.reshape(-1), g.uniform(-1.0, 1.0, n)])


def _drift(c, params, x):
    """f(x) for x of shape (..., n): numpy arrays or tensors (a list of components is returned)."""
    y = [x[..., k] for k in range(c["n"])]
    n, a = c["n"], [float(v) for v in params]
    if c["dyn"] == "constant":
        return [y[0] * 0 + a[j] for j in range(n)]
    if c["dyn"] == "linear":
        out = []
        for j in range(n):
            s = y[0] * 0
            for k in range(n):
                s = s + a[j * n + k] * y[k]
            out.append(s + a[n * n + j])
        return out
    if c["dyn"] == "l63":
        return [a[0] * (y[1] - y[0]), y[0] * (a[1] - y[2]) - y[1], y[0] * y[1] - a[2] * y[2]]
    if c["dyn"] == "l63s":
        return [a[0] * (y[1] - y[0]), -y[1] - y[0] * y[2], (-a[1] * y[2] + y[0] * y[1]) - a[1] * a[2]]
    return [((y[(j + 1) % n] - y[(j - 2) % n]) * y[(j - 1) % n] - y[j]) + a[0] for j in range(n)]


def _truth(c, params, x, span):
    """The state `span` later (classic RK4)."""
    f = lambda v: np.array(_drift(c, params, v), dtype=np.float64)  # noqa: E731
    k = max(1, int(math.ceil(span / 1e-3)))
    s = span / k
    for _ in range(k):
        k1 = f(x)
        k2 = f(x + 0.5 * s * k1)
        k3 = f(x + 0.5 * s * k2)
        k4 = f(x + s * k3)
        x = x + s / 6.0 * (k1 + 2 * k2 + 2 * k3 + k4)
    return x


def _inputs(c, seed):
    """Everything that the seed decides: priors, measurements, cell lists (host arrays)."""
    g = np.random.default_rng([int(seed), 2508])
    out = {"priors": [], "measurements": [], "cells": None, "t_ends": []}
    for _ in range(c["grids"]):
        out["priors"].append((_mean(c, g), _cov(c, g)))
        out["t_ends"].append(c["t_end"] * (g.uniform(0.5, 1.0) if c["form"] == "batch" else 1.0))
    out["params"] = _params(c, g)
    mean, cov = out["priors"][0]
    if c["measured"]:
        x = mean + 0.5 * np.linalg.cholesky(cov) @ g.standard_normal(c["n"])
        for k in range(c["segments"]):
            x = _truth(c, out["params"], x, c["t_end"] / c["segments"])
            H = np.sort(g.permutation(c["n"])[: c["measured"]]).astype(np.int32)
            y = x[H] + 0.5 * math.sqrt(c["r"]) * g.standard_normal(H.size)
            out["measurements"].append((y, c["r"] * np.eye(H.size), H))
    if c["form"] == "tick":  # a density as the last period left it: a bump of a few cells, a little off its shape
        hw = int(math.ceil(math.sqrt(-2.0 * math.log(c["thr"])) * c["sigma"] * 1.1 / c["h"])) + 1
        axes = np.meshgrid(*[np.arange(-hw, hw + 1)] * c["n"], indexing="ij")
        idx = np.stack([v.reshape(-1) for v in axes], axis=1).astype(np.int32)
        d = idx * c["h"]
        p = np.exp(-0.5 * np.einsum("ia,ab,ib->i", d, np.linalg.inv(cov), d)) * (1.0 + 0.05 * g.random(idx.shape[0]))
        keep = p > c["thr"] * p.max()
        idx, p = np.ascontiguousarray(idx[keep]), p[keep]
        out["cells"] = (idx, p / (p.sum() * c["h"] ** c["n"]))
    return out


def prepare(c, seed):
    s = _inputs(c, seed)
    s["case"] = c
    s["grids"] = []
    for mean, _ in s["priors"]:
        cfg = gbees.make_config(c["n"], DYN[c["dyn"]], s["params"], [c["h"]] * c["n"], mean, c["thr"], c["cfl"],
                                precision=gbees.GBEES_FP32 if c["f32"] else gbees.GBEES_FP64, max_cells=c["cap"])
        s["grids"].append(gbees.Grid(cfg))
    room = (len(s["grids"]), c["cap"] // 2)
    s["idx"], s["p"] = np.zeros((*room, c["n"]), dtype=np.int32), np.zeros(room)
    return s


# ------------------------------------------------------------------ one pass


def _results(s):
    n = s["case"]["n"]
    for k, g in enumerate(s["grids"]):
        rc, _ = gbees.gbees_read_cells(g.ctx, s["idx"][k], s["p"][k], s["case"]["sorted"])
        if rc != 0:
            raise gbees.GbeesError(rc, gbees.gbees_last_error(g.ctx))
    moments = [g.moments() for g in s["grids"]]
    stats = [g.stats() for g in s["grids"]]
    return {"idx": s["idx"].reshape(-1, n), "p": s["p"].reshape(-1),
            "mean": np.stack([m[0] for m in moments]), "cov": np.stack([m[1] for m in moments]),
            "t": np.array([v.t for v in stats]), "steps": np.array([v.total_steps for v in stats]),
            "cells": np.array([v.n_cells for v in stats])}


def run(s):
    c, grids = s["case"], s["grids"]
    if c["form"] == "batch":
        for g, (mean, cov) in zip(grids, s["priors"]):
            g.init_gaussian(mean, cov)
        gbees.propagate_batch(grids, s["t_ends"])
        return _results(s)
    g = grids[0]
    if c["form"] == "tick":
        g.init_cells(*s["cells"])
    else:
        g.init_gaussian(*s["priors"][0])
    for k in range(c["segments"]):
        g.propagate(c["t_end"] * (k + 1) / c["segments"])
        if s["measurements"]:
            g.correct_gaussian(*s["measurements"][k])
    return _results(s)


# ------------------------------------------------------------------ its least work


def _ball(n, thr):
    """Cells of the prior's set where a standard deviation is one cell wide."""
    return math.pi ** (n / 2) / math.gamma(n / 2 + 1) * (-2.0 * math.log(thr)) ** (n / 2)


def work(c):
    """A time step reads and writes the density of its cells once, and takes
    per cell and dimension: the donor flux 3, the transverse sums 6, the limited
    term 8, the conservative update 3 operations. Steps from the CFL rate of the
    prior's set, cells from its volume (neither from a run)."""
    g = np.random.default_rng(0)
    n = c["n"]
    params, mean, r = _params(c, g), _mean(dict(c, form="filter"), g), math.sqrt(-2.0 * math.log(c["thr"]))
    corners = mean + r * c["sigma"] * np.concatenate([np.eye(n), -np.eye(n)])
    rate = max(sum(abs(float(v)) for v in _drift(c, params, x)) / c["h"] for x in corners)
    t = c["t_end"] * (0.75 if c["form"] == "batch" else 1.0)
    steps = max(1.0, t * rate / c["cfl"])
    cells = max(1.0, _ball(n, c["thr"]) * (c["sigma"] / c["h"]) ** n) * c["grids"]
    S = 4 if c["f32"] else 8
    return {"bytes": cells * steps * 2 * S + cells * (4 * n + 8), "flops": cells * steps * 20 * n}


# ------------------------------------------------------------------ the method in plain 64-bit tensors


class _Plain:
    """One grid as sorted packed keys and densities; every step of the method as
    whole-tensor operations on the pool of active cells and their neighbours."""

    def __init__(self, c, params, origin, device):
        self.c, self.params, self.n, self.h, self.dev = c, params, c["n"], c["h"], device
        self.bits = 63 // self.n if self.n > 1 else 32
        self.x0 = torch.tensor(origin, dtype=torch.float64, device=device)
        self.unit = [1 << (self.bits * (self.n - 1 - j)) for j in range(self.n)]
        self.t, self.steps = 0.0, 0

    def pack(self, idx):
        k = torch.zeros(idx.shape[0], dtype=torch.int64, device=self.dev)
        for j in range(self.n):
            k = k * (1 << self.bits) + (idx[:, j].to(torch.int64) + (1 << (self.bits - 1)))
        return k

    def unpack(self, k):
        mask, half = (1 << self.bits) - 1, 1 << (self.bits - 1)
        return torch.stack([((k >> (self.bits * (self.n - 1 - j))) & mask) - half for j in range(self.n)], dim=1)

    def start(self, key, p):
        order = torch.argsort(key)
        self.key, self.p = key[order], p[order]

    def gaussian(self, mean, cov):
        n, icov = self.n, np.linalg.inv(cov)
        thr, ax = self.c["thr"], []
        for k in range(n):
            hw = int(math.ceil(math.sqrt(-2.0 * math.log(thr) * cov[k, k]) / self.h)) + 2
            ax.append(torch.arange(-hw, hw + 1, device=self.dev))
        keys, ps = [], []
        for i0 in ax[0]:  # a slab at a time
            idx = torch.cartesian_prod(i0.reshape(1), *ax[1:]).reshape(-1, n)
            d = self.x0 + idx.to(torch.float64) * self.h - torch.tensor(mean, device=self.dev)
            q = torch.zeros(idx.shape[0], dtype=torch.float64, device=self.dev)
            for a in range(n):
                for b in range(n):
                    if icov[a, b] != 0.0:
                        q = q + d[:, a] * float(icov[a, b]) * d[:, b]
            p = torch.exp(-0.5 * q)
            keep = p > 0.5 * thr
            keys.append(self.pack(idx[keep]))
            ps.append(p[keep])
        key, p = torch.cat(keys), torch.cat(ps)
        keep = p > thr * p.max()
        self.start(key[keep], p[keep])
        self.normalise()

    def normalise(self):
        self.p = self.p / (self.p.sum() * self.h ** self.n)

    def find(self, table, key):
        at = torch.searchsorted(table, key).clamp_(max=table.numel() - 1)
        return torch.where(table[at] == key, at, -1)

    def velocity(self, idx, j, up):
        """f_j at the lower (up = 0) or upper face of the cells in dimension j."""
        x = self.x0 + idx.to(torch.float64) * self.h
        x[:, j] = self.x0[j] + (idx[:, j].to(torch.float64) + (up - 0.5)) * self.h
        return _drift(self.c, self.params, x)[j]

    def downwind(self, key):
        """The cells that the flow leaves `key` towards: faces, and edges of two such faces."""
        idx, out, got = self.unpack(key), [], []
        for j in range(self.n):
            out += [(j, -self.unit[j], self.velocity(idx, j, 0) < 0), (j, self.unit[j], self.velocity(idx, j, 1) > 0)]
        for i, (j, s, a) in enumerate(out):
            got.append(key[a] + s)
            for k, z, b in out[i + 1:]:
                if k != j:
                    got.append(key[a & b] + (s + z))
        return torch.unique(torch.cat(got))

    def significant(self):
        return self.p > self.c["thr"] * self.p.max()

    def step(self, target):
        n, h = self.n, self.h
        key = torch.unique(torch.cat([self.key, self.downwind(self.key[self.significant()])]))
        p = torch.zeros(key.numel(), dtype=torch.float64, device=self.dev)
        p[torch.searchsorted(key, self.key)] = self.p
        idx = self.unpack(key)
        rate = sum(self.velocity(idx, j, 0).abs() / h for j in range(n))
        fastest = float(rate.max())
        dt = self.c["cfl"] / fastest if fastest > 0 else math.inf
        last = dt >= target - self.t
        dt = target - self.t if last else dt
        del idx, rate
        # the pool: active cells and their face neighbours (density 0), an absent cell at its end
        pool = torch.unique(torch.cat([key] + [key + s * self.unit[j] for j in range(n) for s in (-1, 1)]))
        P = torch.zeros(pool.numel() + 1, dtype=torch.float64, device=self.dev)
        mine = torch.searchsorted(pool, key)
        P[mine] = p
        pidx = self.unpack(pool)
        dn = [self.find(pool, pool - self.unit[j]) for j in range(n)]
        up = [self.find(pool, pool + self.unit[j]) for j in range(n)]
        u = [self.velocity(pidx, j, 0) for j in range(n)]
        G, total = [], 0.0
        for d in range(n):
            hi = self.velocity(pidx, d, 1)
            G.append((u[d].clamp(min=0) * (P[:-1] - P[dn[d]]) + hi.clamp(max=0) * (P[up[d]] - P[:-1])) / (2 * h))
            total = total + G[d]
        del pidx
        absent = torch.zeros(1, dtype=torch.float64, device=self.dev)
        new = p
        for j in range(n):
            S = torch.cat([total - G[j], absent])
            W = torch.cat([P[:-1] - P[dn[j]], absent])  # jump across the lower face
            fwd = u[j] > 0
            f = u[j] * torch.where(fwd, P[dn[j]] - dt * S[dn[j]], P[:-1] - dt * S[:-1])
            Wu, w = torch.where(fwd, W[dn[j]], P[up[j]] - P[:-1]), W[:-1]
            lim = torch.minimum(torch.minimum(0.5 * (w + Wu).abs(), 2 * w.abs()), 2 * Wu.abs())
            lim = torch.where(w * Wu > 0, torch.sign(w) * lim, torch.zeros_like(lim))
            # a face that touches no active cell is not one of the method's: only active cells read fluxes
            f = f + 0.5 * u[j].abs() * (1.0 - dt / h * u[j].abs()) * lim
            F = torch.cat([f, absent])
            new = new - dt / h * (F[up[j]][mine] - F[mine])
        self.key, self.p = key, new
        self.t = target if last else self.t + dt
        self.steps += 1
        if not last and not self.t < target:
            self.t, last = target, True
        if self.steps % 20 == 0:
            self.prune()
        self.normalise()
        return last

    def prune(self):
        S = self.significant()
        keep = S | (self.find(self.downwind(self.key[S]), self.key) >= 0)
        self.key, self.p = self.key[keep], self.p[keep]

    def propagate(self, target):
        while self.t < target and not self.step(target):
            pass

    def update(self, y, R, H):
        x = self.x0 + self.unpack(self.key).to(torch.float64) * self.h
        r = torch.tensor(y, device=self.dev) - x[:, torch.tensor(H, dtype=torch.int64, device=self.dev)]
        self.p = self.p * torch.exp(-0.5 * ((r @ torch.tensor(np.linalg.inv(R), device=self.dev)) * r).sum(1))
        self.prune()
        self.normalise()

    def moments(self):
        x = self.x0 + self.unpack(self.key).to(torch.float64) * self.h
        w = (self.p * self.h ** self.n)[:, None]
        mean = (x * w).sum(0)
        return mean.cpu().numpy(), (((x - mean) * w).T @ (x - mean)).cpu().numpy()


def exact(c, seed):
    """run()'s results by _Plain. With densities stored in 32 bits a cell at the
    threshold may fall on the other side: the moments alone have a value then."""
    s, dev = _inputs(c, seed), "cuda:0" if torch.cuda.is_available() else "cpu"
    if work(c)["flops"] > 8e9 and c["grids"] == 1:
        return None  # over about 20 seconds
    plain = []
    for i, (mean, cov) in enumerate(s["priors"]):
        if c["grids"] > 24:
            return None
        g = _Plain(c, s["params"], mean, dev)
        if c["form"] == "tick":
            g.start(g.pack(torch.tensor(s["cells"][0], device=dev)), torch.tensor(s["cells"][1], device=dev))
        else:
            g.gaussian(mean, cov)
        for k in range(c["segments"]):
            g.propagate(s["t_ends"][i] * (k + 1) / c["segments"])
            if s["measurements"]:
                g.update(*s["measurements"][k])
        plain.append(g)
    m = [g.moments() for g in plain]
    p = np.zeros((len(plain), c["cap"] // 2))
    for k, g in enumerate(plain):
        p[k, : g.p.numel()] = g.p.cpu().numpy()
    return {"idx": None, "p": None if c["f32"] else p.reshape(-1), "mean": np.stack([v[0] for v in m]),
            "cov": np.stack([v[1] for v in m]), "t": None, "steps": None, "cells": None}
