"""The work users of this library have it do, as cases that can be timed and checked.

Each case is a dict with a "kind":
  simulate   one market of M outer paths: factors, exposures, inner defaults, targets; with
             "regress" the least squares of every date and portfolio on top (one batched step)
  regress    least squares [1, Y] at one date, on arrays the user already has
  lsq        least squares of every date of a simulated market
  alive      least squares on (default indicators, state) over the M N hierarchical sample
  fit        the NN+ network trained at one date (Algorithm 1)
  learn      the NN+ network learnt backwards over every date (Algorithm 2)
  adjoint    CVA_0 and its sensitivities through torch.autograd
  nested     nested Monte Carlo reference of the conditional CVA at the middle date

Everything random follows from (case, seed): the model, the trades, the simulation's key and the
network's initial weights. exact() states the same quantities in 64 bits with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2211_17005_gb300 import api, workload

BOOKS = {1: (500,), 4: (20, 60, 150, 300), 6: (50, 120, 300, 500, 1000, 2000)}


def listed():
    return [
        # the smallest market: one economy, two constant hazards, quadratic least squares; launches count
        {"name": "small_step", "kind": "simulate", "model": "small", "M": 16384, "N": 8, "n": 50, "S": 1,
         "books": 1, "regress": "poly2"},
        # the paper's market (10 economies, 8 counterparties, 500 swaps) on the benchmark's grid
        {"name": "paper_sim", "kind": "simulate", "model": "paper", "M": 131072, "N": 64, "n": 100, "S": 1,
         "books": 1, "regress": ""},
        # the paper's own accuracy setting: 25 Euler sub-steps a date, few paths, many inner draws
        {"name": "paper_fine_grid", "kind": "simulate", "model": "paper", "M": 32768, "N": 1024, "n": 100, "S": 25,
         "books": 1, "regress": ""},
        # six uneven portfolios on one market, tile shapes tuned, every date regressed
        {"name": "six_books_step", "kind": "simulate", "model": "paper", "M": 262144, "N": 256, "n": 120, "S": 1,
         "books": 6, "regress": "linear"},
        # a market of no compiled shape, a ragged number of paths: the run-time-shape kernels
        {"name": "mixed_step", "kind": "simulate", "model": "mixed", "M": 20011, "N": 50, "n": 40, "S": 1,
         "books": 4, "regress": "linear"},
        # one date's fit on the user's own arrays, odd length
        {"name": "regress_one_date", "kind": "regress", "M": 100003, "F": 27},
        # every date's linear fit of the paper's market
        {"name": "lsq_all_dates", "kind": "lsq", "model": "paper", "M": 131072, "N": 64, "n": 100},
        # the learner on (default indicators, state): 8.4M rows a date
        {"name": "alive_all_dates", "kind": "alive", "model": "paper", "M": 131072, "N": 64, "n": 100},
        # Algorithm 2 with the 64-wide network over the paper's 99 dates (the benchmark's step)
        {"name": "learn_64", "kind": "learn", "model": "paper", "M": 131072, "N": 64, "n": 100, "hidden": 64,
         "batches": 32, "epochs": 8},
        # one date of the 128-wide network on a million paths
        {"name": "fit_128", "kind": "fit", "M": 1048576, "hidden": 128, "batches": 32, "epochs": 8},
        # CVA_0 with 53 sensitivities, as a hedging loop calls it
        {"name": "adjoint", "kind": "adjoint", "model": "paper", "M": 131072, "n": 100, "S": 1},
        # the validation run: too few paths to fill the card by themselves, many copies
        {"name": "nested", "kind": "nested", "model": "paper", "M": 16384, "N": 64, "n": 100, "copies": 32},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["simulate", "simulate", "simulate", "regress", "lsq", "alive", "fit", "learn", "adjoint",
                       "nested"])
    n = rng.choice([20, 30, 40, 50, 60, 80, 100, 110, 120])
    if kind == "simulate":
        model = rng.choice(["small", "paper", "paper", "mixed"])
        if model == "small":
            return {"kind": kind, "model": model, "M": log(1000, 400000), "N": log(1, 256), "n": rng.choice([25, 50, 100]),
                    "S": rng.choice([1, 1, 4]), "books": 1, "regress": rng.choice(["poly2", "linear"])}
        if model == "mixed":
            return {"kind": kind, "model": model, "M": log(1000, 60000), "N": log(1, 256), "n": n,
                    "S": 1, "books": 4, "regress": "linear"}
        return {"kind": kind, "model": model, "M": log(1000, 130000), "N": log(1, 512), "n": n,
                "S": rng.choice([1, 1, 2, 5]), "books": rng.choice([1, 6]), "regress": rng.choice(["", "linear", "poly2"])}
    if kind == "regress":
        return {"kind": kind, "M": log(2000, 1000000), "F": rng.randint(1, 31)}
    if kind in ("lsq", "alive"):
        return {"kind": kind, "model": rng.choice(["small", "paper", "paper"]), "M": log(4000, 130000),
                "N": log(16, 128), "n": n if kind == "lsq" else min(n, 100)}
    if kind == "fit":
        hidden, batches = rng.choice([64, 128]), rng.choice([8, 16, 32])
        return {"kind": kind, "M": 128 * batches * rng.randint(1, 32), "hidden": hidden, "batches": batches,
                "epochs": rng.choice([2, 4, 8])}
    if kind == "learn":
        batches = rng.choice([8, 16, 32])
        return {"kind": kind, "model": "paper", "M": 128 * batches * rng.randint(1, 24), "N": log(16, 128),
                "n": rng.choice([20, 30, 40]), "hidden": rng.choice([64, 128]), "batches": batches,
                "epochs": rng.choice([2, 4, 8])}
    if kind == "adjoint":
        return {"kind": kind, "model": "paper", "M": log(1000, 120000), "n": rng.choice([20, 50, 100]),
                "S": rng.choice([1, 1, 2])}
    return {"kind": kind, "model": "paper", "M": log(1000, 16000), "N": log(8, 128), "n": n,
            "copies": rng.randint(4, 24)}


# ------------------------------------------------------------- inputs -----


def _books(rng, sizes, model, horizon):
    out = []
    for s in sizes:
        out.append(workload.Portfolio(
            ccy=rng.integers(0, model.E, size=s).astype(np.int32),
            cpty=rng.integers(0, model.C, size=s).astype(np.int32),
            notional=rng.lognormal(0.0, 0.5, size=s),
            omega=np.where(rng.uniform(size=s) < 0.5, 1, -1).astype(np.int32),
            n_periods=np.maximum(1, np.rint(rng.uniform(1.0, horizon, size=s))).astype(np.int32)))
    return out


def _market(case, seed):
    """(model, portfolios, grid) of a case: drawn from the seed."""
    rng = np.random.default_rng([22111, seed])
    if case["model"] == "small":
        model, horizon, sizes = workload.small_model(), 5.0, (10,)
    elif case["model"] == "mixed":
        model, horizon, sizes = workload.mixed_model(rng), 10.0, BOOKS[case["books"]]
    else:
        model, horizon, sizes = workload.paper_model(rng), 10.0, BOOKS[case.get("books", 1)]
    return model, _books(rng, sizes, model, horizon), workload.Grid(horizon, case["n"], case.get("S", 1))


def _key(seed):
    return 1 + seed % (1 << 40)


def _date_of_fit(case):
    """The single-date cases take date 5 of a yearly simulation of the paper's market."""
    return {"model": "paper", "M": case["M"], "N": 64, "n": 10}


def _regress_arrays(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    F, M = case["F"], case["M"]
    mix = torch.eye(F, device="cuda") + 0.3 * torch.randn(F, F, generator=g, device="cuda") / math.sqrt(F)
    level = 0.01 + 0.02 * torch.rand(F, 1, generator=g, device="cuda")
    features = level + 0.01 * (mix @ torch.randn(F, M, generator=g, device="cuda"))
    slope = torch.randn(F, generator=g, device="cuda")
    targets = torch.relu(0.02 + (slope @ (features - level)) + 0.01 * torch.randn(M, generator=g, device="cuda"))
    return targets.contiguous(), features.contiguous()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "regress":
        targets, features = _regress_arrays(case, seed)
        return {"case": case, "targets": targets, "features": features}
    if kind == "adjoint":
        model, books, grid = _market(case, seed)
        theta = torch.tensor(api.grad_params(model), dtype=torch.float32, device="cuda", requires_grad=True)
        return {"case": case, "model": model, "book": api.frozen(model, books[0]), "grid": grid, "theta": theta,
                "key": _key(seed)}
    inner = _date_of_fit(case) if kind == "fit" else case
    model, books, grid = _market(inner, seed)
    sim = api.Simulation(model, books, grid, inner["M"], inner["N"], keep_defaults=kind == "alive")
    state = {"case": case, "sim": sim, "key": _key(seed)}
    if kind == "simulate":
        if case["books"] == 6:
            sim.autotune(_key(seed), case["regress"] or "linear")
        state["views"] = (sim.features(), sim.discount_integral(), sim.thresholds(), sim.exposures(), sim.targets())
        if case["regress"]:
            state["pred"] = torch.zeros(sim.n_pf, sim.n, sim.M, device="cuda")
        return state
    if kind == "nested":
        return state
    sim.run(state["key"])
    if kind in ("fit", "learn"):
        p = workload.mlp_init(sim.F, case["hidden"], seed=1000 + seed)
        state["init"] = api.mlp_pack(p, case["hidden"])
        state["params"] = state["init"].clone()
        if kind == "fit":
            state["features"], state["targets"] = sim.features()[5].clone(), sim.targets()[0, 5].clone()
            sim.close()
    else:
        state["pred"] = torch.zeros((sim.n_pf, sim.n, sim.M) if kind == "lsq" else (sim.n, sim.M), device="cuda")
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "simulate":
        state["sim"].run(state["key"])
        out = dict(zip(("features", "discount", "thresholds", "exposures", "targets"), state["views"]))
        if case["regress"]:
            out["predictions"] = state["sim"].regress_portfolios(case["regress"], pred=state["pred"])[0]
        return out
    if kind == "regress":
        return api.regress(state["targets"], state["features"], want_coef=False)[0]
    if kind == "lsq":
        return state["sim"].regress_portfolios("linear", pred=state["pred"])[0]
    if kind == "alive":
        return state["sim"].regress_alive(0, pred=state["pred"], want_coef=False)[0]
    if kind == "fit":
        state["params"].copy_(state["init"])
        pred, losses = api.mlp_fit(state["targets"], state["features"], state["params"], hidden=case["hidden"],
                                   n_batches=case["batches"], epochs=case["epochs"])
        return {"predictions": pred, "losses": losses, "params": state["params"]}
    if kind == "learn":
        state["params"].copy_(state["init"])
        pred = api.mlp_regress_all(state["sim"], state["params"], hidden=case["hidden"], n_batches=case["batches"],
                                   epochs=case["epochs"])
        return {"predictions": pred, "params": state["params"]}
    if kind == "adjoint":
        state["theta"].grad = None
        cva0 = api.SmoothCVA0.apply(state["theta"], state["model"], state["book"], state["grid"], case["M"],
                                    state["key"])
        cva0.backward()
        return {"cva0": cva0.detach(), "grad": state["theta"].grad}
    return state["sim"].nested_reference(state["key"], case["n"] // 2, case["copies"])


# --------------------------------------------------------------- work -----


def _shape(case):
    if case["model"] == "small":
        return 1, 2, 0, 1
    if case["model"] == "mixed":
        return 3, 5, 3, 4
    return 10, 8, 8, case.get("books", 1)


def _sim_work(case):
    """Bytes and operations of one simulation: every output written once; the correlation, the factor
    steps, the bond prices and the date-bucketed portfolio sums, the search of every inner clock."""
    E, C, CS, P = _shape(case)
    F, M, N, n, S = 2 * E - 1 + CS, case["M"], case["N"], case["n"], case.get("S", 1)
    written = 4.0 * M * ((n + 1) * (F + 1 + C + P * C) + P * n)
    steps = M * n * S * (F * (F + 1) + 40.0 * F)
    prices = M * n * (E * 100.0 + P * C * E * 20.0)
    inner = M * float(N) * C * (2 * math.log2(n) + 20) + M * n * P * C * 2.0
    return written, steps + prices + inner


def _lsq_work(M, F, n, P, poly2):
    """The state and the targets read once, the predictions written once; normal equations and fits."""
    m = 3 if poly2 else F + 1
    cols = 1 if poly2 else F
    return 4.0 * M * (n - 1) * (cols + 2 * P), M * (n - 1.0) * (m * (m + 1) + 4 * m * P)


def _mlp_work(M, F, u, epochs):
    fwd = 2.0 * (F * u + u * u + u)
    train = fwd + 2.0 * (2 * u * u + F * u + 2 * u)
    return M * (epochs * train + (epochs + 1) * fwd)


def work(case):
    kind = case["kind"]
    if kind == "simulate":
        b, f = _sim_work(case)
        if case["regress"]:
            E, C, CS, P = _shape(case)
            rb, rf = _lsq_work(case["M"], 2 * E - 1 + CS, case["n"], P, case["regress"] == "poly2")
            b, f = b + 4.0 * case["M"] * (case["n"] - 1) * P, f + rf
        return {"bytes": b, "flops": f}
    if kind == "regress":
        b, f = _lsq_work(case["M"], case["F"], 2, 1, False)
        return {"bytes": b, "flops": f}
    if kind == "fit":
        F, u = 27, case["hidden"]
        return {"bytes": 4.0 * case["M"] * (F + 2), "flops": _mlp_work(case["M"], F, u, case["epochs"])}
    E, C, CS, P = _shape(case)
    F, M, n = 2 * E - 1 + CS, case["M"], case["n"]
    if kind == "lsq":
        b, f = _lsq_work(M, F, n, 1, False)
        return {"bytes": b, "flops": f}
    if kind == "alive":
        m = 1 + F + C
        return {"bytes": M * (n - 1.0) * 4 * (F + 2) + 4.0 * M * n * (C + 1) + M * case["N"] * C,
                "flops": M * (n - 1.0) * (m * (m + 1) + 4 * m) + 4.0 * M * case["N"] * C * C}
    if kind == "learn":
        return {"bytes": 4.0 * M * (n - 1) * (F + 2), "flops": (n - 1) * _mlp_work(M, F, case["hidden"], case["epochs"])}
    if kind == "adjoint":
        _, f = _sim_work({**case, "N": 0})
        return {"bytes": 8.0 * (3 * E + 3 * C), "flops": 3.0 * f}
    _, f = _sim_work(case)
    return {"bytes": 4.0 * M, "flops": case["copies"] * f / 2}


# ------------------------------------------ the same in 64 bits, plain torch


def _philox(ctr, seed):
    """Philox4x32-10 of the four counter words (int64 tensors below 2^32), key = seed."""
    low = 0xFFFFFFFF
    k0, k1 = seed & low, (seed >> 32) & low

    def mul(a, b):   # (high, low) words of a * b, a a constant: 16-bit halves keep int64 exact
        p0, p1 = a * (b & 0xFFFF), a * (b >> 16)
        t = (p0 >> 16) + p1
        return t >> 16, ((t & 0xFFFF) << 16) | (p0 & 0xFFFF)

    x0, x1, x2, x3 = ctr
    for _ in range(10):
        h0, l0 = mul(0xD2511F53, x0)
        h1, l1 = mul(0xCD9E8D57, x2)
        x0, x1, x2, x3 = h1 ^ x1 ^ k0, l1, h0 ^ x3 ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & low, (k1 + 0xBB67AE85) & low
    return x0, x1, x2, x3


def _uniform(x):
    return ((x >> 9).double() + 0.5) * 2.0 ** -23


def _normals(seed, k, q, copy, F):
    """Standard normals [paths, F] of fine step q; copy is the third counter word."""
    b = torch.arange((F + 3) // 4, device="cuda")
    k2 = k[:, None].expand(-1, b.numel())
    x = _philox((k2, torch.full_like(k2, q), copy[:, None].expand_as(k2), ((1 << 24) + b).expand_as(k2)), seed)
    u = [_uniform(v) for v in x]
    r0, r1 = (torch.sqrt(-2.0 * torch.log(v)) for v in (u[0], u[2]))
    a0, a1 = 2.0 * math.pi * u[1], 2.0 * math.pi * u[3]
    z = torch.stack([r0 * torch.cos(a0), r0 * torch.sin(a0), r1 * torch.cos(a1), r1 * torch.sin(a1)], dim=2)
    return z.reshape(k.numel(), -1)[:, :F]


class _Market64:
    """The market of a case for the outer paths k, date by date, in 64 bits. theta (the parameters of
    the sensitivities) may carry gradients."""

    def __init__(self, model, books, grid, theta=None):
        t = lambda x: torch.as_tensor(np.asarray(x, dtype=np.float64), device="cuda")   # noqa: E731
        E, C = model.E, model.C
        self.E, self.C, self.n, self.S = E, C, grid.n_steps, grid.substeps
        self.cir = torch.as_tensor(np.flatnonzero(np.asarray(model.cir_nu) > 0), device="cuda")
        self.F = 2 * E - 1 + self.cir.numel()
        if theta is None:
            theta = t(np.concatenate([model.curve, model.hw_sigma, model.fx_vol[1:], model.cir_kappa, model.cir_theta,
                                      model.cir_nu]))
        self.f, self.sr, sx, self.kappa, self.theta, self.nu = torch.split(theta, [E, E, E - 1, C, C, C])
        self.sx = torch.cat([torch.zeros(1, dtype=torch.float64, device="cuda"), sx])
        self.a, self.chi0, self.gamma0, self.lgd = t(model.hw_a), t(model.fx0), t(model.gamma0), 1.0 - t(model.recovery)
        corr = t(model.corr)
        self.L = torch.linalg.cholesky(corr)
        self.rho = torch.stack([torch.zeros((), dtype=torch.float64, device="cuda")]
                               + [corr[e, E - 1 + e] for e in range(1, E)])
        self.delta = books[0].delta
        self.dt = grid.horizon / grid.n_steps
        self.ds = self.dt / grid.substeps
        self.ppp = int(round(self.delta / self.dt))
        self.G = max(int(b.n_periods.max()) for b in books)
        wA, wK = (np.zeros((len(books), C, E, self.G)) for _ in range(2))
        for i, b in enumerate(books):
            fixed = b.fixed_rate if b.fixed_rate is not None else self._par(model, b)
            for s in range(b.n_swaps):
                live = np.arange(self.G) < b.n_periods[s]
                wA[i, b.cpty[s], b.ccy[s]] += live * (b.omega[s] * b.notional[s])
                wK[i, b.cpty[s], b.ccy[s]] += live * (b.omega[s] * b.notional[s] * b.delta * fixed[s])
        # [e, (differences, prices), (book, counterparty)]
        self.w = t(np.concatenate([wA, -wK], axis=3)).permute(2, 3, 0, 1).reshape(E, 2 * self.G, -1)

    @staticmethod
    def _par(model, book):
        a, s, f = model.hw_a, model.hw_sigma, model.curve
        out = np.zeros(book.n_swaps)
        for i in range(book.n_swaps):
            e = book.ccy[i]
            T = book.delta * np.arange(1, book.n_periods[i] + 1)
            B = (1 - np.exp(-a[e] * T)) / a[e]
            zc = np.exp(-f[e] * T + B * f[e] - B * f[e])
            out[i] = (1 - zc[-1]) / (book.delta * zc.sum())
        return out

    def _log_zc(self, t, T):
        """(ln A, B) [E, len(T)] of ZC_t(T) = exp(ln A - B r)."""
        tau = torch.as_tensor(np.atleast_1d(T) - t, dtype=torch.float64, device="cuda")
        a, f, s = self.a[:, None], self.f[:, None], self.sr[:, None]
        B = -torch.expm1(-a * tau) / a
        return -f * tau + B * f - s * s / (4 * a) * (-torch.expm1(-2 * a * t)) * B * B, B

    def _exposure(self, j, r, lchi, r_fix, I0):
        """Exposures [book, C, paths] at date j >= 1."""
        t = j * self.dt
        p = (j - 1) // self.ppp
        Z = torch.zeros(r.shape[0], self.E, self.G, dtype=torch.float64, device="cuda")
        if p >= self.G:
            return torch.zeros(self.w.shape[2] // self.C, self.C, r.shape[0], dtype=torch.float64, device="cuda")
        lnA, B = self._log_zc(t, self.delta * np.arange(p + 1, self.G + 1))
        live = torch.exp(lnA - B * r[:, :, None])
        fA, fB = self._log_zc(p * self.delta, (p + 1) * self.delta)
        first = live[:, :, :1] * torch.expm1((fB * r_fix[:, :, None]) - fA)
        D = torch.cat([Z[:, :, :p], first, live[:, :, :-1] - live[:, :, 1:]], dim=2)
        Z = torch.cat([Z[:, :, :p], live], dim=2)
        X = torch.exp(lchi)[:, :, None] * torch.cat([D, Z], dim=2)
        mtm = (X.reshape(r.shape[0], -1) @ self.w.reshape(self.E * 2 * self.G, -1)).T.reshape(-1, self.C, r.shape[0])
        return self.lgd[:, None] * torch.exp(-I0) * torch.relu(mtm)

    def dates(self, k, seed, branch_date=1 << 30, copy=None):
        """Yields (features [F, paths], int r^0, Lambda [C, paths], exposures) at dates 0..n."""
        none = torch.zeros_like(k)
        copy = none if copy is None else copy
        P = k.numel()
        r, lchi = self.f.expand(P, -1), torch.log(self.chi0).expand(P, -1)
        gam, Lam = self.gamma0.expand(P, -1), torch.zeros(P, self.C, dtype=torch.float64, device="cuda")
        I0 = torch.zeros(P, dtype=torch.float64, device="cuda")
        at = lambda: torch.cat([r, lchi[:, 1:], gam[:, self.cir]], dim=1).T   # noqa: E731
        shape = (self.w.shape[2] // self.C, self.C, P)
        yield at(), I0, Lam.T, torch.zeros(shape, dtype=torch.float64, device="cuda")
        r_fix, sq = r, math.sqrt(self.ds)
        for j in range(1, self.n + 1):
            for s in range(self.S):
                q = (j - 1) * self.S + s
                W = _normals(seed, k, q, copy if j > branch_date else none, self.F) @ self.L.T
                t = q * self.ds
                drift = (self.a * self.f + self.sr ** 2 / (2 * self.a) * (-torch.expm1(-2 * self.a * t))
                         - self.rho * self.sx * self.sr - self.a * r)
                gp = torch.relu(gam)
                I0, Lam = I0 + r[:, 0] * self.ds, Lam + gp * self.ds
                dx = (r[:, :1] - r - 0.5 * self.sx ** 2) * self.ds
                Wx = torch.cat([torch.zeros(P, 1, dtype=torch.float64, device="cuda"), W[:, self.E:2 * self.E - 1]], dim=1)
                lchi = torch.cat([lchi[:, :1], (lchi + dx + self.sx * sq * Wx)[:, 1:]], dim=1)
                r = r + drift * self.ds + self.sr * sq * W[:, :self.E]
                if self.cir.numel():
                    c = self.cir
                    # sqrt as a power of the clamped value: its slope at 0 is not asked for
                    root = torch.where(gp[:, c] > 0, torch.sqrt(torch.where(gp[:, c] > 0, gp[:, c], 1.0)), 0.0)
                    step = self.kappa[c] * (self.theta[c] - gp[:, c]) * self.ds + self.nu[c] * root * sq * W[:, 2 * self.E - 1:]
                    gam = gam.index_add(1, c, step)
            yield at(), I0, Lam.T, self._exposure(j, r, lchi, r_fix, I0)
            if j % self.ppp == 0:
                r_fix = r


def _default_steps(thr, k, seed, N, copy=None):
    """Default steps [paths, N, C] (n + 1: none) of the thresholds thr [n+1, C, paths]."""
    n, C, P = thr.shape[0] - 1, thr.shape[1], thr.shape[2]
    copy = torch.zeros_like(k) if copy is None else copy
    out = torch.empty(P, N, C, dtype=torch.int16, device="cuda")
    T = thr[1:].permute(2, 1, 0).contiguous()
    step = max(1, (1 << 24) // N)
    for i in range(0, P, step):
        kk = k[i:i + step, None].expand(-1, N)
        cc = copy[i:i + step, None].expand(-1, N)
        l = torch.arange(N, device="cuda").expand_as(kk)   # noqa: E741
        for b in range((C + 3) // 4):
            x = _philox((kk, l, cc, torch.full_like(kk, (2 << 24) + b)), seed)
            for t in range(min(4, C - 4 * b)):
                c = 4 * b + t
                out[i:i + step, :, c] = 1 + torch.searchsorted(T[i:i + step, c].contiguous(), _uniform(x[t]).contiguous())
    return out


def _simulate64(case, seed, chunk=1 << 16):
    """Everything run() returns for a simulation, and its default steps, chunk by chunk of paths."""
    m = _Market64(*_market(case, seed))
    parts = []
    for k0 in range(0, case["M"], chunk):
        k = torch.arange(k0, min(case["M"], k0 + chunk), device="cuda")
        ft, I0, Lam, ex = (torch.stack(v) for v in zip(*m.dates(k, _key(seed))))
        thr = -torch.expm1(-Lam)
        steps = _default_steps(thr, k, _key(seed), case["N"])
        targets = _targets(m, steps, ex, I0, case["N"])
        parts.append((ft, I0, thr, ex.permute(1, 0, 2, 3), targets, steps if case["kind"] == "alive" else None))
    ft, I0, thr, ex, targets = (torch.cat([p[i] for p in parts], dim=-1) for i in range(5))
    steps = torch.cat([p[5] for p in parts]) if case["kind"] == "alive" else None
    return m, ft, I0, thr, ex, targets, steps


def _counts(steps, n):
    P, N, C = steps.shape
    cnt = torch.zeros(P, C, n + 2, dtype=torch.float64, device="cuda")
    idx = steps.permute(0, 2, 1).long()
    return cnt.scatter_add_(2, idx, torch.ones(1, dtype=torch.float64, device="cuda").expand_as(idx))


def _targets(m, steps, ex, I0, N):
    """Averaged targets [book, n, paths]."""
    cnt = _counts(steps, m.n)[:, :, 1:m.n + 1].permute(2, 1, 0)
    loss = (ex[1:] * cnt[:, None]).sum(2) / N
    later = torch.flip(torch.cumsum(torch.flip(loss, (0,)), 0), (0,))
    return (torch.exp(I0[:m.n])[:, None] * later).permute(1, 0, 2)


def _fit64(basis, y):
    """Fitted values [cols, paths] of the targets y on the rows of basis (constant rows add nothing)."""
    B = basis - basis.mean(1, keepdim=True)
    scale = B.norm(dim=1, keepdim=True)
    B = B[(scale > 1e-12 * math.sqrt(B.shape[1])).squeeze(1)]
    B = B / B.norm(dim=1, keepdim=True)
    mean = y.mean(1, keepdim=True)
    for _ in range(2):   # the second pass removes what rounding of the normal equations left
        w = torch.linalg.solve(B @ B.T, B @ (y - mean).T) if _ == 0 else w + torch.linalg.solve(
            B @ B.T, B @ (y - mean - w.T @ B).T)
    return mean + w.T @ B


def _fits64(m, features, targets, basis):
    """Predictions [book, n, paths] at every date (date 0: none)."""
    out = torch.zeros_like(targets)
    for j in range(1, m.n):
        f = features[j]
        rows = torch.stack([f[0], (f[0] - f[0].mean()) ** 2]) if basis == "poly2" else f
        out[:, j] = _fit64(rows, targets[:, j])
    return out


def _alive64(case, m, ft, I0, ex, steps):
    """Fit at "all alive" of the single-draw targets on (state, default indicators) at every date."""
    n, C, N, P = m.n, m.C, case["N"], case["M"]
    out = torch.zeros(n, P, dtype=torch.float64, device="cuda")
    step = 1 << 14
    for j in range(1, n):
        f = ft[j]
        shift = f.mean(1, keepdim=True)
        Y = f - shift
        spread = Y.norm(dim=1, keepdim=True) / math.sqrt(P)
        Y = (Y / spread)[(spread > 1e-12).squeeze(1)]
        rows = torch.cat([torch.ones(1, P, dtype=torch.float64, device="cuda"), Y])
        d = torch.zeros(C, P, dtype=torch.float64, device="cuda")
        xx = torch.zeros(C, C, dtype=torch.float64, device="cuda")
        xy = torch.zeros(C, dtype=torch.float64, device="cuda")
        tot = torch.zeros(P, dtype=torch.float64, device="cuda")
        for i in range(0, P, step):
            s = steps[i:i + step].long()
            X = (s <= j).double()
            V = ex[0, :, :, i:i + step].permute(2, 0, 1)                    # [paths, n+1, C]
            V = torch.cat([V, torch.zeros_like(V[:, :1])], dim=1)
            loss = torch.where(s > j, torch.gather(V, 1, s), 0.0).sum(2) * torch.exp(I0[j, i:i + step])[:, None]
            d[:, i:i + step] = X.sum(1).T
            flat = X.reshape(-1, C)
            xx += flat.T @ flat
            xy += flat.T @ loss.reshape(-1)
            tot[i:i + step] = loss.sum(1)
        has = d.sum(1) > 0
        A = torch.cat([torch.cat([N * rows @ rows.T, rows @ d[has].T], 1),
                       torch.cat([d[has] @ rows.T, xx[has][:, has]], 1)])
        b = torch.cat([rows @ tot, xy[has]])
        s = 1.0 / torch.sqrt(torch.diagonal(A))
        w = s * torch.linalg.solve(s[:, None] * A * s, s * b)
        out[j] = w[:rows.shape[0]] @ rows
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind in ("fit", "learn"):      # training in 16-bit operands has no value in 64 bits
        return None
    if kind == "regress":
        targets, features = _regress_arrays(case, seed)
        return _fit64(features.double(), targets.double()[None])[0]
    if kind == "simulate":
        m, ft, I0, thr, ex, targets, _ = _simulate64(case, seed)
        out = {"features": ft, "discount": I0, "thresholds": thr, "exposures": ex, "targets": targets}
        if case["regress"]:
            out["predictions"] = _fits64(m, ft, targets, case["regress"])
        return out
    if kind == "lsq":
        m, ft, _, _, _, targets, _ = _simulate64(case, seed)
        return _fits64(m, ft, targets, "linear")
    if kind == "alive":
        m, ft, I0, _, ex, _, steps = _simulate64(case, seed)
        return _alive64(case, m, ft, I0, ex, steps)
    if kind == "adjoint":
        model, books, grid = _market(case, seed)
        book = books[0]
        book.fixed_rate = _Market64._par(model, book)
        theta = torch.tensor(np.concatenate([model.curve, model.hw_sigma, model.fx_vol[1:], model.cir_kappa,
                                             model.cir_theta, model.cir_nu]), dtype=torch.float32, device="cuda")
        theta = theta.double().requires_grad_()
        total = 0.0
        for k0 in range(0, case["M"], 16384):
            k = torch.arange(k0, min(case["M"], k0 + 16384), device="cuda")
            m, last, s = _Market64(model, [book], grid, theta), 0.0, 0.0
            for j, (_, _, Lam, ex) in enumerate(m.dates(k, _key(seed))):
                alive = torch.exp(-Lam)
                if j:
                    s = s + (ex[0] * (last - alive)).sum()
                last = alive
            (s / case["M"]).backward()
            total += float(s.detach()) / case["M"]
        return {"cva0": torch.tensor(total, dtype=torch.float64, device="cuda"), "grad": theta.grad}
    date, copies = case["n"] // 2, case["copies"]
    m = _Market64(*_market(case, seed))
    out = torch.zeros(case["M"], dtype=torch.float64, device="cuda")
    for c0 in range(1, copies + 1, 8):
        ids = torch.arange(c0, min(copies, c0 + 7) + 1, device="cuda")
        k = torch.arange(case["M"], device="cuda").repeat(ids.numel())
        copy = ids.repeat_interleave(case["M"])
        _, I0, Lam, ex = (torch.stack(v) for v in zip(*m.dates(k, _key(seed), date, copy)))
        steps = _default_steps(-torch.expm1(-Lam), k, _key(seed), case["N"], copy)
        out += _targets(m, steps, ex, I0, case["N"])[0, date].reshape(ids.numel(), -1).sum(0)
    return out / copies
