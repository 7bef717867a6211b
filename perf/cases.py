"""Performance cases of the Black-Scholes Parareal library.

Each case is one call (or one pass over what a user's program holds) of a public entry point of
``paper_2404_02521_gb300``: the fine propagator F, the numerical and the PINO coarse propagators
G, the training loss's PDE term with its gradient, and whole Parareal solves for two and for
three assets.  A case is a dict of plain values:

  op        "fine", "coarse", "pino", "physics", "solve" or "solve3"
  M, xmax   nodes per axis on [0, xmax]^d
  payoff    "basket", "exchange", "call" or "cash"
  batch     independent states of the call; params: distinct option parameter sets among them
            (one: the time slices of one solve; several: requests or training problems)
  dtau      step size of F, or slice length of G and of the physics loss
  steps     implicit steps of the call (fine, coarse), per slice
  and for solves N, fine_steps, coarse_steps, tol.

``exact`` restates the mathematics in 64 bits with torch alone: the 9- and 19-point centred
differences, implicit Euler with a converged solve per step, the textbook Parareal iteration,
and the Fourier neural operator with FFTs.
"""
from __future__ import annotations

import math
import os
import tempfile
from types import SimpleNamespace

import numpy as np
import torch

import paper_2404_02521_gb300 as bs
from paper_2404_02521_gb300 import pino_io

PAYOFFS = {"basket": bs.BASKET, "exchange": bs.EXCHANGE, "call": bs.CALL1, "cash": bs.CASH_OR_NOTHING}
DEV = "cuda"


# ------------------------------------------------------------------------------------------
# The cases
# ------------------------------------------------------------------------------------------

def listed():
    return [
        # F on all 8 slices of the small basket solve, one whole slice of 256 steps each: the
        # smallest Parareal solve, where latency counts.
        dict(name="fine64", op="fine", M=64, xmax=4.0, payoff="basket", batch=8, params=1,
             dtau=1.0 / 2048, steps=256),
        # Serial fine stepping of the 256 x 256 exchange option: one state, one slice.
        dict(name="fine256_one", op="fine", M=256, xmax=4.0, payoff="exchange", batch=1, params=1,
             dtau=1.0 / 32768, steps=512),
        # F on all 64 slices of that solve at once: one Parareal iteration's fine work.
        dict(name="fine256_batch", op="fine", M=256, xmax=4.0, payoff="exchange", batch=64, params=1,
             dtau=1.0 / 32768, steps=512),
        # The paper's cash-or-nothing grid (301 nodes, odd) with a quarter of 64 slices for two
        # options at once, as the server batches requests.
        dict(name="fine301_two_options", op="fine", M=301, xmax=300.0, payoff="cash", batch=16, params=2,
             dtau=1.0 / 16384, steps=256),
        # One chunk (a quarter of 128 slices) of F in the large 1024 x 1024 basket solve.
        dict(name="fine1024_chunk", op="fine", M=1024, xmax=4.0, payoff="basket", batch=32, params=1,
             dtau=1.0 / 131072, steps=1024),
        # The numerical G of one slice of the exchange solve: the unit of the serial sweep.
        dict(name="coarse256", op="coarse", M=256, xmax=4.0, payoff="exchange", batch=1, params=1,
             dtau=1.0 / 64, steps=4),
        # The numerical G of a 512 x 512 serving request on its own grid (one step per slice of
        # T = 1, N = 32; four slices' worth of steps).
        dict(name="coarse512", op="coarse", M=512, xmax=4.0, payoff="exchange", batch=1, params=1,
             dtau=4.0 / 32, steps=4),
        # The PINO as G: one slice of the 128 x 128 basket (PINO-Parareal's serial sweep) ...
        dict(name="pino128_one", op="pino", M=128, xmax=4.0, payoff="basket", batch=1, params=1,
             dtau=1.0 / 64, steps=1),
        # ... and 128 concurrent solves' slices in one call, each with its own option.
        dict(name="pino128_batch", op="pino", M=128, xmax=4.0, payoff="basket", batch=128, params=128,
             dtau=1.0 / 64, steps=1),
        # The physics-informed loss term and its gradient for one training batch.
        dict(name="physics128", op="physics", M=128, xmax=4.0, payoff="basket", batch=32, params=32,
             dtau=1.0 / 64, steps=1),
        # Whole solves to tolerance: the 256 x 256 exchange option, and a three-asset basket.
        dict(name="solve256", op="solve", M=256, xmax=4.0, payoff="exchange", N=64, fine_steps=512,
             coarse_steps=4, tol=1e-4),
        dict(name="solve3_64", op="solve3", M=64, xmax=4.0, payoff="basket", N=16, fine_steps=40,
             coarse_steps=2, tol=1e-5),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["fine", "fine", "fine", "coarse", "coarse", "pino", "physics", "solve", "solve3"])
    c = dict(op=op, xmax=4.0, payoff=rng.choice(["basket", "exchange"]))
    if op == "fine":
        # any grid from the smallest to the large solve's, a batch of slices of one or several
        # options, the Jacobi bound of a step between easy and the server's limit
        c["payoff"] = rng.choice(["basket", "exchange", "call"])
        c["M"] = M = _log_int(rng, 33, 1024)
        cap = 64 * 256 * 256 * 512 / (M * M)             # node-steps
        c["steps"] = steps = max(4, min(_log_int(rng, 32, 1024), int(cap)))
        c["batch"] = max(1, min(_log_int(rng, 1, 64), int(cap / steps)))
        c["params"] = rng.choice([1, 1, min(4, c["batch"]), c["batch"]])
        c["dtau"] = rng.uniform(0.3, 0.65) / (0.1225 * 1.7 * M * M)
    elif op == "coarse":
        c["M"] = M = _log_int(rng, 48, 600)
        c["batch"] = 1 if M > 256 else rng.choice([1, 1, _log_int(rng, 2, 64)])
        c["params"] = rng.choice([1, min(4, c["batch"])])
        c["dtau"] = 1.0 / rng.choice([16, 32, 64])
        c["steps"] = rng.choice([1, 2, 4])
    elif op == "pino":
        c["M"] = M = rng.choice([64, 96, 128, 128, 200, 256, 512])
        c["batch"] = rng.choice([1, 1, _log_int(rng, 2, 96 if M <= 128 else 16)])
        c["params"] = c["batch"]
        c["dtau"] = 1.0 / rng.choice([12, 16, 32, 64])
        c["steps"] = 1
    elif op == "physics":
        c["M"] = _log_int(rng, 33, 256)
        c["batch"] = c["params"] = _log_int(rng, 1, 64)
        c["dtau"] = 1.0 / rng.choice([12, 16, 32, 64])
        c["steps"] = 1
    elif op == "solve":
        c["M"] = M = _log_int(rng, 40, 256)
        c["N"] = rng.choice([8, 16, 32, 64])
        per_year = 0.1225 * 1.7 * M * M / 0.65            # steps that keep the Jacobi bound <= 0.65
        c["fine_steps"] = max(16, int(math.ceil(per_year / c["N"])))
        c["coarse_steps"] = rng.choice([1, 2, 4])
        c["tol"] = 1e-4
    else:
        c["M"] = M = rng.randint(20, 60)
        c["N"] = rng.choice([4, 8, 12])
        c["fine_steps"] = max(8, -(-M * M // 90)) + rng.randint(0, 8)   # Jacobi bound <= 0.72
        c["coarse_steps"] = rng.choice([1, 2])
        c["tol"] = 1e-4
        c["T"] = c["N"] / 16.0
    return c


# ------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------

def _options(case, seed):
    """The case's option parameter sets.  A single one is the configuration's own option with a
    strike (or, for the exchange option, a second volatility) of the seed; several are drawn from
    the ranges that requests and training problems have."""
    rng = np.random.default_rng([seed, 1])
    n = int(case.get("params", 1))
    pay = case["payoff"]
    T = float(case.get("T", 1.0))
    out = []
    for k in range(n):
        if pay == "cash":      # the paper's own problem: strikes around 100 on [0, 300]
            out.append(SimpleNamespace(sigma1=0.3, sigma2=0.3, rho=0.5, r=1.0, T=T, strike=float(rng.uniform(90, 110)),
                                       w1=0.5, w2=0.5, payoff=PAYOFFS[pay], strike2=float(rng.uniform(90, 110)),
                                       cash=1.0))
            continue
        if n == 1 and pay == "exchange":
            s1, s2, rho, r = 0.25, 0.35, float(rng.uniform(0.68, 0.70)), 0.03
        elif n == 1:
            s1, s2, rho, r = 0.3, 0.2, 0.5, 0.05
        else:
            s1, s2 = float(rng.uniform(0.1, 0.35)), float(rng.uniform(0.1, 0.35))
            rho, r = float(rng.uniform(-0.7, 0.7)), float(rng.uniform(0.0, 0.08))
        out.append(SimpleNamespace(sigma1=s1, sigma2=s2, rho=rho, r=r, T=T, strike=float(rng.uniform(0.9, 1.1)),
                                   w1=0.5, w2=0.5, payoff=PAYOFFS[pay], strike2=0.0, cash=1.0))
    return out


def _options3(case, seed):
    rng = np.random.default_rng([seed, 1])
    return SimpleNamespace(sigma=(0.3, 0.2, 0.25), rho=(0.5, -0.3, 0.2), r=0.05, strike=float(rng.uniform(0.9, 1.1)),
                           w=(0.4, 0.35, 0.25), payoff=PAYOFFS[case["payoff"]])


def _items(case, seed):
    """Per state of the call: its option and its time tau0 (slices of a solve on [0, 0.5])."""
    opts = _options(case, seed)
    B = int(case["batch"])
    per = -(-B // len(opts))
    ps = [opts[min(b // per, len(opts) - 1)] for b in range(B)]
    tau0 = [0.02 + 0.48 * (b % per) / max(1, per) for b in range(B)]
    return ps, tau0


def _coords(M, xmax):
    x = torch.arange(M, dtype=torch.float64, device=DEV) * (xmax / (M - 1))
    return x.view(1, M), x.view(M, 1)


def _state(p, M, xmax, tau):
    """A price surface at time tau as a solve meets it: the payoff smoothed over the option's own
    standard deviation (float32, on the GPU)."""
    X, Y = _coords(M, xmax)
    sd = math.sqrt(max(tau, 1e-3))
    if p.payoff == bs.BASKET:
        f, w = p.w1 * X + p.w2 * Y - p.strike * math.exp(-p.r * tau), 0.5 * (p.sigma1 + p.sigma2) * sd * p.strike
    elif p.payoff == bs.EXCHANGE:
        f, w = X - Y, 0.5 * (p.sigma1 + p.sigma2) * sd
    elif p.payoff == bs.CALL1:
        f, w = X - p.strike * math.exp(-p.r * tau) + 0.0 * Y, p.sigma1 * sd * p.strike
    else:
        sx, sy = p.sigma1 * sd * p.strike, p.sigma2 * sd * p.strike2
        u = p.cash * math.exp(-p.r * tau) * torch.special.ndtr((X - p.strike) / sx) * torch.special.ndtr(
            (Y - p.strike2) / sy)
        return u.float()
    w = 0.5 * w
    return torch.where(f > 20 * w, f + 0.0 * w, w * torch.log1p(torch.exp(torch.clamp(f / w, max=20.0)))).float()


PINO = dict(in_channels=9, width=32, modes_x=12, modes_y=12, layers=4, proj_hidden=128)


def _pino_weights(seed):
    """Network weights of a trained coarse model's magnitudes: the increment is a few percent of
    the state."""
    rng = np.random.default_rng([seed, 2])
    C, H, L, my2, mx = PINO["width"], PINO["proj_hidden"], PINO["layers"], 2 * PINO["modes_y"], PINO["modes_x"]
    s = 4.0 / (C * C)
    w = {"lift_w": rng.standard_normal((9, C)) / 3.0, "lift_b": 0.1 * rng.standard_normal(C),
         "spec_w": s * (rng.random((L, my2, mx, C, C)) + 1j * rng.random((L, my2, mx, C, C))),
         "pw_w": rng.standard_normal((L, C, C)) / math.sqrt(C), "pw_b": 0.1 * rng.standard_normal((L, C)),
         "proj1_w": rng.standard_normal((C, H)) / math.sqrt(C), "proj1_b": 0.1 * rng.standard_normal(H),
         "proj2_w": 0.01 * rng.standard_normal(H) / math.sqrt(H), "proj2_b": np.float64(0.0)}
    for k, v in w.items():     # the float32 values the file holds
        w[k] = np.asarray(v).astype(np.complex64 if np.iscomplexobj(v) else np.float32)
    return w


def _load_pino(seed):
    fd, path = tempfile.mkstemp(suffix=".bin")
    os.close(fd)
    try:
        pino_io.write_weights(path, _pino_weights(seed), *PINO.values())
        return bs.Pino(path)
    finally:
        os.unlink(path)


def prepare(case, seed):
    op, M = case["op"], int(case["M"])
    s = SimpleNamespace(case=case, M=M)
    if op == "solve3":
        s.p = _options3(case, seed)
        s.U = torch.empty((case["N"] + 1, M, M, M), device=DEV)
        return s
    s.grid = bs.Grid(M, case["xmax"])
    if op == "solve":
        (s.p,) = _options(case, seed)
        s.U = torch.empty((case["N"] + 1, M, M), device=DEV)
        return s
    s.p, s.tau0 = _items(case, seed)
    s.u = [_state(p, M, case["xmax"], t) for p, t in zip(s.p, s.tau0)]
    s.dtaus = [case["dtau"]] * len(s.u)
    if op == "physics":
        # a prediction of the next state: the state there, a few tenths of a percent off
        gen = torch.Generator(device=DEV).manual_seed(seed)
        s.pred = torch.stack([_state(p, M, case["xmax"], t + case["dtau"]) for p, t in zip(s.p, s.tau0)])
        s.pred += 2e-3 * torch.randn(s.pred.shape, generator=gen, device=DEV)
        s.loss = torch.empty(len(s.u), dtype=torch.float64, device=DEV)
        s.grad = torch.empty_like(s.pred)
        s.preds, s.grads = list(s.pred), list(s.grad)
        return s
    s.out = torch.empty((len(s.u), M, M), device=DEV)
    s.outs = list(s.out)
    s.net = _load_pino(seed) if op == "pino" else None
    return s


# ------------------------------------------------------------------------------------------
# One pass
# ------------------------------------------------------------------------------------------

def run(s):
    c = s.case
    op = c["op"]
    if op == "fine":
        bs.fine_propagate_batched(s.grid, s.p, s.u, s.outs, s.tau0, s.dtaus, c["steps"])
        return s.outs
    if op in ("coarse", "pino"):
        kind = bs.COARSE_PINO if op == "pino" else bs.COARSE_NUM
        if len(s.u) == 1:
            bs.coarse_propagate(s.grid, kind, s.net, s.p[0], s.u[0], s.outs[0], s.tau0[0], c["dtau"], c["steps"])
        else:
            bs.coarse_propagate_batched(s.grid, kind, s.net, s.p, s.u, s.outs, s.tau0, c["dtau"], c["steps"])
        return s.out
    if op == "physics":
        bs.pino_physics_loss(s.grid, s.p, s.preds, s.u, s.dtaus, s.loss, s.grads)
        return {"loss": s.loss, "grad": s.grad}
    # The iteration count and the whole trajectory; the defects beside them are residual norms at
    # the level of the coarse solver's tolerance.
    if op == "solve":
        _, k, _ = bs.parareal_solve(s.grid, s.p, c["N"], c["fine_steps"], bs.COARSE_NUM, c["coarse_steps"], None,
                                    c["tol"], c["N"], s.U)
    else:
        _, k, _ = bs.parareal_solve3(s.M, c["xmax"], s.p, c.get("T", 1.0), c["N"], c["fine_steps"],
                                     c["coarse_steps"], c["tol"], c["N"], s.U)
    return {"u": s.U, "iterations": k}


# ------------------------------------------------------------------------------------------
# What a pass cannot do without
# ------------------------------------------------------------------------------------------

def work(case):
    op, M = case["op"], case["M"]
    if op == "solve3":
        # one serial coarse sweep and one fine pass, the least a solve takes; a fine step is two
        # Jacobi sweeps of the 19-point update with the right-hand side and the compensated add
        n, N = M ** 3, case["N"]
        return {"bytes": 4.0 * n * (N + 1), "flops": float(n * N * (case["fine_steps"] * 122 + case["coarse_steps"] * 5 * 110))}
    n = M * M
    if op == "solve":
        N = case["N"]
        return {"bytes": 4.0 * n * (N + 1), "flops": float(n * N * (case["fine_steps"] * 54 + case["coarse_steps"] * 5 * 55))}
    B = case["batch"]
    if op == "fine":       # two Jacobi sweeps, the right-hand side and the compensated add per step
        return {"bytes": 8.0 * n * B, "flops": 54.0 * n * B * case["steps"]}
    if op == "coarse":     # five unpreconditioned BiCGSTAB iterations per step
        return {"bytes": 8.0 * n * B, "flops": 275.0 * n * B * case["steps"]}
    if op == "physics":    # prediction and previous state in, gradient out; residual and adjoint
        return {"bytes": 12.0 * n * B, "flops": 60.0 * n * B}
    # PINO: lifting, four layers (truncated transforms as products, mode mixing, pointwise), projection
    Mp = 128 if M <= 128 else 256
    P, C, mx, my2, H = Mp * Mp, 32, 12, 24, 128
    layer = (2 * C * P * 2 * mx + 8 * C * mx * Mp * my2) * 2 + 8 * C * C * mx * my2 + 2 * P * C * C
    weights = 4 * (8 * C * C * mx * my2 // 4 * 2 + C * C) * 2
    return {"bytes": 8.0 * n * B + weights, "flops": float(B * (2 * 9 * C * P + 4 * layer + 2 * P * C * H + 2 * P * H))}


# ------------------------------------------------------------------------------------------
# The same in 64 bits
# ------------------------------------------------------------------------------------------

def _far(p, X, Y, tau):
    """Far-field Dirichlet data at tau (X, Y broadcast, float64)."""
    ndtr = torch.special.ndtr
    X, Y = torch.broadcast_tensors(X, Y)
    if p.payoff == bs.BASKET:
        return torch.clamp(p.w1 * X + p.w2 * Y - p.strike * math.exp(-p.r * tau), min=0.0)
    tiny = 1e-300
    if p.payoff == bs.EXCHANGE:
        v = p.sigma1 ** 2 + p.sigma2 ** 2 - 2 * p.rho * p.sigma1 * p.sigma2
        sq = math.sqrt(v * tau)
        d1 = (torch.log(X.clamp(min=tiny) / Y.clamp(min=tiny)) + 0.5 * v * tau) / sq
        g = X * ndtr(d1) - Y * ndtr(d1 - sq)
        return torch.where(Y <= 0, X, torch.where(X <= 0, torch.zeros_like(X), g))
    if p.payoff == bs.CALL1:
        sq = p.sigma1 * math.sqrt(tau)
        d1 = (torch.log(X.clamp(min=tiny) / p.strike) + (p.r + 0.5 * p.sigma1 ** 2) * tau) / sq
        return torch.where(X <= 0, torch.zeros_like(X),
                           X * ndtr(d1) - p.strike * math.exp(-p.r * tau) * ndtr(d1 - sq))
    st = math.sqrt(tau)
    h = (torch.log(X.clamp(min=tiny) / p.strike) + (p.r - 0.5 * p.sigma1 ** 2) * tau) / (p.sigma1 * st)
    k = (torch.log(Y.clamp(min=tiny) / p.strike2) + (p.r - 0.5 * p.sigma2 ** 2) * tau) / (p.sigma2 * st)
    xg, wg = np.polynomial.legendre.leggauss(64)     # Plackett's identity for the bivariate normal
    acc = ndtr(h) * ndtr(k)
    for x, w in zip(xg, wg):
        t = 0.5 * p.rho * (1 + x)
        om = 1 - t * t
        acc = acc + 0.5 * p.rho * w * torch.exp(-(h * h - 2 * t * h * k + k * k) / (2 * om)) / (
            2 * math.pi * math.sqrt(om))
    return torch.where((X <= 0) | (Y <= 0), torch.zeros_like(X), p.cash * math.exp(-p.r * tau) * acc)


class _Scheme:
    """Implicit Euler with the centred differences on a batch of states, two or three assets.
    ``off`` adds the weighted neighbours of a field padded by one node on every side."""

    def __init__(self, M, xmax, ps, dtau, dims=2):
        self.M, self.n, self.ps, self.dtau, self.dims = M, M - 1, ps, dtau, dims
        idx = torch.arange(M - 1, dtype=torch.float64, device=DEV)
        self.x = torch.arange(M, dtype=torch.float64, device=DEV) * (xmax / (M - 1))
        # axis a (0 = the fastest) lies along tensor dimension -1 - a
        view = lambda v, a: v.view([len(ps)] + [-1 if d == dims - 1 - a else 1 for d in range(dims)])  # noqa: E731
        col = lambda f: torch.tensor([float(f(p)) for p in ps], dtype=torch.float64, device=DEV).view(-1, 1)  # noqa: E731
        self.i = [view(idx.expand(len(ps), -1).contiguous(), a) for a in range(dims)]
        sig = [(lambda p, a=a: p.sigma[a] if dims == 3 else (p.sigma1, p.sigma2)[a]) for a in range(dims)]
        self.hi, self.lo = [], []
        self.diag1 = col(lambda p: dtau * p.r).view([-1] + [1] * dims)     # diagonal minus one
        for a in range(dims):
            dif = view(col(lambda p: 0.5 * dtau * sig[a](p) ** 2) * idx * idx, a)
            dri = view(col(lambda p: 0.5 * dtau * p.r) * idx, a)
            self.hi.append(dif + dri)
            self.lo.append(dif - dri)
            self.diag1 = self.diag1 + 2.0 * dif
        rho = lambda p, a, b: p.rho[{(0, 1): 0, (0, 2): 1, (1, 2): 2}[a, b]] if dims == 3 else p.rho  # noqa: E731
        self.cross = {(a, b): col(lambda p: 0.25 * dtau * rho(p, a, b) * sig[a](p) * sig[b](p)).view([-1] + [1] * dims)
                      * self.i[a] * self.i[b] for a in range(dims) for b in range(a + 1, dims)}

    def _sh(self, P, *moves):
        s = [1] * self.dims
        for a, d in moves:
            s[self.dims - 1 - a] += d
        return P[tuple([slice(None)] + [slice(k, k + self.n) for k in s])]

    def off(self, P):
        acc = torch.zeros_like(self._sh(P))
        for a in range(self.dims):
            acc.addcmul_(self.hi[a], self._sh(P, (a, 1))).addcmul_(self.lo[a], self._sh(P, (a, -1)))
        for (a, b), w in self.cross.items():
            d = self._sh(P, (a, 1), (b, 1)) + self._sh(P, (a, -1), (b, -1))
            acc.addcmul_(w, d.sub_(self._sh(P, (a, 1), (b, -1))).sub_(self._sh(P, (a, -1), (b, 1))))
        return acc

    def pad(self, v):
        return torch.nn.functional.pad(v, [1, 1] * self.dims)

    def A(self, v):
        return v + self.diag1 * v - self.off(self.pad(v))

    def boundary(self, u, taus):
        """u with the far-field data at tau on its far edges."""
        M, x = self.M, self.x
        u = u.clone()
        for b, (p, t) in enumerate(zip(self.ps, taus)):
            if self.dims == 2:
                u[b, M - 1, :] = _far(p, x, x[M - 1], t)
                u[b, :, M - 1] = _far(p, x[M - 1], x, t)
                continue
            c = [x.view([-1 if d == 2 - a else 1 for d in range(3)]) for a in range(3)]
            if p.payoff == bs.BASKET:
                g = torch.clamp(p.w[0] * c[0] + p.w[1] * c[1] + p.w[2] * c[2] - p.strike * math.exp(-p.r * t), min=0.0)
            else:
                q = SimpleNamespace(payoff=bs.EXCHANGE, sigma1=p.sigma[0], sigma2=p.sigma[1], rho=p.rho[0])
                g = _far(q, c[0], c[1], t).expand(M, M, M)
            u[b, M - 1] = g[M - 1]
            u[b, :, M - 1] = g[:, M - 1]
            u[b, :, :, M - 1] = g[:, :, M - 1]
        return u

    def solve(self, rhs, guess, tol=1e-11, maxit=400):
        """A d = rhs by BiCGSTAB on the diagonally scaled system, all states together."""
        inv = 1.0 / (1.0 + self.diag1)
        dims = tuple(range(1, self.dims + 1))
        dot = lambda a, b: (a * b).sum(dims, keepdim=True)                            # noqa: E731
        div = lambda a, b: torch.where(b == 0, torch.zeros_like(a), a / torch.where(b == 0, torch.ones_like(b), b))  # noqa: E731
        b = rhs * inv
        d = guess
        r = b - self.A(d) * inv
        stop = tol * tol * dot(b, b) + 1e-300
        rh, p, rho = r, r, dot(r, r)
        for it in range(maxit):
            if it % 3 == 0 and bool((dot(r, r) <= stop).all()):
                break
            v = self.A(p) * inv
            al = div(rho, dot(rh, v))
            s = r - al * v
            t = self.A(s) * inv
            om = div(dot(t, s), dot(t, t))
            d = d + al * p + om * s
            r = s - om * t
            new = dot(rh, r)
            p = r + div(new, rho) * div(al, om) * (p - om * v)
            rho = new
        return d

    def propagate(self, u, tau0, steps, guess=None):
        n = self.n
        inner = tuple([slice(None)] + [slice(0, n)] * self.dims)
        d1 = torch.zeros_like(u[inner]) if guess is None else guess
        d2 = d1
        for m in range(steps):
            w = self.boundary(u, [t + (m + 1) * self.dtau for t in tau0])
            P = torch.nn.functional.pad(w, [1, 0] * self.dims)
            rhs = self.off(P) - self.diag1 * w[inner]
            d = self.solve(rhs, 2.0 * d1 - d2)
            d1, d2 = d, (d if m == 0 else d1)
            u = w
            u[inner] += d
        return u


def _parareal(u0, F, G, N, tol):
    """Textbook Parareal: F(states, slices) on many slices at once, G(state, slice) on one."""
    norm = lambda v: float(torch.linalg.vector_norm(v))  # noqa: E731
    U, old = [u0], []
    for n in range(N):
        old.append(G(U[n], n))
        U.append(old[n])
    for k in range(N):
        Fk = F(torch.stack(U[k:N]), list(range(k, N)))
        new = list(U[:k + 1])
        for n in range(k, N):
            g = old[n] if n == k else G(new[n], n)
            new.append(Fk[n - k] + (g - old[n]))
            old[n] = g
        num, den = max(norm(a - b) for a, b in zip(new[1:], U[1:])), max(norm(a) for a in new[1:])
        U = new
        if num <= tol * den:
            break
    return torch.stack(U)


def _fno(a, w, mx, my):
    """Fourier neural operator on input channels a [B][9][M][M] in float64."""
    t = {k: torch.tensor(v, device=DEV).to(torch.complex128 if np.iscomplexobj(v) else torch.float64) for k, v in w.items()}
    v = torch.einsum("bcyx,co->boyx", a, t["lift_w"]) + t["lift_b"].view(-1, 1, 1)
    M = a.shape[-1]
    rows = list(range(my)) + list(range(M - my, M))
    for R, W, b in zip(t["spec_w"], t["pw_w"], t["pw_b"]):
        V = torch.fft.rfft2(v)
        out = torch.zeros_like(V)
        out[:, :, rows, :mx] = torch.einsum("bcyx,yxco->boyx", V[:, :, rows, :mx], R)
        v = torch.relu(torch.fft.irfft2(out, s=(M, M)) + torch.einsum("bcyx,co->boyx", v, W) + b.view(-1, 1, 1))
    h = torch.relu(torch.einsum("bcyx,ch->bhyx", v, t["proj1_w"]) + t["proj1_b"].view(-1, 1, 1))
    return torch.einsum("bhyx,h->byx", h, t["proj2_w"]) + t["proj2_b"]


def _resample(u, m):
    """Bilinear interpolation of node fields [B][M][M] to m nodes per axis."""
    M = u.shape[-1]
    if M == m:
        return u
    t = torch.arange(m, dtype=torch.float64, device=DEV) * ((M - 1) / (m - 1))
    i = t.floor().long().clamp(max=M - 2)
    f = t - i
    rows = u[:, i] * (1 - f).view(1, -1, 1) + u[:, i + 1] * f.view(1, -1, 1)
    return rows[:, :, i] * (1 - f) + rows[:, :, i + 1] * f


def exact(case, seed):
    op, M, xmax = case["op"], int(case["M"]), case["xmax"]
    if op == "solve3":
        p, N, T = _options3(case, seed), case["N"], case.get("T", 1.0)
        sl = T / N
        c = [torch.arange(M, dtype=torch.float64, device=DEV).mul(xmax / (M - 1)).view(
            [-1 if d == 2 - a else 1 for d in range(3)]) for a in range(3)]
        f = c[0] - c[1] + 0 * c[2] if p.payoff == bs.EXCHANGE else p.w[0] * c[0] + p.w[1] * c[1] + p.w[2] * c[2] - p.strike
        u0 = torch.clamp(f, min=0.0).expand(M, M, M).contiguous()
        Gs = _Scheme(M, xmax, [p], sl / case["coarse_steps"], 3)

        def F(S, ns):
            fs = _Scheme(M, xmax, [p] * len(ns), sl / case["fine_steps"], 3)
            return fs.propagate(S, [n * sl for n in ns], case["fine_steps"])
        return {"u": _parareal(u0, F, lambda u, n: Gs.propagate(u[None], [n * sl], case["coarse_steps"])[0], N,
                               case["tol"]), "iterations": None}
    if op == "solve":
        (p,), N = _options(case, seed), case["N"]
        sl = p.T / N
        X, Y = _coords(M, xmax)
        f = X - Y if p.payoff == bs.EXCHANGE else p.w1 * X + p.w2 * Y - p.strike
        Gs = _Scheme(M, xmax, [p], sl / case["coarse_steps"])

        def F(S, ns):
            fs = _Scheme(M, xmax, [p] * len(ns), sl / case["fine_steps"])
            return fs.propagate(S, [n * sl for n in ns], case["fine_steps"])
        if M * M * N * case["fine_steps"] > 2 ** 31:     # minutes of 64-bit stepping
            return None
        return {"u": _parareal(torch.clamp(f, min=0.0), F,
                               lambda u, n: Gs.propagate(u[None], [n * sl], case["coarse_steps"])[0], N, case["tol"]),
                "iterations": None}
    ps, tau0 = _items(case, seed)
    B = len(ps)
    if op in ("fine", "coarse"):
        dtau = case["dtau"] if op == "fine" else case["dtau"] / case["steps"]
        # as many of the states as take seconds: each on its own is the same computation
        k = B if op == "coarse" else max(1, min(B, int(2 ** 30 / (M * M * case["steps"]))))
        u = torch.stack([_state(ps[b], M, xmax, tau0[b]) for b in range(k)]).double()
        out = _Scheme(M, xmax, ps[:k], dtau).propagate(u, tau0[:k], case["steps"])
        return out if op == "coarse" else list(out) + [None] * (B - k)
    u = torch.stack([_state(p, M, xmax, t) for p, t in zip(ps, tau0)]).double()
    if op == "physics":
        s = prepare(case, seed)
        pred = s.pred.double().requires_grad_(True)
        sc = _Scheme(M, xmax, ps, case["dtau"])
        P = torch.nn.functional.pad(pred, [1, 0, 1, 0])
        n = M - 1
        r = ((pred - u)[:, :n, :n] - (sc.off(P) - sc.diag1 * pred[:, :n, :n])) / case["dtau"]
        loss = (r * r).sum((1, 2)) / (n * n)
        (grad,) = torch.autograd.grad(loss.sum(), pred)
        return {"loss": loss.detach(), "grad": grad}
    w, Mp = _pino_weights(seed), 128 if M <= 128 else 256
    up = _resample(u, Mp)
    X, Y = _coords(Mp, xmax)
    Xe, Ye = _coords(M, xmax)
    out = torch.empty_like(u)
    for b, (p, t) in enumerate(zip(ps, tau0)):
        one = torch.ones_like(up[b])
        a = torch.stack([up[b], X * one, Y * one, t * one, case["dtau"] * one, p.sigma1 * one, p.sigma2 * one,
                         p.rho * one, p.r * one])
        out[b] = u[b] + _resample(_fno(a[None], w, PINO["modes_x"], PINO["modes_y"]), M)[0]
        out[b, M - 1, :] = _far(p, Xe[0], Xe[0, M - 1], t + case["dtau"])
        out[b, :, M - 1] = _far(p, Xe[0, M - 1], Xe[0], t + case["dtau"])
    return out
