"""Performance cases of the dispersion-curve engine: what a program that uses
it calls, through the Python binding of the C ABI, at the sizes of the
repository's workloads (paper_2003_02256_gb300/workloads.py) and around them.

``listed()`` names the cases, ``draw(rng)`` gives one more of the same ranges,
``prepare(case, seed)`` makes the inputs and the handle a program keeps,
``run(state)`` makes one pass, ``work(case)`` counts what a pass cannot do
without and ``exact(case, seed)`` computes the outputs in plain FP64 torch,
without the library.
"""
from __future__ import annotations

import math
import os
import sys

import numpy as np
import torch

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_2003_02256_gb300 import autograd, masw, serving  # noqa: E402
from paper_2003_02256_gb300 import workloads as W  # noqa: E402

SIGMA = 2.0


def listed():
    return [
        # one theoretical curve (the single-curve workload), host arrays in and
        # out: an analyst trying one model, the smallest call there is
        {"name": "curve", "kind": "curve", "layers": 4, "lambdas": 60},
        # a gradient of a handful of candidate models (a small descent)
        {"name": "descent", "kind": "gradient", "models": 16, "layers": 6, "lambdas": 60},
        # the differentiation workload: 512 candidates, 12 layers, 150
        # wavelengths, misfit and adjoint gradient as torch.autograd gives them
        {"name": "gradient", "kind": "gradient", "models": 512, "layers": 12, "lambdas": 150},
        # one step of 512 Metropolis chains: new (beta, h) on the device, then
        # every chain's least-squares misfit
        {"name": "chains", "kind": "chains", "models": 512, "layers": 12, "lambdas": 150},
        # the uniform batch: 1024 models x 8 layers x 200 wavelengths, curves
        # left on the device
        {"name": "uniform", "kind": "uniform", "models": 1024, "layers": 8, "lambdas": 200},
        # a ragged batch of ordinary size, models uploaded from pinned host
        # memory and curves read back, as an exhaustive search on the host does
        {"name": "search_step", "kind": "search_step", "models": 701},
        # the ragged batch: 8192 models of 3..30 layers, 30..400 wavelengths,
        # 10 % with a low-velocity layer; curves and misfits on the device
        {"name": "ragged", "kind": "ragged", "models": 8192},
        # the first three sign changes of every item (higher modes)
        {"name": "modes", "kind": "modes", "models": 1024, "layers": 8, "lambdas": 200,
         "changes": 3},
        # the leaky continuation on the grid above most fundamental modes
        {"name": "leaky", "kind": "leaky", "models": 256, "layers": 8, "lambdas": 200},
        # models outside the paper's ranges (thin and thick layers, inverted
        # speeds): the counting search's fallback paths carry part of the work
        {"name": "extreme", "kind": "extreme", "models": 1000},
        # continuous batching: a burst of random-walk requests, host to host
        {"name": "serve", "kind": "serve", "requests": 300},
        # the entry point that allocates nothing
        {"name": "noalloc", "kind": "noalloc", "models": 320, "layers": 8, "lambdas": 200},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["curve", "gradient", "chains", "uniform", "search_step", "ragged", "modes",
                       "leaky", "extreme", "serve", "noalloc"])
    if kind == "curve":
        return {"kind": kind, "layers": _log(rng, 1, 30), "lambdas": _log(rng, 20, 400)}
    if kind in ("gradient", "chains"):
        return {"kind": kind, "models": _log(rng, 8, 512), "layers": rng.randint(2, 12),
                "lambdas": rng.randint(20, 150)}
    if kind == "uniform":
        return {"kind": kind, "models": _log(rng, 16, 2048), "layers": rng.randint(3, 12),
                "lambdas": rng.randint(30, 200)}
    if kind == "search_step":
        return {"kind": kind, "models": _log(rng, 50, 2000)}
    if kind == "ragged":
        return {"kind": kind, "models": _log(rng, 200, 8000)}
    if kind == "modes":
        return {"kind": kind, "models": _log(rng, 32, 1000), "layers": rng.randint(3, 8),
                "lambdas": rng.randint(30, 200), "changes": rng.randint(2, 4)}
    if kind == "leaky":
        return {"kind": kind, "models": _log(rng, 16, 256), "layers": rng.randint(3, 8),
                "lambdas": rng.randint(30, 200)}
    if kind == "extreme":
        return {"kind": kind, "models": _log(rng, 64, 1000)}
    if kind == "serve":
        return {"kind": kind, "requests": _log(rng, 8, 300)}
    n_models = _log(rng, 8, 400)
    return {"kind": kind, "models": n_models, "layers": rng.randint(3, 12),
            "lambdas": rng.randint(30, min(200, 65000 // n_models))}


# ------------------------------------------------------------------ inputs

def _vary(models, seed):
    """Other models of the same layer and wavelength counts: the speeds of
    each model scaled by U[0.85, 1.2] and of each layer by 1 + N(0, 0.03^2),
    each thickness by U[0.8, 1.25], the wavelengths with the total thickness."""
    rng = np.random.default_rng(seed)
    owner = np.repeat(np.arange(models.n_models), models.n_layers + 1)
    speed = rng.uniform(0.85, 1.2, models.n_models)[owner]
    speed = speed * (1.0 + 0.03 * np.clip(rng.standard_normal(owner.size), -3.0, 3.0))
    h = models.h * rng.uniform(0.8, 1.25, models.h.size)
    lo = np.concatenate([[0], np.cumsum(models.n_layers)])
    lam = np.concatenate([np.geomspace(1.0, 2.0 * h[lo[m]:lo[m + 1]].sum(), n)
                          for m, n in enumerate(models.n_lambda)])
    return W.Models(models.n_layers, h, models.alpha * speed, models.beta * speed, models.rho,
                    models.n_lambda, lam)


def _inputs(case, seed):
    """(models, grid, C_e) of a case: the workloads' distributions from the
    seed; C_e is 0.92 x the shear speed at a third of the wavelength, smoothed
    over depth, plus N(0, 2^2)."""
    kind = case["kind"]
    seed = int(seed)
    if kind == "curve":
        models, _ = W.uniform_batch(1, case["layers"], case["lambdas"], lam_max=60.0, seed=seed)
        grid = W.Grid(50.0, 0.5, 901)
    elif kind in ("gradient", "chains"):
        models, grid, _ = W.differentiation_batch(case["models"], case["layers"],
                                                  case["lambdas"], seed=seed)
    elif kind in ("uniform", "modes", "noalloc"):
        models, grid = W.uniform_batch(case["models"], case["layers"], case["lambdas"], seed=seed)
    elif kind == "leaky":
        models, _ = W.uniform_batch(case["models"], case["layers"], case["lambdas"], seed=seed)
        grid = W.Grid(700.0, 0.25, 4001)
    elif kind in ("search_step", "ragged"):
        models, grid = W.ragged_batch(case["models"], seed=W.SEED + case["models"])
        models = _vary(models, seed)
    elif kind == "extreme":
        models, grid = W.extreme_batch(case["models"], seed=seed)
    elif kind == "serve":
        sampler = W.RandomWalkSampler(seed=W.SEED + case["requests"], chain_len=8)
        models = W.concat([sampler.next() for _ in range(case["requests"])])
        models = _vary(models, seed)
        grid = W.Grid(50.0, 0.25, 4601)
    else:
        raise ValueError(kind)
    rng = np.random.default_rng(seed + 1)
    ce = np.empty(models.n_items)
    w0 = 0
    for m in range(models.n_models if kind in ("gradient", "chains", "search_step", "ragged") else 0):
        h, _, beta, _, lam = models.model(m)
        mid = np.concatenate([np.cumsum(h) - 0.5 * h, [h.sum() + h[-1]]])
        ce[w0:w0 + lam.size] = 0.92 * np.interp(lam / 3.0, mid, beta)
        w0 += lam.size
    ce += SIGMA * rng.standard_normal(models.n_items) if w0 else 0.0
    return models, grid, ce


def _pinned(a, dtype=np.float64):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=dtype)).pin_memory()


def prepare(case, seed):
    models, grid, ce = _inputs(case, seed)
    kind = case["kind"]
    st = {"kind": kind, "models": models, "grid": grid}
    n, M = models.n_items, models.n_models
    f64, i32 = torch.float64, torch.int32
    if kind == "serve":
        st["server"] = serving.Server(grid, max_slots=512)
        st["arrivals"] = np.zeros(case["requests"])
        return st
    if kind == "noalloc":
        st["args"] = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in
                      (models.n_layers, models.h, models.alpha, models.beta, models.rho,
                       models.n_lambda, models.lam)]
    else:
        st["batch"] = masw.Batch(models, grid)
    if kind == "curve":
        return st
    if kind in ("gradient", "chains"):
        st["beta"] = torch.from_numpy(models.beta).cuda().requires_grad_(kind == "gradient")
        st["h"] = torch.from_numpy(models.h).cuda().requires_grad_(kind == "gradient")
        st["ce"] = torch.from_numpy(ce).cuda()
        st["phi"] = torch.empty(M, dtype=f64, device="cuda")
        return st
    if kind == "search_step":
        st["up"] = [_pinned(a) for a in (models.h, models.alpha, models.beta, models.rho)]
        st["ce"] = _pinned(ce)
        make = lambda size, dt: torch.empty(size, dtype=dt, pin_memory=True)  # noqa: E731
    else:
        st["ce"] = torch.from_numpy(ce).cuda() if kind == "ragged" else None
        make = lambda size, dt: torch.empty(size, dtype=dt, device="cuda")  # noqa: E731
    st["phi"] = make(M, f64)
    per = case.get("changes", 1)
    st["out"] = {"ct": make(n * per, f64), "idx": make(n * per, i32), "status": make(n * per, i32)}
    if kind == "modes":
        st["changes"] = per
        st["out"]["delta"] = make(n * per, i32)
    return st


def run(st):
    kind = st["kind"]
    if kind == "curve":
        ct, idx, status = st["batch"].dispersion()
        return {"ct": ct, "idx": idx, "status": status}
    if kind == "serve":
        _, ct, idx, status, _ = st["server"].run_trace(st["models"], st["arrivals"])
        return {"ct": ct, "idx": idx, "status": status}
    if kind == "gradient":
        phi = autograd.misfit(st["beta"], st["h"], st["batch"], st["ce"], masw.MISFIT_LSQ, SIGMA)
        gb, gh = torch.autograd.grad(phi.sum(), (st["beta"], st["h"]))
        return {"phi": phi.detach(), "grad_beta": gb, "grad_h": gh}
    if kind == "chains":
        masw.model_batch_update_beta_h(st["batch"].handle, st["h"], st["beta"])
        masw.misfit(st["batch"].handle, st["ce"], masw.MISFIT_LSQ, SIGMA, st["phi"])
        return {"phi": st["phi"]}
    o = st["out"]
    if kind == "noalloc":
        g = st["grid"]
        masw.dispersion_noalloc(*st["args"], (g.c0, g.dc, g.n_c), o["ct"], o["idx"], o["status"])
        return o
    handle = st["batch"].handle
    if kind in ("uniform", "extreme"):
        masw.dispersion(handle, o["ct"], o["idx"], o["status"])
    elif kind == "leaky":
        masw.dispersion_leaky(handle, o["ct"], o["idx"], o["status"])
    elif kind == "modes":
        masw.dispersion_changes(handle, st["changes"], o["ct"], o["idx"], o["status"], o["delta"])
    else:
        if kind == "search_step":
            masw.model_batch_update(handle, *st["up"])
        masw.misfit_curves(handle, st["ce"], masw.MISFIT_PAPER, 1.0, st["phi"], o["ct"], o["idx"],
                           o["status"])
        return {"phi": st["phi"], **o}
    return o


# -------------------------------------------------------------------- work

# FP64 flops of one layer-evaluation (one layer's element stiffness and its
# elimination step)
EVAL_FLOPS = 149


def work(case):
    """Each input read once and each output written once; layer-evaluations:
    two per layer and reported change (the points on its two sides decide
    it), and for the gradient two more at the refined root plus four for its
    derivatives. The ragged kinds count their distributions' means."""
    kind = case["kind"]
    models = case.get("models", case.get("requests", 1))
    if kind in ("search_step", "ragged", "serve"):
        layers, lambdas = 16.5, 215.0
    elif kind == "extreme":
        layers, lambdas = 15.5, 32.0
    else:
        layers, lambdas = case["layers"], case["lambdas"]
    items = models * lambdas
    evals, out = 2 * case.get("changes", 1), 16 * case.get("changes", 1)
    if kind == "modes":
        out = 20 * case["changes"]
    if kind in ("gradient", "chains"):
        out = 8  # C_e read
    if kind in ("search_step", "ragged"):
        out += 8
    if kind == "gradient":
        evals = 8
    par = 8 * (4 * layers + 3) * models
    return {"bytes": int(par + (8 + out) * items + 8 * models),
            "flops": int(evals * (layers + 1) * items * EVAL_FLOPS)}


# ------------------------------------------------------- plain FP64 outputs

class _Exact:
    """Algorithm 1 in FP64 torch for a ragged batch: items padded to the most
    layers (a padding layer is skipped), the 2 x 2 block elimination of the
    stiffness matrix, signs at every grid point until the wanted changes."""

    def __init__(self, models, grid):
        self.dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        self.grid = grid
        M = models.n_models
        nl = models.n_layers.astype(np.int64)
        L = max(int(nl.max()), 1)
        loff = np.concatenate([[0], np.cumsum(nl + 1)])
        hoff = np.concatenate([[0], np.cumsum(nl)])
        par = np.ones((4, M, L + 1))
        for m in range(M):
            n = nl[m]
            par[0, m, :n] = models.h[hoff[m]:hoff[m + 1]]
            for q, a in enumerate((models.alpha, models.beta, models.rho)):
                par[q + 1, m, :n] = a[loff[m]:loff[m] + n]
                par[q + 1, m, L] = a[loff[m] + n]  # half-space last
        t = lambda a: torch.as_tensor(a, device=self.dev)  # noqa: E731
        self.h, self.alpha, self.beta, self.rho = (t(p) for p in par)
        self.nl, self.L = t(nl), L
        self.im = t(np.repeat(np.arange(M), models.n_lambda))
        self.k = 2.0 * math.pi / t(np.ascontiguousarray(models.lam))
        # grid points below the half-space shear speed
        v = grid.c0 + grid.dc * np.arange(grid.n_c)
        self.nlim = t(np.searchsorted(v, models.beta[loff[1:] - 1], side="left"))

    @staticmethod
    def wave(kh, w2):
        """(E, C, Sd, Sm) = e^-x (1, cosh x, sinh(x)/w, w sinh x) for real w,
        (1, cos, sin/w, -w sin) for imaginary w."""
        w = w2.abs().sqrt().clamp_min(1e-9)
        x = kh * w
        real = w2 > 0
        e = torch.where(real, torch.exp(-x), torch.ones_like(x))
        e2 = torch.where(real, torch.exp(-2 * x), torch.ones_like(x))
        s = torch.where(real, -0.5 * torch.expm1(-2 * x), torch.sin(x))
        c = torch.where(real, 0.5 + 0.5 * e2, torch.cos(x))
        return e, c, s / w, torch.where(real, s * w, -s * w)

    def element(self, k, c, h, alpha, beta, rho):
        """The seven entries (A, B, D, E, F, G) of a layer's stiffness over k."""
        c2 = c * c
        q = c2 / (beta * beta)
        r2, s2 = 1 - c2 / (alpha * alpha), 1 - q
        er, cr, sdr, smr = self.wave(k * h, r2)
        es, cs, sds, sms = self.wave(k * h, s2)
        u = er * es - cr * cs
        ss = sdr * sds
        d = 2 * u + smr * sms + ss
        rc2, mu = rho * c2 / d, rho * beta * beta / d
        b1 = -(s2 + 3) * u - sms * (2 * smr + sdr) - ss
        return (rc2 * (cr * sds - cs * smr), mu * b1, rc2 * (cs * sdr - cr * sms),
                rc2 * (smr * es - er * sds), rc2 * (er * cs - cr * es), rc2 * (sms * er - es * sdr))

    def half(self, c, alpha, beta, rho, leaky):
        """The half-space block over k: (h00, h01, h11), complex with leaky."""
        c2 = c * c
        q, p = c2 / (beta * beta), c2 / (alpha * alpha)
        if leaky:
            s = torch.sqrt((1 - q).to(torch.complex128))
            r = torch.sqrt((1 - p).to(torch.complex128))
            den = 1 - r * s
        else:
            s, r = torch.sqrt(1 - q), torch.sqrt(1 - p)
            den = (p + q - p * q) / (1 + r * s)
        return rho * c2 * r / den, rho * beta * beta * (q - 2 * den) / den, rho * c2 * s / den

    def eliminate(self, items, c):
        """(sign of the finite layers' pivots, P00, P01, P11) at c for items."""
        im = self.im[items]
        h, alpha, beta, rho = self.h, self.alpha, self.beta, self.rho
        k, n = self.k[items], self.nl[im]
        p00 = torch.zeros_like(c)
        p01, p11, sg = p00, p00, torch.ones_like(c)
        for j in range(self.L):
            A, B, D, E, F, G = self.element(k, c, h[im, j], alpha[im, j], beta[im, j], rho[im, j])
            s00, s01, s11 = p00 + A, p01 + B, p11 + D
            det = s00 * s11 - s01 * s01
            t00, t01 = (s11 * E + s01 * F) / det, (s11 * F - s01 * G) / det
            t10, t11 = -(s01 * E + s00 * F) / det, (s00 * G - s01 * F) / det
            on = j < n
            p00 = torch.where(on, A - (E * t00 - F * t10), p00)
            p01 = torch.where(on, -B - (E * t01 - F * t11), p01)
            p11 = torch.where(on, D - (F * t01 + G * t11), p11)
            sg = torch.where(on, sg * torch.sign(det), sg)
        return sg, p00, p01, p11

    def last(self, items, c, p, leaky):
        """det of the last pivot (its real part with leaky)."""
        im = self.im[items]
        alpha, beta, rho = self.alpha, self.beta, self.rho
        h00, h01, h11 = self.half(c, alpha[im, self.L], beta[im, self.L], rho[im, self.L], leaky)
        det = (p[0] + h00) * (p[2] + h11) - (p[1] + h01) ** 2
        return det.real if leaky else det

    def sign(self, items, c, leaky):
        sg, *p = self.eliminate(items, c)
        return (sg * torch.sign(self.last(items, c, p, leaky))).to(torch.int8)

    def changes(self, count=1, leaky=False):
        """[n_items, count] grid indices of the first sign changes, -1: none."""
        n_items = self.k.numel()
        found = torch.full((n_items, count), -1, dtype=torch.int64, device=self.dev)
        got = torch.zeros(n_items, dtype=torch.int64, device=self.dev)
        lim = torch.full_like(got, self.grid.n_c) if leaky else self.nlim[self.im]
        prev = torch.zeros(n_items, dtype=torch.int8, device=self.dev)
        live = torch.nonzero(lim >= 2).flatten()
        base = 0
        while live.numel():
            width = max(1, min(256, (1 << 22) // live.numel()))
            n = base + torch.arange(width, device=self.dev)
            it = live.repeat_interleave(width)
            nn = n.repeat(live.numel())
            keep = nn < lim[it]
            sg = torch.zeros(it.numel(), dtype=torch.int8, device=self.dev)
            at, where = it[keep], nn[keep].to(torch.float64)
            sg[keep] = self.sign(at, self.grid.c0 + self.grid.dc * where, leaky)
            sg = sg.view(live.numel(), width)
            before = torch.cat([prev[live].unsqueeze(1), sg[:, :-1]], 1)
            change = (sg != before) & keep.view_as(sg) & (n >= 1)
            rank = got[live].unsqueeze(1) + torch.cumsum(change, 1)
            row, col = torch.nonzero(change & (rank <= count), as_tuple=True)
            found[live[row], rank[row, col] - 1] = n[col]
            got[live] += change.sum(1)
            prev[live] = sg[:, -1]
            base += width
            live = live[(got[live] < count) & (lim[live] > base)]
        return found

    def speeds(self, index):
        v = self.grid.c0 + self.grid.dc * index.to(torch.float64)
        return torch.where(index >= 1, v, torch.full_like(v, float("nan")))

    def per_model(self, values):
        out = torch.zeros(self.nl.numel(), dtype=torch.float64, device=self.dev)
        return out.index_add_(0, self.im, values)

    def refined(self, index):
        """The root inside each bracket [V[index-1], V[index]], by bisection."""
        items = torch.arange(index.numel(), device=self.dev)
        lo, hi = self.speeds(index) - self.grid.dc, self.speeds(index)
        s_lo = self.sign(items, lo, False)
        for _ in range(52):
            mid = 0.5 * (lo + hi)
            same = self.sign(items, mid, False) == s_lo
            lo, hi = torch.where(same, mid, lo), torch.where(same, hi, mid)
        return 0.5 * (lo + hi)

    def mode_shape(self, c):
        """The null vector of each item's K(c) at its root, by inverse
        iteration on the dense matrix (all models with as many layers)."""
        n, L = c.numel(), self.L
        items = torch.arange(n, device=self.dev)
        K = torch.zeros(n, 2 * L + 2, 2 * L + 2, dtype=torch.float64, device=self.dev)
        im = self.im[items]
        for j in range(L):
            A, B, D, E, F, G = self.element(self.k, c, self.h[im, j], self.alpha[im, j],
                                            self.beta[im, j], self.rho[im, j])
            rows = [[A, B, E, F], [B, D, -F, G], [E, -F, A, -B], [F, G, -B, D]]
            K[:, 2 * j:2 * j + 4, 2 * j:2 * j + 4] += torch.stack(
                [torch.stack(r, -1) for r in rows], -2)
        h00, h01, h11 = self.half(c, self.alpha[im, L], self.beta[im, L], self.rho[im, L], False)
        K[:, 2 * L:, 2 * L:] += torch.stack([torch.stack([h00, h01], -1),
                                             torch.stack([h01, h11], -1)], -2)
        lu = torch.linalg.lu_factor(K)
        u = torch.cos(torch.arange(2.0 * L + 2, dtype=torch.float64, device=self.dev))
        u = u.expand(n, -1).unsqueeze(-1)
        for _ in range(4):
            u = torch.linalg.lu_solve(*lu, u)
            u = u / u.abs().amax(1, keepdim=True)
        return u[..., 0]

    def gradient(self, ce):
        """(phi, dphi/dbeta, dphi/dh) of the least-squares misfit at the
        refined roots: dC/dtheta = -(u' dK/dtheta u) / (u' dK/dc u), u the null
        vector of K, with alpha/beta and rho held."""
        root = self.refined(self.changes(1)[:, 0])
        u = self.mode_shape(root)
        c = root.clone().requires_grad_(True)
        h = self.h.clone().requires_grad_(True)
        beta = self.beta.clone().requires_grad_(True)
        alpha, im, L = beta * (self.alpha / self.beta), self.im, self.L
        form = 0.0
        for j in range(L):
            A, B, D, E, F, G = self.element(self.k, c, h[im, j], alpha[im, j], beta[im, j],
                                            self.rho[im, j])
            x0, z0, x1, z1 = (u[:, 2 * j + q] for q in range(4))
            form = form + ((x0 * x0 + x1 * x1) * A + (z0 * z0 + z1 * z1) * D +
                           2 * (x0 * z0 - x1 * z1) * B + 2 * x0 * x1 * E +
                           2 * (x0 * z1 - z0 * x1) * F + 2 * z0 * z1 * G)
        h00, h01, h11 = self.half(c, alpha[im, L], beta[im, L], self.rho[im, L], False)
        x, z = u[:, 2 * L], u[:, 2 * L + 1]
        form = form + x * x * h00 + 2 * x * z * h01 + z * z * h11
        (fc,) = torch.autograd.grad(form.sum(), c, retain_graph=True)
        weight = -((root - ce) / (SIGMA * SIGMA)) / fc
        gb, gh = torch.autograd.grad(form, (beta, h), weight.detach())
        phi = self.per_model((root - ce) ** 2) / (2 * SIGMA * SIGMA)
        return phi, gb.flatten(), gh[:, :L].flatten()


def exact(case, seed):
    kind = case["kind"]
    if kind == "ragged" and case["models"] > 1500:
        return None  # some 27 G FP64 layer-evaluations for 8192 models
    models, grid, ce = _inputs(case, seed)
    ex = _Exact(models, grid)
    ce = torch.as_tensor(ce, device=ex.dev)
    host = lambda x: x.cpu().numpy() if isinstance(x, torch.Tensor) else x  # noqa: E731
    if kind == "gradient":
        phi, gb, gh = ex.gradient(ce)
        return {"phi": host(phi), "grad_beta": host(gb), "grad_h": host(gh)}
    index = ex.changes(case.get("changes", 1), leaky=kind == "leaky")
    ct = ex.speeds(index)
    if kind == "chains":
        return {"phi": host(ex.per_model((ct[:, 0] - ce) ** 2) / (2 * SIGMA * SIGMA))}
    out = {"ct": host(ct.flatten()), "idx": None, "status": None}
    if kind == "modes":
        out["delta"] = None
    if kind in ("search_step", "ragged"):
        n = torch.as_tensor(models.n_lambda, device=ex.dev)
        out["phi"] = host(ex.per_model((ct[:, 0] - ce).abs() / ce) / n)
    return out
