"""The work that users of this framework have it do, as timed cases.

Every case is a dict of plain values.  `listed()` names twelve of them, `draw(rng)` gives more of the same ranges,
`prepare` makes what a user's program holds before the call (initial fields, a Solver or an Ensemble), `run` is one
pass through the public entry points, `work` what such a pass cannot do without, and `exact` the same outputs from
plain torch and numpy in 64 bits: the asynchrony-tolerant step written out with rolls and concatenations, its delays
from a separate Philox, its gradient by torch's own differentiation.

Kinds of case:
  step        Solver.reset(u0), Solver.step(n): a time-stepping run from a caller's field (1D or 3D; forward Euler or
              Adams-Bashforth; advection-diffusion or Burgers; any order and PE split, with or without the delay log)
  ensemble    Ensemble.run(): many delay realizations of the 1D problem at once, fields and statistics of each
  gradient    at_forward(...) and backward(): the gradient of a misfit in the initial field and the diffusivity
  statistics  Solver.reset(u), error_stats(), reset(): error measures of a field against the analytic solution, and
              the initial condition written anew
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1702_00496_gb300 import Ensemble, Solver, at_forward

SYNC, ASYNC_STD, AT = 0, 1, 2
TWO_PI = 2.0 * math.pi
LARGEST = 512 ** 3 * 13 * 10  # tap evaluations of the largest listed case; a drawn case has at most as many
COMMON = {"scheme": AT, "tsteps": 1, "burgers": False, "binned": False, "log": False, "c": 1.0, "r_alpha": 0.1}


# ------------------------------------------------------------------ the cases
def listed():
    def case(name, kind, **kw):
        return {"name": name, "kind": kind, **COMMON, **kw}

    return [
        # the smallest runs: a textbook grid, one launch after another; latency is all there is
        case("1d_small", "step", nx=256, px=8, order=2, L=3, modes=4, steps=400, log=True),
        # an ordinary 1D study: a few hundred cells per PE, every delay logged for replay
        case("1d_ordinary", "step", nx=12000, px=30, order=4, L=4, modes=10, steps=300, log=True),
        # the large 1D run: 4096 PEs of 4096 cells, fourth order, four delay levels
        case("1d_large", "step", nx=1 << 24, px=4096, order=4, L=4, modes=10, steps=96),
        # PEs whose width is no multiple of four
        case("1d_ragged", "step", nx=750000, px=3000, order=4, L=3, modes=6, steps=50, binned=True),
        # the paper's Case 4 at scale: Adams-Bashforth 2, fourth order
        case("1d_ab2", "step", nx=1 << 24, px=4096, order=4, L=3, modes=3, steps=40, tsteps=2, r_alpha=0.05),
        # the paper's Case 5: diffusion, Adams-Bashforth 3, sixth order
        case("1d_ab3", "step", nx=1 << 22, px=1024, order=6, L=3, modes=3, steps=100, tsteps=3, c=0.0, r_alpha=0.01),
        # the paper's Case 6: the viscous Burgers' equation
        case("1d_burgers", "step", nx=1 << 22, px=1024, order=4, L=3, modes=3, steps=60, tsteps=2, burgers=True, c=0.0,
             r_alpha=0.05),
        # the 3D production run: 512^3 points in 8^3 PEs, fourth order
        case("3d_large", "step", nx=512, ny=512, nz=512, px=8, py=8, pz=8, order=4, L=3, modes=3, steps=10,
             r_alpha=0.05),
        # a 3D box that fits no tile: odd PE widths on every axis, second order
        case("3d_ragged", "step", nx=150, ny=126, nz=90, px=3, py=3, pz=2, order=2, L=3, modes=3, steps=40,
             r_alpha=0.05, log=True),
        # averages over delay realizations: a thousand members of many sizes
        case("ensemble", "ensemble", count=1024, lo=10, hi=16, width=64, order=4, modes=4, steps=250),
        # fitting an initial field and a diffusivity to a target
        case("gradient_3d", "gradient", nx=128, ny=128, nz=128, px=2, py=2, pz=2, order=4, L=3, modes=3, steps=40,
             r_alpha=0.05),
        # error measures of a large field, and its initial condition
        case("statistics", "statistics", nx=1 << 24, px=4096, order=4, L=4, modes=10),
    ]


def _spread(rng, lo, hi):
    """A whole number of lo..hi, spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["step1", "step3", "ensemble", "gradient", "statistics"], [10, 5, 2, 2, 1])[0]
    order = rng.choice([2, 4, 4, 6])
    L = rng.randint(1, 6)
    c = dict(COMMON, order=order, L=L, modes=rng.randint(2, 10), binned=rng.random() < 0.3, log=rng.random() < 0.3,
             scheme=rng.choice([AT, AT, AT, ASYNC_STD, SYNC]))
    r = {2: 0.08, 4: 0.04, 6: 0.01}[order]
    if kind == "ensemble":
        lo = rng.randint(8, 11)
        hi = lo + rng.randint(0, 4)
        count = _spread(rng, 40, 1200)
        c.update(kind="ensemble", count=count, lo=lo, hi=hi, width=rng.choice([16, 32, 64, 128]), scheme=AT,
                 order=min(order, 4), binned=False, log=False, r_alpha=r)
        c.pop("L")
        c["steps"] = _spread(rng, 20, min(1500, max(30, LARGEST // (12 * count << hi))))
        return c
    if kind in ("step1", "statistics"):
        px = _spread(rng, 2, 6000)
        width = max(order, _spread(rng, 8, min(60000, (1 << 24) // px)))
        if rng.random() < 0.7:
            width = (width + 3) // 4 * 4
        c.update(nx=px * width, px=px)
        if kind == "statistics":
            c.update(kind="statistics", scheme=AT, log=False)
            return c
        c["tsteps"] = rng.choice([1, 1, 1, 2, 3])
        c["burgers"] = rng.random() < 0.15
        c["c"] = 0.0 if c["burgers"] else rng.choice([0.0, 1.0, -0.7])
        c["r_alpha"] = min(r, {1: r, 2: 0.04, 3: 0.01}[c["tsteps"]])
        most = LARGEST // 2 // (c["nx"] * (2 * order + 1))
        c.update(kind="step", steps=max(4, min(500, _spread(rng, 20, 500), most)))
        return c
    dims, splits = [], []
    for _ in range(3):
        p = rng.randint(1, 5)
        w = max(order, _spread(rng, 8, 80 if kind == "step3" else 32))
        if rng.random() < 0.6:
            w = (w + 3) // 4 * 4
        dims.append(p * w)
        splits.append(p)
    c.update(nx=dims[0], ny=dims[1], nz=dims[2], px=splits[0], py=splits[1], pz=splits[2], c=rng.choice([1.0, 0.3]),
             r_alpha=min(r, 0.04), kind="step" if kind == "step3" else "gradient")
    most = LARGEST // (dims[0] * dims[1] * dims[2] * (3 * order + 1))
    if kind == "gradient":
        c.update(log=False, steps=max(4, min(60, most // 4, _spread(rng, 8, 60))))
    else:
        c["tsteps"] = rng.choice([1, 1, 1, 2])
        c["steps"] = max(3, min(80, most, _spread(rng, 6, 80)))
    return c


# ------------------------------------------------------------------ inputs
def _dims(case):
    return [case["nx"], case.get("ny", 1), case.get("nz", 1)], [case["px"], case.get("py", 1), case.get("pz", 1)]


def _probs(L):
    p = np.array([1.0 / (m + 1.0) for m in range(L)])
    return p / p.sum()


def _spec(case, seed):
    """The problem as Solver takes it: the case's sizes, amplitudes, phases and delay key from the seed."""
    n, pe = _dims(case)
    dim = 3 if "ny" in case else 1
    rng = np.random.default_rng([seed, 7])
    dx = TWO_PI / max(n)
    alpha = 0.05 if dim == 3 else 0.1
    m = case["modes"]
    L = case["L"]
    thr = None
    if case["binned"] and L > 1:
        thr = np.array([min(int(round(v * 2.0 ** 32)), 2 ** 32) for v in np.cumsum(_probs(L))[:-1]], dtype=np.uint64)
    spec = {"dim": dim, "n": n[:dim], "pe": pe[:dim], "order": case["order"], "L": L, "scheme": case["scheme"],
            "c": [case["c"]] * dim, "alpha": alpha, "dt": case["r_alpha"] * dx * dx / alpha, "seed": 1000 + seed,
            "tsteps": case["tsteps"], "thresholds": thr, "nmodes": m, "amp": rng.uniform(0.5, 1.0, (dim, m)),
            "phase": rng.uniform(0.0, TWO_PI, (dim, m)), "kappa": np.tile(np.arange(1, m + 1, dtype=np.int32), (dim, 1))}
    if case["burgers"]:
        spec["burgers"] = 1
    return spec


def _initial(spec, device="cuda"):
    """The multi-sine field of the spec on its grid: the product over the axes of sum A sin(kappa x + phi)."""
    axes = []
    for a in range(spec["dim"]):
        x = torch.arange(spec["n"][a], dtype=torch.float64, device=device) * (TWO_PI / spec["n"][a])
        s = torch.zeros_like(x)
        for A, ph, k in zip(spec["amp"][a], spec["phase"][a], spec["kappa"][a]):
            s = s + float(A) * torch.sin(float(k) * x + float(ph))
        axes.append(s)
    if spec["dim"] == 1:
        return axes[0]
    return axes[2][:, None, None] * axes[1][None, :, None] * axes[0][None, None, :]


def _perturbed(spec, seed):
    """A field near the analytic one, as a measured or a coarse run's field is."""
    u = _initial(spec)
    g = torch.Generator(device="cuda").manual_seed(seed)
    return u + 1e-3 * torch.randn(u.shape, dtype=torch.float64, device="cuda", generator=g)


def _members(case, seed):
    """Specs of the ensemble's members: sizes 2^lo..2^hi, delay ranges 2..4, phases and keys of their own."""
    rng = np.random.default_rng([seed, 11])
    size = np.random.default_rng([case["count"], case["lo"], case["hi"]])  # sizes belong to the case, not to the seed
    out = []
    for r in range(case["count"]):
        n = 1 << int(size.integers(case["lo"], case["hi"] + 1))
        out.append({"dim": 1, "n": [n], "pe": [max(1, n // case["width"])], "order": case["order"],
                    "L": int(size.integers(2, 5)), "scheme": AT, "c": [1.0], "alpha": 0.1,
                    "dt": case["r_alpha"] * (TWO_PI / n) ** 2 / 0.1, "seed": 1000 * seed + r, "tsteps": 1,
                    "thresholds": None, "nmodes": case["modes"], "amp": rng.uniform(0.5, 1.0, (1, case["modes"])),
                    "phase": rng.uniform(0.0, TWO_PI, (1, case["modes"])),
                    "kappa": np.arange(1, case["modes"] + 1, dtype=np.int32)[None, :]})
    return out


def prepare(case, seed):
    if case["kind"] == "ensemble":
        specs = _members(case, seed)
        return {"case": case, "ens": Ensemble(specs, case["steps"])}
    spec = _spec(case, seed)
    if case["kind"] == "gradient":
        u0 = _initial(spec)
        target = _initial(_spec(case, seed + 500)) * 0.8
        alpha = torch.tensor(spec["alpha"], dtype=torch.float64, device="cuda")
        return {"case": case, "spec": spec, "u0": u0, "alpha": alpha, "target": target}
    if case["kind"] == "statistics":
        return {"case": case, "solver": Solver(spec), "u0": _perturbed(spec, seed)}
    return {"case": case, "solver": Solver(spec, log_steps=case["steps"] if case["log"] else 0), "u0": _initial(spec)}


def run(state):
    case = state["case"]
    if case["kind"] == "ensemble":
        ens = state["ens"]
        ens.run()
        members, _ = ens.stats()
        # the members' errors themselves are not compared: after so few steps on the larger grids they are differences
        # at the rounding level of the fields, which are returned whole
        fields = torch.cat([ens.field(r) for r in range(case["count"])])
        return {"fields": fields, "ua_rms": np.array([m["ua_rms"] for m in members])}
    if case["kind"] == "gradient":
        u0 = state["u0"].detach().requires_grad_(True)
        alpha = state["alpha"].detach().requires_grad_(True)
        u = at_forward(u0, alpha, state["spec"], case["steps"])
        loss = 0.5 * ((u - state["target"]) ** 2).sum()
        loss.backward()
        return {"u": u.detach(), "grad_u0": u0.grad, "grad_alpha": alpha.grad}
    s = state["solver"]
    s.reset(state["u0"])
    if case["kind"] == "statistics":
        st = s.error_stats()
        s.reset()
        return {"stats": {k: float(st[k]) for k in ("rms", "max_abs", "mean_abs", "rms_I", "rms_B", "ua_rms")},
                "points": [int(st["n_I"]), int(st["n_B"])], "field": s.field()}
    s.step(case["steps"])
    return {"field": s.field(), "delays": s.delays()} if case["log"] else {"field": s.field()}


def work(case):
    """Each point's taps once per step (a multiply and an add each), plus one of each per Adams-Bashforth level;
    the initial field read and the result written once."""
    if case["kind"] == "ensemble":
        cells = sum(s["n"][0] for s in _members(case, 0))
        return {"bytes": 8 * cells, "flops": cells * case["steps"] * (4 * (case["order"] // 2) + 1)}
    n, _ = _dims(case)
    cells = n[0] * n[1] * n[2]
    taps = (3 if "ny" in case else 1) * case["order"] + 1
    if case["kind"] == "statistics":
        # a sine and a cosine term per mode for the analytic value, twice (the statistics, the initial condition)
        return {"bytes": 16 * cells, "flops": cells * (8 * case["modes"] + 16)}
    per = 2 * taps - 1 + (2 * case["tsteps"] if case["tsteps"] > 1 else 0)
    if case["burgers"]:
        per += 2 * case["order"] + 2
    if case["kind"] == "gradient":
        # the forward pass, the transposed taps and the second-derivative taps of the diffusivity's derivative
        return {"bytes": 32 * cells, "flops": cells * case["steps"] * (3 * per + 2)}
    return {"bytes": 16 * cells, "flops": cells * case["steps"] * per}


# ------------------------------------------------------------------ the same in 64 bits, from plain torch and numpy
CD1 = {2: [-1 / 2, 0.0, 1 / 2], 4: [1 / 12, -2 / 3, 0.0, 2 / 3, -1 / 12],
       6: [-1 / 60, 3 / 20, -3 / 4, 0.0, 3 / 4, -3 / 20, 1 / 60]}
CD2 = {2: [1.0, -2.0, 1.0], 4: [-1 / 12, 4 / 3, -5 / 2, 4 / 3, -1 / 12],
       6: [1 / 90, -3 / 20, 3 / 2, -49 / 18, 3 / 2, -3 / 20, 1 / 90]}
BETA = {1: [1.0], 2: [1.5, -0.5], 3: [23 / 12, -16 / 12, 5 / 12]}


def _philox(step, sides, seed):
    """First word of Philox4x32-10 at counter (step, side, 0, 0) under the 64-bit key (numpy, all sides at once)."""
    mask, m0, m1 = np.uint64(0xFFFFFFFF), np.uint64(0xD2511F53), np.uint64(0xCD9E8D57)
    c = [np.full(sides.shape, step, np.uint64), sides.astype(np.uint64), np.zeros(sides.shape, np.uint64),
         np.zeros(sides.shape, np.uint64)]
    k0, k1 = seed & mask, seed >> np.uint64(32)
    for _ in range(10):
        p0, p1 = c[0] * m0, c[2] * m1
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ k0, p1 & mask, (p0 >> np.uint64(32)) ^ c[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & mask, (k1 + np.uint64(0xBB67AE85)) & mask
    return c[0]


def _extrapolation(T, k):
    """Weights of levels n-k, n-k-1, ... for the value at level n: the polynomial through T of them."""
    w = []
    for m in range(T):
        v = 1.0
        for q in range(T):
            if q != m:
                v *= (k + q) / float(q - m)
        w.append(v)
    return w


class _Exact:
    """The step of B problems of one shape, fields as [B, nz, ny, nx]."""

    def __init__(self, specs, alpha=None, dev="cuda"):
        s = specs[0]
        self.order, self.L, self.scheme = s["order"], s["L"], s["scheme"]
        self.h, self.dim, self.dev = self.order // 2, s["dim"], dev
        self.n = list(s["n"]) + [1] * (3 - self.dim)
        self.pe = list(s["pe"]) + [1] * (3 - self.dim)
        self.T = self.order // 2 + 1 if self.scheme == AT else 1
        self.ts, self.burgers, self.thr = max(1, s["tsteps"]), bool(s.get("burgers", 0)), s["thresholds"]
        self.seed = np.array([t["seed"] for t in specs], dtype=np.uint64)[:, None]
        self.sides = np.arange(2 * self.dim * self.pe[0] * self.pe[1] * self.pe[2])[None, :].repeat(len(specs), 0)
        col = lambda f: torch.tensor([f(t) for t in specs], dtype=torch.float64, device=dev).view(-1, 1, 1, 1)  # noqa: E731
        al = col(lambda t: t["alpha"]) if alpha is None else alpha
        dt = col(lambda t: t["dt"])
        self.b1, self.b2, self.taps = [], [], []
        for a in range(self.dim):
            dx = TWO_PI / self.n[a]
            d1, d2 = CD1[self.order], CD2[self.order]
            self.b1.append([dt * v / dx for v in d1])
            self.b2.append([dt * al * v / (dx * dx) for v in d2])
            self.taps.append([dt * (-col(lambda t: t["c"][a]) * p / dx + al * q / (dx * dx)) for p, q in zip(d1, d2)])

    def delays(self, n):
        """(raw, effective) delays of step n, [B, sides]."""
        if self.scheme == SYNC:
            z = np.zeros(self.sides.shape, np.int64)
            return z, z
        x = _philox(n, self.sides, self.seed)
        if self.thr is None:
            raw = (x * np.uint64(self.L)) >> np.uint64(32)
        else:
            raw = sum(((x >= t).astype(np.int64) for t in self.thr), np.zeros(x.shape, np.int64))
        raw = raw.astype(np.int64)
        return raw, np.where(raw > 0, np.minimum(raw, max(0, n - (self.T - 1))), 0)

    def padded(self, levels, n, a, keff):
        """U^n split along axis a into PEs, each with its buffer points: [.., P, h + S + h, ..] from dimension 3 - a."""
        d, P, h = 3 - a, self.pe[a], self.h
        S = self.n[a] // P

        def halo(level, hi):
            v = level.unflatten(d, (P, S))
            return v.roll(-1 if hi else 1, d).narrow(d + 1, 0 if hi else S - h, h)

        out = []
        for hi in (0, 1):
            v = halo(levels[n], hi)
            if P > 1:
                k = keff.reshape(keff.shape[0], self.pe[2], self.pe[1], self.pe[0], 2 * self.dim)[..., 2 * a + hi]
                kt = torch.as_tensor(k, device=self.dev)
                for b in range(3):
                    if b != a:
                        kt = kt.repeat_interleave(self.n[b] // self.pe[b], 3 - b)
                kt = kt.unsqueeze(d + 1)
                for kk in range(1, int(k.max()) + 1 if k.size else 1):
                    old = 0.0
                    for m, w in enumerate(_extrapolation(self.T, kk)):
                        if n - kk - m >= 0:
                            old = old + w * halo(levels[n - kk - m], hi)
                    v = torch.where(kt == kk, old, v)
            out.append(v)
        return torch.cat([out[0], levels[n].unflatten(d, (P, S)), out[1]], d + 1), d, S

    def run(self, u0, steps):
        """Level `steps` from u0, and the raw delays drawn, [steps, B, sides]."""
        levels, rhs, log = {0: u0}, [], []
        h = self.h
        for n in range(steps):
            raw, keff = self.delays(n)
            log.append(raw)
            u = levels[n]
            f = 0.0
            for a in range(self.dim):
                ext, d, S = self.padded(levels, n, a, keff)
                part = lambda taps: sum(t.unsqueeze(-1) * ext.narrow(d + 1, j, S)  # noqa: E731
                                        for j, t in enumerate(taps)).flatten(d, d + 1)
                f = f + (part(self.b2[a]) - u * part(self.b1[a]) if self.burgers else part(self.taps[a]))
            rhs = [f] + rhs[: self.ts - 1]
            v = u
            for b, r in zip(BETA[len(rhs)], rhs):
                v = v + b * r
            levels[n + 1] = v
            levels.pop(n - self.L - self.T - h, None)
        return levels[steps], np.stack(log) if log else None


def exact(case, seed):
    if case["kind"] == "ensemble":
        specs = _members(case, seed)
        fields, ua_rms, shapes = {}, {}, {}
        for r, s in enumerate(specs):
            shapes.setdefault((s["n"][0], s["L"]), []).append(r)
        if len(shapes) * case["steps"] > 12000:
            return None
        for (n, _), idx in shapes.items():
            part = [specs[r] for r in idx]
            u0 = torch.stack([_initial(s) for s in part]).view(len(part), 1, 1, n)
            u = _Exact(part).run(u0, case["steps"])[0].view(len(part), n)
            for q, r in enumerate(idx):
                s = specs[r]
                t = case["steps"] * s["dt"]
                sol = dict(s, amp=s["amp"] * np.exp(-s["alpha"] * s["kappa"].astype(np.float64) ** 2 * t),
                           phase=s["phase"] - s["kappa"] * s["c"][0] * t)
                fields[r], ua_rms[r] = u[q], float(_initial(sol).square().mean().sqrt())
        R = range(case["count"])
        return {"fields": torch.cat([fields[r] for r in R]), "ua_rms": np.array([ua_rms[r] for r in R])}
    spec = _spec(case, seed)
    n, pe = _dims(case)
    shape = (1, n[2], n[1], n[0])
    plain = (n[2], n[1], n[0]) if "ny" in case else (n[0],)
    cells = n[0] * n[1] * n[2]
    if case["kind"] == "statistics":
        u, ua = _perturbed(spec, seed), _initial(spec)
        e = u - ua
        pos = torch.arange(n[0], device="cuda") % (n[0] // pe[0])
        h, S = case["order"] // 2, n[0] // pe[0]
        edge = (pos < h) | (pos >= S - h) if pe[0] > 1 else torch.zeros_like(pos, dtype=torch.bool)
        rms = lambda v: float(v.square().mean().sqrt()) if v.numel() else 0.0  # noqa: E731
        return {"stats": {"rms": rms(e), "max_abs": float(e.abs().max()), "mean_abs": float(e.abs().mean()),
                          "rms_I": rms(e[~edge]), "rms_B": rms(e[edge]), "ua_rms": rms(ua)},
                "points": [int((~edge).sum()), int(edge.sum())], "field": ua}
    if case["kind"] == "gradient":
        if cells * case["steps"] > 200_000_000:  # torch keeps every tap's operand for the diffusivity's derivative
            return None
        u0 = _initial(spec).requires_grad_(True)
        alpha = torch.tensor(spec["alpha"], dtype=torch.float64, device="cuda", requires_grad=True)
        u = _Exact([spec], alpha).run(u0.view(shape), case["steps"])[0].view(plain)
        target = _initial(_spec(case, seed + 500)) * 0.8
        (0.5 * ((u - target) ** 2).sum()).backward()
        return {"u": u.detach(), "grad_u0": u0.grad, "grad_alpha": alpha.grad}
    u, log = _Exact([spec]).run(_initial(spec).view(shape), case["steps"])
    out = {"field": u.view(plain)}
    if case["log"]:
        out["delays"] = torch.as_tensor(log[:, 0].astype(np.uint8), device="cuda")
    return out
