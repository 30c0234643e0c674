"""What a user of this library has it do, as cases that can be timed.

Every case is one call sequence through the public Python entry points (solver.Mpdata and
autograd.rollout): `prepare` makes the handle and the seeded device buffers a program holds,
`run` advances them once, `work` counts what the call cannot do without, and `exact` computes the
same result in 64 bits with plain torch operations and nothing of this library.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1407_1309_gb300 import capi
from paper_1407_1309_gb300.autograd import rollout
from paper_1407_1309_gb300.solver import Mpdata

BITS = {"fct": capi.FCT, "tot": capi.TOT, "iga": capi.IGA, "nug": capi.NUG, "kahan": capi.KAHAN, "abs": capi.ABS,
        "dfl": capi.DFL}


def listed():
    return [
        # A small 2D field advanced by a short call: the test-sized runs of a user who sets a
        # problem up, and members of a parameter sweep advanced one by one.  Launches dominate.
        {"name": "small2d_f32", "kind": "field2d", "n0": 59, "n1": 61, "dtype": "f32", "opts": "fct", "n_iters": 2,
         "steps": 20},
        # The benchmark's headline: solid-body rotation on 1024^2 with the compensated FP32 state.
        {"name": "rotation1024_comp_f32", "kind": "compensated2d", "n0": 1024, "n1": 1024, "dtype": "f32",
         "opts": "fct", "n_iters": 2, "steps": 10},
        # The same flow at production size with the plain FP32 state.
        {"name": "rotation4096_f32", "kind": "field2d", "n0": 4096, "n1": 4096, "dtype": "f32", "opts": "fct",
         "n_iters": 2, "steps": 2},
        # The FP64 run that the FP32 results are held against.
        {"name": "rotation1024_f64", "kind": "field2d", "n0": 1024, "n1": 1024, "dtype": "f64", "opts": "fct",
         "n_iters": 2, "steps": 4},
        # A variable-sign field (the |psi| option) on a ragged grid: the options of Sect. 3.1.5.
        {"name": "varsign2d_f32", "kind": "field2d", "n0": 1021, "n1": 1000, "dtype": "f32", "opts": "fct+abs",
         "n_iters": 2, "steps": 4},
        # 3D deformational flow, the benchmark's 3D configuration: three passes, third-order
        # terms, limiter, non-unit G, time-dependent advector.
        {"name": "deform256_f32", "kind": "field3d", "n0": 256, "n1": 256, "n2": 256, "dtype": "f32",
         "opts": "fct+tot+nug", "n_iters": 3, "steps": 1},
        # Its infinite-gauge variant on a small grid of odd sides.
        {"name": "deform_odd_f32", "kind": "field3d", "n0": 101, "n1": 97, "n2": 103, "dtype": "f32",
         "opts": "fct+tot+nug+iga", "n_iters": 2, "steps": 2},
        # The 1D periodic test: 500 cells, 1000 steps in one call.
        {"name": "hello1d_f64", "kind": "line1d", "n": 500, "dtype": "f64", "opts": "fct", "n_iters": 2,
         "steps": 1000},
        # The translating oscillator of Sect. 4.2: two 1D equations coupled by trapezoidal sources,
        # the library's default options.
        {"name": "oscillator1d_f64", "kind": "oscillator1d", "n": 1000, "dtype": "f64", "opts": "fct+iga+kahan",
         "n_iters": 2, "steps": 200},
        # The ensemble: 512 fields with sides of 64 to 512 in one batched handle.
        {"name": "ensemble512_f32", "kind": "ensemble2d", "fields": 512, "least": 64, "most": 512, "multiple": 32,
         "pick": 0, "dtype": "f32", "opts": "fct", "n_iters": 2, "steps": 2},
        # Variational data assimilation: a checkpointed rollout on 512^2 and its gradients with
        # respect to the initial field and the advector.
        {"name": "adjoint512_f32", "kind": "rollout2d", "n0": 512, "n1": 512, "dtype": "f32", "opts": "fct",
         "n_iters": 2, "steps": 40, "every": 20},
        # The shallow-water drop of Sect. 5.4: prognosed velocity, three coupled fields, open edges.
        {"name": "drop320_f64", "kind": "drop2d", "n0": 320, "n1": 320, "dtype": "f64", "opts": "fct+abs+dfl",
         "n_iters": 2, "steps": 20},
    ]


def _side(rng, least, most):
    return int(round(math.exp(rng.uniform(math.log(least), math.log(most)))))


def draw(rng):
    kind = rng.choice(["field2d", "field2d", "field2d", "compensated2d", "field3d", "field3d", "line1d",
                       "oscillator1d", "ensemble2d", "rollout2d", "drop2d"])
    dtype = "f32" if rng.random() < 0.7 else "f64"
    if kind == "field2d":
        n0, n1 = _side(rng, 40, 4096), _side(rng, 40, 4096)
        opts, n_iters = rng.choice([("fct", 2), ("fct", 2), ("fct", 2), ("fct+iga", 2), ("fct+nug", 2),
                                    ("fct+iga+kahan", 2), ("fct+abs", 2), ("fct+abs", 2), ("fct+dfl", 2),
                                    ("fct+tot", 3), ("fct+tot+iga", 2), ("fct", 3), ("", 2)])
        if dtype == "f64" and n0 * n1 > 1 << 21:
            n0 = (1 << 21) // n1
        steps = max(1, min(rng.randint(1, 20), (1 << 23) // (n0 * n1)))
        return {"kind": kind, "n0": n0, "n1": n1, "dtype": dtype, "opts": opts, "n_iters": n_iters, "steps": steps}
    if kind == "compensated2d":
        n0, n1 = _side(rng, 200, 3000), _side(rng, 200, 3000)
        return {"kind": kind, "n0": n0, "n1": n1, "dtype": "f32", "opts": "fct", "n_iters": 2,
                "steps": max(1, min(rng.randint(1, 10), (1 << 24) // (n0 * n1)))}
    if kind == "field3d":
        n = [_side(rng, 24, 200 if dtype == "f32" else 80) for _ in range(3)]
        opts, n_iters = rng.choice([("fct+tot+nug", 3), ("fct+tot+nug+iga", 2), ("fct", 2), ("fct+nug", 2),
                                    ("tot", 2), ("fct+abs+tot", 2)])
        return {"kind": kind, "n0": n[0], "n1": n[1], "n2": n[2], "dtype": dtype, "opts": opts, "n_iters": n_iters,
                "steps": rng.randint(1, 2)}
    if kind == "line1d":
        opts, n_iters = rng.choice([("fct", 2), ("fct+iga+kahan", 2), ("fct+tot", 3), ("iga+tot", 2)])
        return {"kind": kind, "n": _side(rng, 100, 2000), "dtype": dtype, "opts": opts, "n_iters": n_iters,
                "steps": _side(rng, 50, 300)}
    if kind == "oscillator1d":
        return {"kind": kind, "n": _side(rng, 250, 2000), "dtype": dtype, "opts": "fct+iga+kahan", "n_iters": 2,
                "steps": rng.randint(40, 120)}
    if kind == "ensemble2d":
        most = rng.randint(96, 512)
        return {"kind": kind, "fields": _side(rng, 8, 256), "least": max(40, most // 4), "most": most, "multiple": 1,
                "pick": rng.randint(1, 1 << 20), "dtype": "f32", "opts": "fct", "n_iters": 2,
                "steps": rng.randint(1, 2)}
    if kind == "rollout2d":
        n0, n1 = _side(rng, 64, 700), _side(rng, 64, 700)
        steps = rng.randint(8, 24)
        return {"kind": kind, "n0": n0, "n1": n1, "dtype": "f32" if n0 * n1 > 1 << 17 else dtype, "opts": "fct",
                "n_iters": 2, "steps": steps, "every": rng.randint(4, 12)}
    n0, n1 = _side(rng, 80, 400), _side(rng, 80, 400)
    return {"kind": "drop2d", "n0": n0, "n1": n1, "dtype": dtype, "opts": "fct+abs+dfl", "n_iters": 2,
            "steps": 2 * rng.randint(1, 8)}


# ------------------------------------------------------------------------------------ inputs

DEVICE = torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.float64


def _opts(case):
    return [w for w in case["opts"].split("+") if w]


def _range(n, offset=0.0):
    return torch.arange(n, dtype=torch.float64, device=DEVICE) + offset


def _modes(rng, shape, count, kmax=3, offset=0.5):
    """Sum of `count` periodic Fourier modes with random wave vectors, phases and amplitudes."""
    f = torch.zeros(shape, dtype=torch.float64, device=DEVICE)
    for _ in range(count):
        k = [0] * len(shape)
        while not any(k):
            k = [int(v) for v in rng.integers(-kmax, kmax + 1, size=len(shape))]
        arg = float(rng.uniform(0, 2 * math.pi))
        for d, n in enumerate(shape):
            x = _range(n, offset).mul_(2 * math.pi * k[d] / n)
            arg = arg + x.reshape([-1 if e == d else 1 for e in range(len(shape))])
        f.add_(torch.cos(arg), alpha=float(rng.normal()))
    return f


def _swirl(rng, shape, courant):
    """Discretely nondivergent 2D advector: differences of a streamfunction at the cell corners."""
    p = _modes(rng, shape, 6, offset=1.0)
    gc = [p - torch.roll(p, 1, 1), torch.roll(p, 1, 0) - p]
    s = courant / max(float(gc[0].abs().max()), float(gc[1].abs().max()))
    return [v * s for v in gc]


def _rotation(shape, courant):
    """Solid-body rotation about the domain's centre, its largest Courant number given."""
    n0, n1 = shape
    w = 2.0 * courant / max(shape)
    gc0 = (w * (_range(n1, 0.5) - 0.5 * n1))[None, :].expand(n0, n1).contiguous()
    gc1 = (-w * (_range(n0, 0.5) - 0.5 * n0))[:, None].expand(n0, n1).contiguous()
    return [gc0, gc1]


def _blob(shape, centre, width):
    """Periodic Gaussian of peak 1; centre and width in units of the domain's sides."""
    r2 = 0.0
    for d, n in enumerate(shape):
        x = (_range(n, 0.5) / n - centre[d]).abs()
        x = torch.minimum(x, 1.0 - x)
        r2 = r2 + (x * x).reshape([-1 if e == d else 1 for e in range(len(shape))])
    return torch.exp(r2 * (-0.5 / width ** 2))


def _g_factor(rng, shape, modes):
    f = _modes(rng, shape, modes)
    return 1.0 + 0.2 * f / f.abs().max()


def _inputs(case, seed):
    """The case's input fields in its own data type."""
    rng = np.random.default_rng(seed)
    kind, opts = case["kind"], _opts(case)
    signed = "abs" in opts or "iga" in opts
    r = {}
    if kind in ("field2d", "compensated2d"):
        shape = (case["n0"], case["n1"])
        # with room below the stability limit for G < 1 and the divergent part
        courant = 0.4 if "nug" in opts or "dfl" in opts else 0.5
        r["gc"] = _swirl(rng, shape, courant) if signed else _rotation(shape, courant)
        if signed:  # two blobs of opposite sign
            r["psi"] = sum(s * _blob(shape, rng.uniform(0.2, 0.8, 2), rng.uniform(0.06, 0.12)) for s in (1.0, -1.0))
        else:       # a cone on a background of 1
            x = [(_range(n, 0.5) - 0.5 * n) / max(shape) for n in shape]
            a = rng.uniform(0, 2 * math.pi)
            rad = 0.25 * min(shape) / max(shape)
            d2 = (x[0][:, None] - rad * math.cos(a)) ** 2 + (x[1][None, :] - rad * math.sin(a)) ** 2
            t = (1.0 - d2 / (0.6 * rad) ** 2).clamp_(min=0.0)
            r["psi"] = 1.0 + rng.uniform(3.0, 5.0) * t * t
        if "dfl" in opts:  # a divergent flow: one component modulated along itself
            r["gc"][1] = r["gc"][1] + 0.15 * torch.sin(_range(shape[1], 1.0) * (2 * math.pi / shape[1]))[None, :]
        if "nug" in opts:
            r["g"] = _g_factor(rng, shape, 4)
    elif kind == "field3d":
        shape = (case["n0"], case["n1"], case["n2"])
        # the curl of a smooth vector potential held on the cell edges, scaled to |C| <= 0.4 / 1.2
        A = [_modes(rng, shape, 2, kmax=2, offset=0.5) for _ in range(3)]
        dif = lambda f, d: f - torch.roll(f, 1, d)
        gc = [dif(A[2], 1) - dif(A[1], 2), dif(A[0], 2) - dif(A[2], 0), dif(A[1], 0) - dif(A[0], 1)]
        s = 0.33 / max(float(v.abs().max()) for v in gc)
        r["gc"] = [v.mul_(s) for v in gc]
        r["psi"] = sum(s * _blob(shape, rng.uniform(0.35, 0.65, 3), 0.08 * rng.uniform(0.9, 1.1))
                       for s in (1.0, -1.0 if signed else 1.0))
        if "nug" in opts:
            r["g"] = _g_factor(rng, shape, 4)
        r["scale"] = [float(np.float32(math.cos(math.pi * (t + 0.5) / 1280))) for t in range(case["steps"])]
    elif kind in ("line1d", "oscillator1d"):
        n = case["n"]
        x = _range(n)
        c = float(rng.uniform(0.3, 0.6))
        if kind == "line1d":  # a box and a Gaussian
            lo = int(rng.integers(n // 20, n // 5))
            psi = ((x >= lo) & (x <= lo + n // 10)).double() * float(rng.uniform(0.5, 1.0))
            r["psi"] = psi + torch.exp(-0.5 * ((x - 0.6 * n) / (0.03 * n)) ** 2)
            r["gc"] = [torch.full((n,), c, dtype=torch.float64, device=DEVICE)]
        else:                 # psi a raised cosine, phi zero
            lo = float(rng.uniform(20.0, 100.0))
            y = x + 0.5 - lo
            psi = torch.where((y > 0) & (y < 100.0), 0.5 * (1.0 - torch.cos(y * (2 * math.pi / 100.0))), 0.0 * y)
            r["psi"] = torch.cat([psi, torch.zeros_like(psi)])
            r["gc"] = [torch.full((2 * n,), c, dtype=torch.float64, device=DEVICE)]
            r["omega"] = 2 * math.pi / 1400.0
    elif kind == "ensemble2d":
        psi, gc0, gc1 = [], [], []
        for n in _members(case):
            gc = _swirl(rng, (n, n), 0.5)
            gc0.append(gc[0].flatten())
            gc1.append(gc[1].flatten())
            psi.append((1.0 + _blob((n, n), rng.uniform(0, 1, 2), rng.uniform(0.05, 0.15))).flatten())
        r["psi"], r["gc"] = torch.cat(psi), [torch.cat(gc0), torch.cat(gc1)]
    elif kind == "rollout2d":
        shape = (case["n0"], case["n1"])
        f = _modes(rng, shape, 6)
        r["psi"] = 2.0 + 0.5 * f / f.abs().max()
        r["gc"] = _swirl(rng, shape, 0.5)
        f = _modes(rng, shape, 6)
        r["bar"] = f / f.square().mean().sqrt()
    else:  # drop2d
        dx = 0.05
        x = [(_range(n, 0.5) - 0.5 * n) * dx + float(rng.uniform(-0.3, 0.3)) for n in (case["n0"], case["n1"])]
        h = (float(rng.uniform(0.8, 1.2)) - x[0][:, None] ** 2 - x[1][None, :] ** 2).clamp_(min=0.0)
        r["psi"] = torch.cat([h.flatten(), torch.zeros(2 * h.numel(), dtype=torch.float64, device=DEVICE)])
        r["dx"], r["dt"] = dx, 0.01
    dt = _dtype(case)
    for k in ("psi", "g", "bar"):
        if k in r:
            r[k] = r[k].to(dt).contiguous()
    if "gc" in r:
        r["gc"] = [v.to(dt).contiguous() for v in r["gc"]]
    return r


def _members(case):
    """Sides of the ensemble's square fields."""
    rng = random.Random(case["pick"])
    m = case["multiple"]
    return [m * rng.randint(-(-case["least"] // m), case["most"] // m) for _ in range(case["fields"])]


# --------------------------------------------------------------------------- prepare and run

def prepare(case, seed):
    x = _inputs(case, seed)
    kind = case["kind"]
    opts = sum(BITS[w] for w in _opts(case))
    new = lambda shapes, bits=0: Mpdata(shapes, dtype=_dtype(case), n_iters=case["n_iters"], opts=opts | bits)
    s = {"case": case, "x": x}
    if kind == "field3d":
        s["m"] = new((case["n0"], case["n1"], case["n2"]))
    elif kind == "line1d":
        s["m"] = new((case["n"],))
    elif kind == "oscillator1d":
        s["m"] = new([(case["n"],)] * 2, capi.RHS_TRAPEZ)
        s["m"].set_rhs_linear([[0.0, x["omega"]], [-x["omega"], 0.0]])
    elif kind == "ensemble2d":
        s["m"] = new([(n, n) for n in _members(case)])
    elif kind == "drop2d":
        s["m"] = new([(case["n0"], case["n1"])] * 3, capi.SW | capi.OPEN0 | capi.OPEN1)
    else:
        s["m"] = new((case["n0"], case["n1"]))
    if kind == "rollout2d":
        x["psi"].requires_grad_(True)
        for v in x["gc"]:
            v.requires_grad_(True)
    else:
        s["out"] = torch.empty_like(x["psi"])
    if kind == "compensated2d":
        s["lo"], s["lo_out"] = torch.zeros_like(x["psi"]), torch.empty_like(x["psi"])
    return s


def run(s):
    case, x, m = s["case"], s["x"], s["m"]
    kind, steps = case["kind"], case["steps"]
    if kind == "compensated2d":
        m.advance_compensated(x["psi"], s["lo"], s["out"], s["lo_out"], x["gc"], n_steps=steps)
        return {"psi": s["out"], "lo": s["lo_out"]}
    if kind == "rollout2d":
        psi = rollout(m, x["psi"], x["gc"], steps, case["every"])
        bars = torch.autograd.grad(psi, [x["psi"], *x["gc"]], x["bar"])
        return {"psi": psi.detach(), "psi_bar": bars[0], "gc0_bar": bars[1], "gc1_bar": bars[2]}
    if kind == "drop2d":
        s["out"].copy_(x["psi"])
        m.sw_reset()
        return m.sw_advance(s["out"], x["dt"], x["dx"], n_steps=steps)
    if kind == "oscillator1d":
        return m.advance(x["psi"], s["out"], x["gc"], dt=1.0, n_steps=steps)
    return m.advance(x["psi"], s["out"], x["gc"], g=x.get("g"), n_steps=steps, gc_scale=x.get("scale"))


def work(case):
    kind, opts, steps = case["kind"], _opts(case), case["steps"]
    size = 4 if case["dtype"] == "f32" else 8
    fields = 1
    if kind in ("line1d", "oscillator1d"):
        nd, cells = 1, case["n"]
    elif kind == "field3d":
        nd, cells = 3, case["n0"] * case["n1"] * case["n2"]
    elif kind == "ensemble2d":
        nd, cells = 2, sum(n * n for n in _members(case))
    else:
        nd, cells = 2, case["n0"] * case["n1"]
    if kind == "oscillator1d":
        fields = 2
    elif kind == "drop2d":
        fields = 3
    # arrays of `cells` values read and written once
    arrays = (2 + nd) * fields + (1 if "nug" in opts else 0)
    if kind == "compensated2d":
        arrays += 2
    elif kind == "rollout2d":
        arrays += 2 + nd  # the cotangent in, the gradients out
    elif kind == "drop2d":
        arrays = 2 * fields
    # arithmetic of one step on one cell: donor-cell passes, pseudo-advectors, limiter
    face = 10 + 12 * (nd - 1) + (12 + 8 * (nd - 1) + (14 if nd == 3 else 0) if "tot" in opts else 0)
    limiter = 10 * nd + 12 + 6 * nd if "fct" in opts else 0
    each = 6 * nd * case["n_iters"] + (case["n_iters"] - 1) * (nd * face + limiter)
    if kind == "rollout2d":
        each *= 3
    return {"bytes": float(arrays * cells * size), "flops": float(each * fields * cells * steps)}


# ------------------------------------------------------------------------- the same in 64 bits

class _Scheme:
    """MPDATA steps in plain torch, periodic or with open edges along every dimension."""

    def __init__(self, opts, n_iters, is_open=False):
        self.o, self.n_iters, self.is_open = set(opts), n_iters, is_open

    def at(self, x, d, s):
        """x at the cell s cells further along d."""
        if not self.is_open:
            return torch.roll(x, -s, d)
        n = x.shape[d]
        return x.index_select(d, (torch.arange(n, device=x.device) + s).clamp_(0, n - 1))

    def face(self, v, d, s=0):
        """The component along d on the face s cells beyond the cell's right one."""
        if not self.is_open:
            return torch.roll(v, -s, d) if s else v
        n = v.shape[d]
        return v.index_select(d, (torch.arange(n, device=v.device) + s).clamp_(0, n - 2))

    @staticmethod
    def frac(n, d):
        ok = d != 0
        return torch.where(ok, n / torch.where(ok, d, torch.ones_like(d)), torch.zeros_like(d))

    @staticmethod
    def flux(left, right, v, unit):
        return v if unit else v.clamp(min=0) * left + v.clamp(max=0) * right

    def fluxes(self, psi, v, d, unit):
        fp = self.flux(psi, self.at(psi, d, 1), self.face(v, d), unit)
        fm = self.flux(self.at(psi, d, -1), psi, self.face(v, d, -1), unit)
        return fp, fm

    def donor(self, psi, gc, G, unit):
        out = psi
        for d, v in enumerate(gc):
            fp, fm = self.fluxes(psi, v, d, unit)
            out = out - (fp - fm) / G
        return out

    def antidiff(self, psi, gc, G):
        iga, nd, at = "iga" in self.o, psi.dim(), self.at
        p = psi.abs() if "abs" in self.o else psi
        res = []
        for d in range(nd):
            V = self.face(gc[d], d)
            r = 2.0 / (G + at(G, d, 1)) if torch.is_tensor(G) else 1.0
            p1 = at(p, d, 1)
            A = (p1 - p) / 2 if iga else self.frac(p1 - p, p1 + p)
            out = (V.abs() - V * V * r) * A
            Vq = {}
            for q in range(nd):
                if q == d:
                    continue
                both = self.face(gc[q], q) + self.face(gc[q], q, -1)
                Vq[q] = (both + at(both, d, 1)) / 4
                a, e = at(p, q, 1), at(p, q, -1)
                b, f = at(a, d, 1), at(e, d, 1)
                n, m = (a + b) - (e + f), (b - a) - (f - e)
                den = (a + b) + (e + f)
                out = out - 0.5 * V * Vq[q] * r * (n / 4 if iga else self.frac(n, den))
                if "tot" in self.o:
                    out = out + V.abs() * Vq[q] * r * (1 - 2 * V.abs() * r) * (m / 4 if iga else self.frac(m, den))
            if "tot" in self.o:
                pm, p2 = at(p, d, -1), at(p, d, 2)
                n = ((p2 - p1) - p) + pm
                D = n / 4 if iga else self.frac(n, ((p2 + p1) + p) + pm)
                out = out + (3 * V * V.abs() * r - 2 * V * V * V * r * r - V) / 3 * D
                if nd == 3:
                    q1, q2 = [q for q in range(3) if q != d]
                    pair = p + p1
                    pr = [at(at(pair, q1, s1), q2, s2) for s1 in (1, -1) for s2 in (1, -1)]
                    n = (pr[0] - pr[1]) - (pr[2] - pr[3])
                    D = n / 8 if iga else self.frac(n, (pr[0] + pr[1]) + (pr[2] + pr[3]))
                    out = out - 2.0 / 3.0 * V * Vq[q1] * Vq[q2] * r * r * D
            if "dfl" in self.o:
                div = sum(self.face(v, q) - self.face(v, q, -1) for q, v in enumerate(gc))
                nxt = sum((self.face(v, d, 1) - self.face(v, d)) if q == d else
                          at(self.face(v, q) - self.face(v, q, -1), d, 1) for q, v in enumerate(gc))
                out = out - 0.25 * V * (div + nxt) * r
            res.append(out)
        return res

    def limited(self, psi, v, G, hi, lo, unit):
        nd, at = psi.dim(), self.at
        inn = out = 0.0
        for d in range(nd):
            fp, fm = self.fluxes(psi, v[d], d, unit)
            inn = inn + fm.clamp(min=0) - fp.clamp(max=0)
            out = out + fp.clamp(min=0) - fm.clamp(max=0)
        one = torch.ones_like(psi)
        factor = lambda room, s: torch.where(s > 0, G * room.clamp(min=0) / torch.where(s > 0, s, one), one)
        up, down = factor(hi - psi, inn), factor(psi - lo, out)
        res = []
        for d in range(nd):
            f = self.flux(psi, at(psi, d, 1), v[d], unit)
            right = (f > 0) | ((f == 0) & (v[d] > 0))
            a = torch.where(right, down, up)
            b = torch.where(right, at(up, d, 1), at(down, d, 1))
            res.append(v[d] * torch.minimum(torch.minimum(a, b), one))
        return res

    def step(self, psi, gc, G=1.0, scale=1.0):
        gc = [v * scale for v in gc] if scale != 1.0 else gc
        unit, fct = "iga" in self.o, "fct" in self.o
        cur = self.donor(psi, gc, G, False)
        hi, lo = torch.maximum(psi, cur), torch.minimum(psi, cur)
        if fct:
            h0, l0 = hi, lo
            for d in range(psi.dim()):
                for s in (-1, 1):
                    hi, lo = torch.maximum(hi, self.at(h0, d, s)), torch.minimum(lo, self.at(l0, d, s))
        v = gc
        for _ in range(1, self.n_iters):
            v = self.antidiff(cur, v, G)
            if fct:
                v = self.limited(cur, v, G, hi, lo, unit)
            cur = self.donor(cur, v, G, unit)
        return cur


def _shallow_water(scheme, state, shape, dt, dx, steps):
    h, q = state[0], [state[1], state[2]]
    prev = None
    grad = lambda f, d: (scheme.at(f, d, 1) - scheme.at(f, d, -1)) / (2 * dx)
    for _ in range(steps):
        wet = h > 1e-8
        u = [torch.where(wet, v / torch.where(wet, h, torch.ones_like(h)), torch.zeros_like(h)) for v in q]
        ext = [1.5 * a - 0.5 * b for a, b in zip(u, prev or u)]
        prev = u
        gc = [0.5 * (e + scheme.at(e, d, 1)) * (dt / dx) for d, e in enumerate(ext)]
        q = [v - 0.5 * dt * h * grad(h, d) for d, v in enumerate(q)]
        h, q = scheme.step(h, gc), [scheme.step(v, gc) for v in q]
        q = [v - 0.5 * dt * h * grad(h, d) for d, v in enumerate(q)]
    return torch.cat([h.flatten()] + [v.flatten() for v in q])


def exact(case, seed):
    x = _inputs(case, seed)
    kind, steps = case["kind"], case["steps"]
    scheme = _Scheme(_opts(case), case["n_iters"], kind == "drop2d")
    psi = x["psi"].double()
    gc = [v.double() for v in x.get("gc", [])]
    G = x["g"].double() if "g" in x else 1.0
    if kind == "rollout2d":
        leaves = [v.requires_grad_(True) for v in [psi, *gc]]
        cur = psi
        for _ in range(steps):
            cur = scheme.step(cur, gc)
        bars = torch.autograd.grad(cur, leaves, x["bar"].double())
        return {"psi": cur.detach(), "psi_bar": bars[0], "gc0_bar": bars[1], "gc1_bar": bars[2]}
    if kind == "drop2d":
        shape = (case["n0"], case["n1"])
        return _shallow_water(scheme, psi.reshape(3, *shape), shape, x["dt"], x["dx"], steps)
    if kind == "oscillator1d":
        n, th = case["n"], 0.5 * x["omega"]
        a, b = psi[:n], psi[n:]
        for _ in range(steps):
            a, b = a + th * b, b - th * a
            a, b = scheme.step(a, [gc[0][:n]]), scheme.step(b, [gc[0][n:]])
            a, b = (a + th * b) / (1 + th * th), (b - th * a) / (1 + th * th)
        return torch.cat([a, b])
    if kind == "ensemble2d":
        res, o = [], 0
        for n in _members(case):
            cut = lambda v: v[o:o + n * n].reshape(n, n)
            cur, v = cut(psi), [cut(w) for w in gc]
            for _ in range(steps):
                cur = scheme.step(cur, v)
            res.append(cur.flatten())
            o += n * n
        return torch.cat(res)
    for t in range(steps):
        psi = scheme.step(psi, gc, G, x["scale"][t] if "scale" in x else 1.0)
    # the low parts of a compensated state are the rounding that 64 bits do not have
    return {"psi": psi, "lo": None} if kind == "compensated2d" else psi
