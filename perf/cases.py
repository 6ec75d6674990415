"""The stencil runs whose speed is measured: sizes, inputs, one pass, its counted work, its value in 64 bits.

Families (the key "run" of a case):
  sweep    one Plan.run: Diffusion or Hotspot, 2D or 3D, float32 or 16-bit grid storage, the
           radius-R star, or diffusion with per-cell coefficients
  batch    one replay of a Batch of uneven 2D grids
  adjoint  one training step of an Adjoint: forward run, then the gradients of a weighted loss

A program keeps its plan (batch, adjoint) across calls, so those are part of the prepared state.
Values and coefficient ranges are those of the seeded workloads in synth/: diffusion fields U[0,1),
temperatures U[320,340) K over power U[0,0.5), ambient 80, positive normalised weights.
"""
from __future__ import annotations

import math
import random

import torch

import paper_1802_00438_gb300 as st

DIFFUSION, THERMAL, VARIABLE = st.ST_DIFFUSION, st.ST_THERMAL, st.ST_DIFFUSION_VAR
STORAGE = {"f32": st.ST_F32, "bf16": st.ST_BF16, "f16": st.ST_F16}
AMBIENT = 80.0
# steps of the largest listed sweep, 16384^2 cells x 400: a drawn case has no more cell updates
MOST_UPDATES = 16384 * 16384 * 400


def _sweep(name, kind, nx, ny, nz, steps, storage="f32", rad=1):
    c = {"name": name} if name else {}
    c.update(run="sweep", kind=kind, nx=nx, ny=ny, nz=nz, steps=steps, storage=storage, rad=rad)
    return c


def listed():
    return [
        # the smallest calls: a few steps of a grid a simulation coupled to other work advances
        # between its own phases; launch and exchange latency count
        _sweep("diff2d_256x192_s20", DIFFUSION, 256, 192, 1, 20),
        # the 1024^2, 100-step configuration
        _sweep("diff2d_1024_s100", DIFFUSION, 1024, 1024, 1, 100),
        # a floorplan-sized thermal map of odd width: rows not on 16-byte boundaries, ragged tiles
        _sweep("therm2d_3001x2003_s150", THERMAL, 3001, 2003, 1, 150),
        # the headline 16384^2 thermal grid, a part of its 1000 steps
        _sweep("therm2d_16384_s400", THERMAL, 16384, 16384, 1, 400),
        # 16-bit storage of the grids between passes
        _sweep("therm2d_8192_bf16_s200", THERMAL, 8192, 8192, 1, 200, storage="bf16"),
        # a small 3D domain with odd sides: unaligned rows, few tile columns for the chip
        _sweep("diff3d_187x141x93_s30", DIFFUSION, 187, 141, 93, 30),
        # the two 3D configurations, a part of their 1000 steps
        _sweep("diff3d_512_s120", DIFFUSION, 512, 512, 512, 120),
        _sweep("therm3d_512x512x256_s120", THERMAL, 512, 512, 256, 120),
        # many uneven grids in one launch: sides 256..4096, 50..500 steps, kinds alternate
        {"name": "batch64", "run": "batch", "count": 64, "layout": 5, "lo": 256, "hi": 4096},
        # the 2048^2, 200-step gradient with checkpoints every 20 steps
        {"name": "adjoint2048_s200", "run": "adjoint", "kind": DIFFUSION, "nx": 2048, "ny": 2048,
         "steps": 200, "ckpt": 20},
        # higher-order diffusion: the 9-point star
        _sweep("star2_2d_8192_s64", DIFFUSION, 8192, 8192, 1, 64, rad=2),
        # heterogeneous media: diffusion with per-cell coefficients
        _sweep("vardiff2d_4096_s100", VARIABLE, 4096, 4096, 1, 100),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    family = rng.choice(["2d", "2d", "2d", "16bit", "3d", "3d", "batch", "adjoint", "star", "variable"])
    if family == "batch":
        return {"run": "batch", "count": rng.randint(16, 64), "layout": rng.randint(6, 10 ** 6),
                "lo": 256, "hi": 4096}
    if family == "adjoint":
        return {"run": "adjoint", "kind": rng.choice([DIFFUSION, THERMAL]), "nx": _log(rng, 256, 2048),
                "ny": _log(rng, 256, 2048), "steps": rng.randint(40, 200),
                "ckpt": rng.choice([10, 20, 25])}
    if family == "3d":
        return _sweep("", rng.choice([DIFFUSION, THERMAL]), _log(rng, 64, 512), _log(rng, 64, 512),
                      _log(rng, 48, 512), _log(rng, 12, 120))
    if family == "star":
        return _sweep("", DIFFUSION, _log(rng, 512, 8192), _log(rng, 512, 8192), 1,
                      rng.randint(8, 64), rad=2)
    if family == "variable":
        return _sweep("", VARIABLE, _log(rng, 512, 4096), _log(rng, 512, 4096), 1, rng.randint(20, 100))
    if family == "16bit":
        return _sweep("", rng.choice([DIFFUSION, THERMAL]), _log(rng, 1024, 8192),
                      _log(rng, 1024, 8192), 1, rng.randint(40, 200),
                      storage=rng.choice(["bf16", "f16"]))
    nx, ny, steps = _log(rng, 192, 16384), _log(rng, 192, 16384), _log(rng, 20, 400)
    return _sweep("", rng.choice([DIFFUSION, THERMAL]), nx, ny, 1, min(steps, MOST_UPDATES // (nx * ny)))


# ---- inputs ------------------------------------------------------------------------------------

def _weights(rng, n, per=0):
    """n positive weights that sum to 1; per > 0: those of distance d (per of each) fall off as 1/d."""
    u = [rng.uniform(0.05, 1.0) for _ in range(n)]
    if per:
        u = [u[0]] + [x / (1 + i // per) for i, x in enumerate(u[1:])]
    total = sum(u)
    return [x / total for x in u]


def _coeffs(rng, kind, ndim, rad):
    """Coefficients as Python floats that are exact in float32."""
    if kind == THERMAL:
        k_dt, rx, ry, rz = rng.uniform(0.5, 1), rng.uniform(0.05, 0.2), rng.uniform(0.05, 0.2), rng.uniform(1e-4, 1e-3)
        k = [k_dt, rx, ry, rz, AMBIENT]
        if ndim == 3:
            ce, cn, ca = k_dt * rx, k_dt * ry, k_dt * rz
            k = [1 - (2 * ce + 2 * cn + 3 * ca), ce, ce, cn, cn, ca, ca, k_dt, AMBIENT]
    else:
        per = 4 if ndim == 2 else 6
        k = _weights(rng, 1 + per * rad, per if rad > 1 else 0)
    return torch.tensor(k, dtype=torch.float32).tolist()


def _field(gen, kind, shape):
    u = torch.rand(shape, generator=gen, device="cuda", dtype=torch.float32)
    return u.mul_(20.0).add_(320.0) if kind == THERMAL else u


def _power(gen, kind, shape):
    if kind == THERMAL:
        return torch.rand(shape, generator=gen, device="cuda", dtype=torch.float32).mul_(0.5)
    if kind == VARIABLE:   # five planes cc, cw, ce, cs, cn that sum to 1 in each cell
        w = torch.rand((5, *shape), generator=gen, device="cuda", dtype=torch.float32).mul_(0.95).add_(0.05)
        return w.div_(w.sum(0, keepdim=True))
    return None


def _inputs(case, seed):
    """The seeded inputs of a sweep or an adjoint: (field, power or planes, coefficients, loss weights)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    kind, nz = case["kind"], case.get("nz", 1)
    ndim = 3 if nz > 1 else 2
    shape = (nz, case["ny"], case["nx"]) if ndim == 3 else (case["ny"], case["nx"])
    u = _field(gen, kind, shape)
    p = _power(gen, kind, shape)
    w = None
    if case["run"] == "adjoint":   # dL/du of a loss with weights U[-1, 1)
        w = torch.rand(shape, generator=gen, device="cuda", dtype=torch.float32).mul_(2.0).sub_(1.0)
    return u, p, _coeffs(random.Random(seed), kind, ndim, case.get("rad", 1)), w


def _grids(case):
    """(kind, nx, ny, steps) of a batch's grids."""
    rng = random.Random(case["layout"])
    return [(THERMAL if g % 2 else DIFFUSION, _log(rng, case["lo"], case["hi"]),
             _log(rng, case["lo"], case["hi"]), rng.randint(50, 500)) for g in range(case["count"])]


def _batch_inputs(case, seed):
    gen, rng = torch.Generator(device="cuda").manual_seed(seed), random.Random(seed)
    out = []
    for kind, nx, ny, steps in _grids(case):
        u = _field(gen, kind, (ny, nx))
        out.append(dict(kind=kind, nx=nx, ny=ny, steps=steps, grid_in=u, power=_power(gen, kind, (ny, nx)),
                        coeffs=_coeffs(rng, kind, 2, 1)))
    return out


def prepare(case, seed):
    if case["run"] == "batch":
        grids = _batch_inputs(case, seed)
        for g in grids:
            g["grid_out"] = torch.empty_like(g["grid_in"])
        return {"batch": st.Batch(grids), "out": [g["grid_out"] for g in grids]}
    u, p, k, w = _inputs(case, seed)
    if case["run"] == "adjoint":
        adj = st.Adjoint(case["kind"], case["nx"], case["ny"], case["steps"], ckpt=case["ckpt"])
        return {"adjoint": adj, "u": u, "power": p, "coeffs": k, "weights": w, "out": torch.empty_like(u)}
    ndim = 3 if case["nz"] > 1 else 2
    plan = st.Plan(case["kind"], ndim, case["nx"], case["ny"], case["nz"], storage=STORAGE[case["storage"]],
                   rad=case["rad"] if case["rad"] > 1 else 0)
    return {"plan": plan, "u": u, "power": p, "coeffs": None if case["kind"] == VARIABLE else k,
            "steps": case["steps"], "out": torch.empty_like(u)}


def run(state):
    if "batch" in state:
        state["batch"].run()
        return state["out"]
    if "adjoint" in state:
        out = state["adjoint"].forward(state["u"], state["coeffs"], state["power"], state["out"])
        gu, gk, gp, _ = state["adjoint"].backward(state["weights"], state["power"])
        return {"u": out, "grad_u": gu, "grad_coeffs": gk, "grad_power": gp}
    return state["plan"].run(state["u"], state["out"], state["coeffs"], state["steps"], power=state["power"])


# ---- counted work ------------------------------------------------------------------------------

def _flops_per_cell(kind, ndim, rad):
    """Table 2's operations per cell update (13 and 17 in 3D); 8R+1 for a star in 2D."""
    if rad > 1:
        return (8 if ndim == 2 else 12) * rad + 1
    if kind == THERMAL:
        return 15 if ndim == 2 else 17
    return 9 if ndim == 2 else 13


def work(case):
    if case["run"] == "batch":
        b = f = 0
        for kind, nx, ny, steps in _grids(case):
            b += nx * ny * (12 if kind == THERMAL else 8)
            f += nx * ny * steps * _flops_per_cell(kind, 2, 1)
        return {"bytes": b, "flops": f}
    ndim = 3 if case.get("nz", 1) > 1 else 2
    n = case["nx"] * case["ny"] * case.get("nz", 1)
    f = n * case["steps"] * _flops_per_cell(case["kind"], ndim, case.get("rad", 1))
    grids = {THERMAL: 3, VARIABLE: 7}.get(case["kind"], 2)
    if case["run"] == "adjoint":
        # forward, transposed sweep, and two per coefficient (five) and cell for its gradient;
        # the weights in and the gradient(s) out besides the forward run's grids
        return {"bytes": 4 * n * (grids + (3 if case["kind"] == THERMAL else 2)),
                "flops": 2 * f + 10 * n * case["steps"]}
    return {"bytes": 4 * n * grids, "flops": f}


# ---- 64 bits -----------------------------------------------------------------------------------

class _Clamped:
    """A grid in float64 with R ghost cells per side that repeat its edges."""

    def __init__(self, u, rad=1):
        self.r, self.dims = rad, u.dim()
        self.g = torch.empty([s + 2 * rad for s in u.shape], dtype=torch.float64, device=u.device)
        self.inner = tuple(slice(rad, rad + s) for s in u.shape)
        self.set(u)

    def set(self, u):
        self.g[self.inner] = u
        r = self.r
        for a in range(self.dims):   # faces suffice: a star reads no corner
            sel = list(self.inner)
            n = self.g.shape[a] - 2 * r
            for side, edge in ((slice(0, r), r), (slice(r + n, r + n + r), r + n - 1)):
                s, e = list(sel), list(sel)
                s[a], e[a] = side, slice(edge, edge + 1)
                self.g[tuple(s)] = self.g[tuple(e)]

    def at(self, axis, d):
        """The grid's cells d further along the axis (0: x, 1: y, 2: z)."""
        a = self.dims - 1 - axis
        sel = list(self.inner)
        sel[a] = slice(sel[a].start + d, sel[a].stop + d)
        return self.g[tuple(sel)]

    @property
    def c(self):
        return self.g[self.inner]


def _neighbours(g, ndim, d=1):
    """w, e, s, n (, b, a) at distance d: x-1, x+1, y+1, y-1, z-1, z+1."""
    out = [g.at(0, -d), g.at(0, d), g.at(1, d), g.at(1, -d)]
    return out + [g.at(2, -d), g.at(2, d)] if ndim == 3 else out


def _advance(g, out, kind, ndim, k, p, rad=1):
    """One Jacobi step of Table 2 from g into out (float64)."""
    c, nb = g.c, _neighbours(g, ndim)
    if kind == VARIABLE:
        torch.mul(p[0], c, out=out)
        for q, x in zip(p[1:], nb):
            out.addcmul_(q, x)
    elif kind == THERMAL and ndim == 2:
        sdc, rx, ry, rz, amb = k
        torch.mul(c, 1.0 - sdc * (2.0 * rx + 2.0 * ry + rz), out=out)
        out.add_(p, alpha=sdc).add_(sdc * amb * rz)
        for q, x in zip((rx, rx, ry, ry), nb):
            out.add_(x, alpha=sdc * q)
    else:
        torch.mul(c, k[0], out=out)
        for d in range(1, rad + 1):
            at = 1 + (d - 1) * 2 * ndim
            for q, x in zip(k[at:at + 2 * ndim], _neighbours(g, ndim, d)):
                out.add_(x, alpha=q)
        if kind == THERMAL:
            out.add_(p, alpha=k[7]).add_(k[6] * k[8])
    return out


def _sweep64(u, p, k, kind, ndim, steps, rad=1, keep=None):
    g, out = _Clamped(u, rad), torch.empty(u.shape, dtype=torch.float64, device=u.device)
    for _ in range(steps):
        if keep is not None:
            keep.append(g.c.clone())
        g.set(_advance(g, out, kind, ndim, k, p, rad))
    return g.c.clone()


def _transpose64(lam, cc, cw, ce, cs, cn):
    """A^T lam of one clamped five-point step."""
    out = lam * cc
    out[:, :-1].add_(lam[:, 1:], alpha=cw)   # x reads x-1
    out[:, 1:].add_(lam[:, :-1], alpha=ce)
    out[:-1].add_(lam[1:], alpha=cn)
    out[1:].add_(lam[:-1], alpha=cs)
    out[:, 0].add_(lam[:, 0], alpha=cw)      # a clamped read is the cell itself
    out[:, -1].add_(lam[:, -1], alpha=ce)
    out[0].add_(lam[0], alpha=cn)
    out[-1].add_(lam[-1], alpha=cs)
    return out


def _adjoint64(case, u, p, k, w):
    kind, states = case["kind"], []
    p = None if p is None else p.double()
    final = _sweep64(u, p, k, kind, 2, case["steps"], keep=states)
    lam = w.double()
    gk = torch.zeros(5, dtype=torch.float64, device=u.device)
    total = torch.zeros_like(lam)
    if kind == THERMAL:
        sdc, rx, ry, rz, amb = k
        weights = (1.0 - sdc * (2.0 * rx + 2.0 * ry + rz), sdc * rx, sdc * rx, sdc * ry, sdc * ry)
    else:
        weights = tuple(k)
    for state in reversed(states):
        g = _Clamped(state)
        x = _neighbours(g, 2)
        if kind == THERMAL:
            dx, dy, dz = x[0] + x[1] - 2.0 * state, x[2] + x[3] - 2.0 * state, amb - state
            terms = [p + dy * ry + dx * rx + dz * rz, dx * sdc, dy * sdc, dz * sdc]
            gk[4] += sdc * rz * lam.sum()
            total += lam
        else:
            terms = [state] + x
        for m, t in enumerate(terms):
            gk[m] += (lam * t).sum()
        lam = _transpose64(lam, *weights)
    return {"u": final, "grad_u": lam, "grad_coeffs": gk, "grad_power": total * k[0] if kind == THERMAL else None}


def exact(case, seed):
    if case["run"] == "batch":
        out = []
        for g in _batch_inputs(case, seed):
            p = None if g["power"] is None else g["power"].double()
            out.append(_sweep64(g["grid_in"], p, g["coeffs"], g["kind"], 2, g["steps"]))
        return out
    u, p, k, w = _inputs(case, seed)
    if case["run"] == "adjoint":
        return _adjoint64(case, u, p, k, w)
    p = None if p is None else p.double()
    return _sweep64(u, p, k, case["kind"], 3 if case["nz"] > 1 else 2, case["steps"], case["rad"])
