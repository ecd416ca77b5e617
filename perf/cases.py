"""The workloads this repository's speed is judged by, and their values in 64 bits.

Every case is work a user has the library do through ``paper_1308_0692_gb300.lbm``: marching
Couette channels and lid-driven cavities (first and second order, FP64 and FP32, small to
larger than the caches), a whole refined solve, batched sweeps, the hybrid coupling, training
steps of the warm-start network and a warm start.  ``listed`` names the cases, ``draw`` gives
others of the same ranges, ``prepare``/``run`` make and run one, ``work`` counts what a pass
cannot do without, ``exact`` evaluates it in plain 64-bit torch.
"""
from __future__ import annotations

import math
import os
import random

import numpy as np
import torch

from paper_1308_0692_gb300 import lbm

L2_BYTES = 126 << 20          # states that fit the L2 cache are read and written once per pass
FLOPS = 15                    # transport 5, moments 5, relaxation 5 per node-velocity update
FLOPS2 = 21                   # second-order transport: four products more
WIDTHS = (4, 256, 256, 256, 6)
MARCH_WARPS = {12: 6, 8: 4, 4: 2}      # warps of the tiled march by nodes per axis
PARAMS = os.path.join(os.path.dirname(os.path.abspath(lbm.__file__)), "data", "warmstart_mlp.npy")


# ---------------------------------------------------------------------------- the cases
def _step(name, geom, nx, ny, n, prec, steps, every=100, set_="half", kn=0.1, order=1, tiled=False):
    c = {"kind": "step", "geom": geom, "nx": nx, "ny": ny, "set": set_, "n": n, "prec": prec, "kn": kn,
         "steps": steps, "every": every, "order": order, "tiled": tiled}
    return {"name": name, **c} if name else c


def listed():
    return [
        _step("couette100_f64", "couette", 1, 100, 4, 64, 100),
        _step("cavity128_f64", "cavity", 128, 128, 4, 64, 100),
        _step("cavity333x251_f32", "cavity", 333, 251, 4, 32, 100, kn=1.0),
        _step("cavity512_q144_f64", "cavity", 512, 512, 6, 64, 10, every=10, kn=0.05),
        _step("cavity2048_q144_f32", "cavity", 2048, 2048, 6, 32, 10, every=10, kn=0.05, tiled=True),
        _step("second_order1024_f32", "cavity", 1024, 1024, 6, 32, 10, every=10, kn=0.05, order=2, tiled=True),
        {"name": "solve128_f32", "kind": "solve", "nx": 128, "ny": 128, "n": 4, "kn": 0.1, "steps": 300},
        {"name": "batch32x128_f32", "kind": "batch", "count": 32, "side": 128, "mixed": 0, "n": 4, "steps": 200},
        {"name": "batch_mixed24_f32", "kind": "batch", "count": 24, "side": 0, "mixed": 7, "n": 4, "steps": 200},
        {"name": "hybrid256_f64", "kind": "hybrid", "nx": 256, "ny": 256, "n": 4, "layer": 16, "prec": 64,
         "kn": 0.1, "steps": 100},
        {"name": "mlp_train8192", "kind": "train", "rows": 8192, "batches": 4},
        {"name": "warm_start128", "kind": "warm", "nx": 128, "ny": 128, "n": 4, "prec": 32},
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step", "step", "step", "step", "solve", "batch", "batch", "hybrid", "train", "warm"))
    kn = round(10.0 ** rng.uniform(-1.5, 1.0), 4)
    if kind == "step":
        shape = rng.choice(("couette", "cavity", "cavity", "march", "second"))
        if shape == "couette":
            return _step(None, "couette", 1, _between(rng, 33, 500), rng.choice((2, 4, 6)), rng.choice((64, 32)),
                         rng.choice((37, 100, 200)), kn=kn)
        if shape == "cavity":
            set_, n = rng.choice((("full", 3), ("half", 2), ("half", 3), ("half", 4), ("half", 6)))
            return _step(None, "cavity", _between(rng, 24, 600), _between(rng, 24, 600), n, rng.choice((64, 32)),
                         rng.choice((10, 37)), every=rng.choice((10, 100)), set_=set_, kn=kn)
        if shape == "march":
            return _step(None, "cavity", 64 * _between(rng, 2, 28), _between(rng, 100, 1800), rng.choice((2, 4, 6)), 32,
                         10, every=10, kn=kn, tiled=True)
        prec = rng.choice((64, 32))
        return _step(None, "cavity", 64 * _between(rng, 2, 12), _between(rng, 100, 700), rng.choice((4, 6)), prec, 10,
                     every=10, kn=kn, order=2, tiled=prec == 32)
    if kind == "solve":
        return {"kind": "solve", "nx": _between(rng, 32, 200), "ny": _between(rng, 32, 200),
                "n": rng.choice((2, 4)), "kn": kn, "steps": 100 * rng.randint(1, 3)}
    if kind == "batch":
        if rng.random() < 0.5:
            return {"kind": "batch", "count": _between(rng, 2, 64), "side": _between(rng, 48, 160), "mixed": 0,
                    "n": rng.choice((2, 4)), "steps": 100 * rng.randint(1, 2)}
        return {"kind": "batch", "count": 2 * _between(rng, 2, 24), "side": 0, "mixed": rng.randint(1, 1 << 20),
                "n": 4, "steps": 100 * rng.randint(1, 2)}
    if kind == "hybrid":
        return {"kind": "hybrid", "nx": _between(rng, 64, 400), "ny": _between(rng, 64, 400), "n": rng.choice((2, 4)),
                "layer": rng.randint(4, 24), "prec": rng.choice((64, 32)), "kn": kn, "steps": rng.choice((37, 100))}
    if kind == "train":
        return {"kind": "train", "rows": _between(rng, 1000, 32768), "batches": rng.randint(2, 4)}
    return {"kind": "warm", "nx": _between(rng, 40, 256), "ny": _between(rng, 40, 256), "n": rng.choice((2, 4)),
            "prec": rng.choice((64, 32))}


def _instances(case):
    """(geometry, nx, ny) of a batch's instances: equal cavities, or half channels and half cavities."""
    if not case["mixed"]:
        return [("cavity", case["side"], case["side"])] * case["count"]
    r = random.Random(case["mixed"])
    return [("couette", 1, r.randint(64, 512)) if i < case["count"] // 2 else ("cavity",) + (r.choice((64, 96, 128, 192, 256)),) * 2
            for i in range(case["count"])]


def work(case):
    kind = case["kind"]
    if kind in ("step", "solve", "batch"):
        m = case["n"] if case.get("set") == "full" else 2 * case["n"]
        cells = sum(nx * ny for _, nx, ny in _instances(case)) if kind == "batch" else case["nx"] * case["ny"]
        unknowns, es = cells * m * m, case.get("prec", 32) // 8
        steps = case["steps"] * (2 if kind == "solve" else 1)
        passes = steps if unknowns * es > L2_BYTES else 1
        out = 24.0 * cells if kind == "batch" else 0.0
        return {"bytes": 2.0 * es * unknowns * passes + out,
                "flops": float(FLOPS2 if case.get("order") == 2 else FLOPS) * unknowns * steps}
    if kind == "hybrid":
        half = int(_half_cells(case["nx"], case["ny"], case["layer"]).sum())
        n = case["n"]
        unknowns = half * 4 * n * n + (case["nx"] * case["ny"] - half) * n * n
        return {"bytes": 2.0 * case["prec"] / 8 * unknowns, "flops": float(FLOPS) * unknowns * case["steps"]}
    params = sum(a * b + b for a, b in zip(WIDTHS[:-1], WIDTHS[1:]))
    madds = sum(a * b for a, b in zip(WIDTHS[:-1], WIDTHS[1:]))
    if kind == "train":
        rows, k = case["rows"], case["batches"]
        return {"bytes": 40.0 * rows * k + 24.0 * params, "flops": 2.0 * k * rows * (3 * madds - WIDTHS[0] * WIDTHS[1])}
    cells = case["nx"] * case["ny"]
    nv = 4 * case["n"] ** 2
    return {"bytes": 4.0 * params + float(cells * nv * case["prec"] // 8), "flops": 2.0 * cells * (madds + 6 * nv)}


# ------------------------------------------------------------------- inputs and one pass
def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _smooth(g, k, ny, nx):
    """k smooth random fields [k, ny, nx] of order one."""
    coarse = torch.randn((1, k, 9, 9), generator=g, device="cuda", dtype=torch.float64)
    return torch.nn.functional.interpolate(coarse, size=(ny, nx), mode="bilinear", align_corners=True)[0]


def _initial_state(case, seed, dtype, out):
    """Perturbation state [n, ny, nx]: a Hermite expansion of smooth random moments with a tenth
    of noise per velocity."""
    x, w = _rule(case["set"], case["n"])
    g = _generator(seed)
    nx, ny, m = case["nx"], case["ny"], len(x)
    f = _smooth(g, 6, ny, nx).float()
    for a in range(m * m):
        ex, ey = x[a % m], x[a // m]
        v = f[0] + ex * f[1] + ey * f[2] + 0.5 * ((ex * ex - 1) * f[3] + 2 * ex * ey * f[4] + (ey * ey - 1) * f[5])
        v += 0.1 * torch.randn((ny, nx), generator=g, device="cuda")
        out[a] = (w[a % m] * w[a // m] * v).to(dtype)
    return out


def _problem(case, geom=None, kn=None, u=(0.0, 0.01), nx=None, ny=None, every=100):
    couette = (geom or case.get("geom")) == "couette"
    return lbm.make_problem(lbm.LBM_COUETTE if couette else lbm.LBM_CAVITY, nx or case["nx"], ny or case["ny"],
                            kn or case.get("kn", 0.1), u[0], u[1],
                            prec=lbm.LBM_FP64 if case.get("prec", 32) == 64 else lbm.LBM_FP32_PERTURB,
                            residual_every=every)


def _walls(case):
    return (0.01, -0.01) if case.get("geom") == "couette" else (0.0, 0.01)


def _sim(case, every=100):
    half = case.get("set", "half") == "half"
    vs = lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH if half else lbm.LBM_FULL_RANGE_GH, case["n"])
    prob = _problem(case, u=_walls(case), every=every)
    buf = torch.empty(lbm.lbm_sim_bytes(vs, prob), dtype=torch.uint8, device="cuda")
    return vs, buf, lbm.lbm_init(vs, prob, device_buf=buf, stream=lbm.PrivateStream())


def _planar(case, buf, sim):
    """The current planar state [n, ny, nx] as a view of the simulation's buffer."""
    dtype = torch.float64 if case.get("prec", 32) == 64 else torch.float32
    at = lbm.lbm_state_device(sim)[0] - buf.data_ptr()
    count = sim.n_vel * sim.ncells
    return buf[at:at + count * dtype.itemsize].view(dtype).view(sim.n_vel, case["ny"], case["nx"])


def _tiles(case, buf, sim):
    """The current strip-tiled state without its padding: the left half tile, the whole tiles, the
    right half tile, each [tiles, ny, n, cells]."""
    width, shift, pitch, _ = lbm.lbm_state_tiling(sim)
    tiles = (case["nx"] + shift + width - 1) // width
    at = lbm.lbm_state_device(sim)[0] - buf.data_ptr()
    t = buf[at:at + 4 * tiles * pitch].view(torch.float32).view(tiles, case["ny"], sim.n_vel, width)
    return t[:1, :, :, shift:], t[1:-1], t[-1:, :, :, :shift]


def _batch_pairs(case, seed):
    r = np.random.default_rng(seed)
    return [(float(10.0 ** r.uniform(-2.0, 1.0)), float(r.uniform(0.005, 0.02))) for _ in range(case["count"])]


def _moment_fields(case, seed):
    """Physical moments rho, u, P [6, ny, nx] (host) of a gently disturbed gas."""
    f = 0.01 * _smooth(_generator(seed), 6, case["ny"], case["nx"]).cpu().numpy()
    f[[0, 3, 5]] += 1.0
    return f


def _hybrid_state(case, seed):
    """Packed host state: smooth moments in every cell's own set and a tenth of noise."""
    half = _half_cells(case["nx"], case["ny"], case["layer"]).reshape(-1)
    f = _smooth(_generator(seed), 3, case["ny"], case["nx"]).cpu().numpy().reshape(3, -1)
    r = np.random.default_rng(seed)
    parts = {}
    for kind, mask in (("half", half), ("full", ~half)):
        x, w = _rule(kind, case["n"])
        wx, ex, ey = np.outer(w, w).ravel(), np.tile(x, len(x)), np.repeat(x, len(x))
        v = f[0, mask, None] + ex * f[1, mask, None] + ey * f[2, mask, None]
        parts[kind] = wx * (v + 0.1 * r.standard_normal(v.shape))
    return _pack(half, parts["half"], parts["full"], np)


def _mlp_params(seed):
    r = np.random.default_rng(seed)
    return np.concatenate([r.uniform(-1, 1, a * b + b) / math.sqrt(a) for a, b in zip(WIDTHS[:-1], WIDTHS[1:])]).astype(np.float32)


def _rows(case, seed):
    """Minibatches of features [k, rows, 4] and of targets [k, rows, 6] that are smooth in them."""
    g = _generator(seed)
    x = 2 * torch.rand((case["batches"], case["rows"], 4), generator=g, device="cuda") - 1
    a = torch.randn((4, 6), generator=g, device="cuda")
    return x, 0.3 * torch.sin(2 * x @ a) + 0.01 * torch.randn(x.shape[:2] + (6,), generator=g, device="cuda")


def _pair(seed):
    r = np.random.default_rng(seed)
    return float(10.0 ** r.uniform(-2.0, 1.0)), float(r.uniform(0.005, 0.02))


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind == "step":
        s["vs"], s["buf"], s["sim"] = _sim(case, case["every"])
        state = _planar(case, s["buf"], s["sim"])
        _initial_state(case, seed, state.dtype, state)
        torch.cuda.synchronize()
        if case["order"] == 2:
            lbm.lbm_set_splitting(s["sim"], lbm.LBM_SPLIT_STRANG_EXACT)
            lbm.lbm_set_transport(s["sim"], 2)
        if case["tiled"]:
            lbm.lbm_set_variant(s["sim"], MARCH_WARPS[2 * case["n"]], 9)
    elif kind == "solve":
        s["vs"], s["buf"], s["sim"] = _sim(case)
        s["moments"] = _moment_fields(case, seed)
    elif kind == "batch":
        pairs = _batch_pairs(case, seed)
        inst = _instances(case)
        s["vs"] = lbm.lbm_make_velocity_set(lbm.LBM_HALF_RANGE_GH, case["n"])
        probs = [_problem(case, geom, kn, (uw, -uw) if geom == "couette" else (0.0, uw), nx, ny)
                 for (geom, nx, ny), (kn, uw) in zip(inst, pairs)]
        s["stream"] = torch.cuda.Stream()
        s["batch"] = lbm.lbm_batch_init(s["vs"], probs, stream=s["stream"])
        cells = [nx * ny for _, nx, ny in inst]
        s["at"] = [48 * sum(cells[:i]) for i in range(len(cells))]
        s["moments"] = torch.empty(6 * sum(cells), dtype=torch.float64, device="cuda")
        s["rest"], s["speed"] = _scales(cells, pairs)
    elif kind == "hybrid":
        s["stream"] = torch.cuda.Stream()
        s["hybrid"] = lbm.lbm_hybrid_init(lbm.LBM_CAVITY, case["n"], case["nx"], case["ny"], case["kn"], 0.0, 0.01,
                                          case["layer"], stream=s["stream"])
        lbm.lbm_hybrid_set_state(s["hybrid"], _hybrid_state(case, seed))
        if case["prec"] == 32:
            lbm.lbm_hybrid_set_precision(s["hybrid"], lbm.LBM_FP32_PERTURB)
    elif kind == "train":
        s["mlp"] = lbm.lbm_mlp_create(case["rows"], seed=0, stream=torch.cuda.Stream())
        lbm.lbm_mlp_set_params(s["mlp"], _mlp_params(seed))
        s["x"], s["t"] = _rows(case, seed)
    else:
        s["vs"], s["buf"], s["sim"] = _sim(case)
        s["mlp"] = lbm.lbm_mlp_create(case["nx"] * case["ny"], seed=0, stream=torch.cuda.Stream())
        lbm.lbm_mlp_set_params(s["mlp"], np.load(PARAMS))
        s["pair"] = _pair(seed)
    torch.cuda.synchronize()
    return s


def _scales(cells, pairs):
    """Rest values and wall speeds beside the flat moments of a batch's instances."""
    rest = torch.tensor([1.0, 0.0, 0.0, 1.0, 0.0, 1.0], dtype=torch.float64, device="cuda")
    return (torch.cat([rest.repeat_interleave(c) for c in cells]),
            torch.cat([torch.full((6 * c,), uw, dtype=torch.float64, device="cuda") for c, (_, uw) in zip(cells, pairs)]))


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "step":
        lbm.lbm_step(s["sim"], case["steps"])
        return _tiles(case, s["buf"], s["sim"]) if case["tiled"] else _planar(case, s["buf"], s["sim"])
    if kind == "solve":
        lbm.lbm_set_moments(s["sim"], s["moments"])
        lbm.lbm_solve(s["sim"], 1e-13, case["steps"], 1, 1e-13)
        return _planar(case, s["buf"], s["sim"])
    if kind == "batch":
        lbm.lbm_batch_advance(s["batch"], case["steps"], 0.0)
        base = s["moments"].data_ptr()
        for i, at in enumerate(s["at"]):
            lbm.lbm_batch_moments(s["batch"], i, base + at)
        with torch.cuda.stream(s["stream"]):
            return ((s["moments"] - s["rest"]) / s["speed"]).float()
    if kind == "hybrid":
        lbm.lbm_hybrid_step(s["hybrid"], case["steps"])
        u = np.stack(lbm.lbm_hybrid_velocity(s["hybrid"]))
        return u if case["prec"] == 64 else u.astype(np.float32)
    if kind == "train":
        for x, t in zip(s["x"], s["t"]):
            lbm.lbm_mlp_train_step(s["mlp"], x.data_ptr(), t.data_ptr(), case["rows"], 1e-3)
        return lbm.lbm_mlp_get_params(s["mlp"])
    lbm.lbm_warm_start(s["sim"], s["mlp"], *s["pair"])
    return _planar(case, s["buf"], s["sim"])


# --------------------------------------------------------------- the same in 64-bit torch
def _rule(kind, n):
    """1-D nodes (ascending) and weights of exp(-x^2/2)/sqrt(2 pi): Gauss-Hermite on the line, or
    the Gauss rule of the half line, mirrored (its recurrence by the Stieltjes procedure on a
    fine Gauss-Legendre grid)."""
    if kind == "full":
        x, w = np.polynomial.hermite_e.hermegauss(n)
        return x, w / math.sqrt(2 * math.pi)
    t, q = np.polynomial.legendre.leggauss(400)
    t = 10.0 * (t + 1.0)
    q = 10.0 * q * np.exp(-0.5 * t * t) / math.sqrt(2 * math.pi)
    a, b = np.zeros(n), np.zeros(n)
    p0, p1, norm0 = np.zeros_like(t), np.ones_like(t), 1.0
    for k in range(n):
        norm = np.sum(q * p1 * p1)
        a[k], b[k] = np.sum(q * t * p1 * p1) / norm, norm / norm0
        p0, p1, norm0 = p1, (t - a[k]) * p1 - (b[k] if k else 0.0) * p0, norm
    x, v = np.linalg.eigh(np.diag(a) + np.diag(np.sqrt(b[1:]), 1) + np.diag(np.sqrt(b[1:]), -1))
    w = np.sum(q) * v[0] ** 2
    return np.concatenate([-x[::-1], x]), np.concatenate([w[::-1], w])


class _March:
    """The scheme on one grid in FP64 torch: upwind transport of first or second order, diffuse
    walls, relaxation; state [n, ny, nx]."""

    def __init__(self, rule, geom, nx, ny, kn, ub, ut, order=1, device="cuda"):
        self.x, self.w = rule
        self.m, self.order, self.cavity = len(self.x), order, geom == "cavity"
        mx = float(np.abs(self.x).max())
        dy = 1.0 / ny
        dx = 1.0 / nx if self.cavity else dy
        column = not self.cavity and nx == 1
        dt = min(0.9 / (mx / dy + (0.0 if column else mx / dx)), kn)
        self.omega = 1.0 - math.exp(-dt / kn) if order == 2 else dt / kn
        self.uref = max(abs(ub), abs(ut)) or 1.0
        self.ub, self.ut = ub, ut
        t = lambda v: torch.as_tensor(v, dtype=torch.float64, device=device)  # noqa: E731
        self.tx, self.tw = t(self.x), t(self.w)
        self.nux, self.nuy = (0.0 if column else dt / dx) * self.tx.abs(), dt / dy * self.tx.abs()
        self.norm = float(np.sum(np.where(self.x > 0, self.x * self.w, 0.0)) * np.sum(self.w))
        self.low, self.high = int(np.sum(self.x < 0)), int(np.sum(self.x <= 0))

    def _face(self, h, inner, nu):
        """Value a population leaves through a wall face with: first order, or extrapolated."""
        return h if self.order == 1 else h + 0.5 * (1 - nu) * (h - inner)

    def _densities(self, h):
        """Wall densities (Eq. 9) of bottom, top [nx], left, right [ny]."""
        m = self.m
        v = h.view(m, m, *h.shape[1:])               # [iy, ix, y, x]
        lo, hi = slice(0, self.low), slice(self.high, m)
        ny_ = self.nuy.view(m, 1, 1)
        nx_ = self.nux.view(1, m, 1)
        e = self.tx.abs()
        bottom = self._face(v[lo, :, 0], v[lo, :, 1], ny_[lo])
        top = self._face(v[hi, :, -1], v[hi, :, -2], ny_[hi])
        out = [(e[lo].view(-1, 1, 1) * bottom).sum((0, 1)), (e[hi].view(-1, 1, 1) * top).sum((0, 1)), None, None]
        if self.cavity:
            left = self._face(v[:, lo, :, 0], v[:, lo, :, 1], nx_[:, lo])
            right = self._face(v[:, hi, :, -1], v[:, hi, :, -2], nx_[:, hi])
            out[2:] = [(e[lo].view(1, -1, 1) * left).sum((0, 1)), (e[hi].view(1, -1, 1) * right).sum((0, 1))]
        return [None if d is None else d / self.norm for d in out]

    def _moved(self, h, dim, up, nu, ghost):
        """Change of h [k, ny, nx] by transport along `dim` towards larger (up) or smaller indices;
        ghost: the wall's populations, or None (periodic)."""
        n = h.shape[dim]
        if not up:
            h = h.flip(dim)
        if ghost is None:
            return _unflip(nu * (h.roll(1, dim) - h), dim, up) if self.order == 1 else _unflip(
                (lambda f: f.roll(1, dim) - f)(nu * (h + 0.5 * (1 - nu) * (h - h.roll(1, dim)))), dim, up)
        flux = nu * h
        if self.order == 2:
            flux = torch.cat([flux.narrow(dim, 0, 1), flux.narrow(dim, 1, n - 1) + nu * 0.5 * (1 - nu) * (
                h.narrow(dim, 1, n - 1) - h.narrow(dim, 0, n - 1))], dim)
        inflow = torch.cat([nu * ghost.unsqueeze(dim), flux.narrow(dim, 0, n - 1)], dim)
        return _unflip(inflow - flux, dim, up)

    def step(self, h):
        m = self.m
        rb, rt, rl, rr = self._densities(h)
        out = torch.empty_like(h)
        rho = jx = jy = 0.0
        col = self.tx.view(m, 1)
        for iy in range(m):
            b = h[iy * m:(iy + 1) * m]
            wa = (self.w[iy] * self.tw).view(m, 1)
            v = b.clone()
            for part, up, wall in ((slice(0, self.low), False, rr), (slice(self.high, m), True, rl)):
                ghost = wa[part] * wall if self.cavity else None
                v[part] += self._moved(b[part], 2, up, self.nux[part].view(-1, 1, 1), ghost)
            if self.x[iy] != 0.0 and not (self.low <= iy < self.high):
                up = self.x[iy] > 0
                u, wall = (self.ub, rb) if up else (self.ut, rt)
                v += self._moved(b, 1, up, float(self.nuy[iy]), wa * (wall * (1 + col * u) + col * u / self.uref))
            out[iy * m:(iy + 1) * m] = v
            r = v.sum(0)
            rho, jx, jy = rho + r, jx + (self.tx.view(m, 1, 1) * v).sum(0), jy + self.x[iy] * r
        for iy in range(m):
            wa = (self.w[iy] * self.tw).view(m, 1, 1)
            eq = wa * ((rho + self.x[iy] * jy) + self.tx.view(m, 1, 1) * jx)
            out[iy * m:(iy + 1) * m].mul_(1.0 - self.omega).add_(eq, alpha=self.omega)
        return out

    def march(self, h, steps):
        for _ in range(steps):
            h = self.step(h)
        return h

    def moments(self, h):
        """rho, u, P [6, ny, nx] in physical units."""
        m = self.m
        v = h.view(m, m, *h.shape[1:])
        r, c = v.sum(1), v.sum(0)                    # row sums by iy, column sums by ix
        e = self.tx.view(m, 1, 1)
        pxy = (e * (e.view(1, m, 1, 1) * v).sum(1)).sum(0)
        rho = 1 + self.uref * r.sum(0)
        return torch.stack([rho, self.uref * (e * c).sum(0) / rho, self.uref * (e * r).sum(0) / rho,
                            1 + self.uref * (e * e * c).sum(0), self.uref * pxy, 1 + self.uref * (e * e * r).sum(0)])


def _unflip(v, dim, up):
    return v if up else v.flip(dim)


def _hermite(rule, f):
    """Second-order Hermite expansion of rho', j', P' [6, ...] on the tensor set."""
    x, w = rule
    m = len(x)
    out = torch.empty((m * m,) + tuple(f.shape[1:]), dtype=torch.float64, device=f.device)
    for a in range(m * m):
        ex, ey = x[a % m], x[a // m]
        out[a] = w[a % m] * w[a // m] * (f[0] + ex * f[1] + ey * f[2] + 0.5 * (
            (f[3] - f[0]) * (ex * ex - 1) + 2 * f[4] * ex * ey + (f[5] - f[0]) * (ey * ey - 1)))
    return out


def _half_cells(nx, ny, layer):
    x, y = np.arange(nx), np.arange(ny)
    return np.minimum(np.minimum(x, nx - 1 - x)[None, :], np.minimum(y, ny - 1 - y)[:, None]) < layer


def _pack(half, h, f, lib):
    """Cell after cell, each cell's values in its own set's order (h, f: rows of the two kinds)."""
    sizes = np.where(half, h.shape[1], f.shape[1])
    at = np.concatenate([[0], np.cumsum(sizes)])
    out = lib.empty(int(at[-1]), dtype=h.dtype)
    for mask, v in ((half, h), (~half, f)):
        out[at[:-1][mask][:, None] + np.arange(v.shape[1])] = v
    return out


class _Hybrid:
    """The half-range / full-range coupling in FP64 torch, both sets kept on the whole grid."""

    def __init__(self, n, nx, ny, layer, kn, u_top, device="cuda"):
        t = lambda v: torch.as_tensor(v, dtype=torch.float64, device=device)  # noqa: E731
        self.half_np = _half_cells(nx, ny, layer)
        self.half = torch.as_tensor(self.half_np, device=device)
        rules = [_rule("half", n), _rule("full", n)]
        present = [r for r, used in zip(rules, (self.half_np.any(), not self.half_np.all())) if used]
        mx = max(float(np.abs(x).max()) for x, _ in present)
        self.dt = min(0.9 / (mx * nx + mx * ny), kn)
        self.rate, self.omega, self.ut = (self.dt * nx, self.dt * ny), self.dt / kn, u_top
        self.sets, he = [], []
        for x, w in rules:
            ex, ey, ww = np.tile(x, len(x)), np.repeat(x, len(x)), np.outer(w, w).ravel()
            tab = np.zeros((n, len(x)))
            for k in range(n):
                tab[k] = 1.0 if k == 0 else x if k == 1 else x * tab[k - 1] - (k - 1) * tab[k - 2]
            he.append((np.stack([np.tile(tab[i], len(x)) * np.repeat(tab[j], len(x)) for i in range(n) for j in range(n)]), ww))
            self.sets.append((t(ex), t(ey), t(ww), float(np.sum(np.where(ex > 0, ex * ww, 0.0)))))
        fact = np.array([math.factorial(i) * math.factorial(j) for i in range(n) for j in range(n)], dtype=float)
        self.to_full = t((he[1][0].T / fact) @ he[0][0] * he[1][1][:, None])
        self.to_half = t((he[0][0].T / fact) @ he[1][0] * he[0][1][:, None])

    def _flux(self, k, v, axis, positive):
        """(mass, x, y momentum) carried along +axis or -axis by the populations v of set k."""
        e = self.sets[k][axis]
        t = torch.where((e > 0) if positive else (e < 0), e.abs(), 0.0).view(-1, 1, 1) * v
        return torch.stack([t.sum(0), (self.sets[k][0].view(-1, 1, 1) * t).sum(0), (self.sets[k][1].view(-1, 1, 1) * t).sum(0)])

    def step(self, h, f):
        half = self.half
        hh = torch.where(half, h, torch.einsum("ab,byx->ayx", self.to_half, f))
        ff = torch.where(half, torch.einsum("ab,byx->ayx", self.to_full, h), f)
        out = []
        for k, v in ((0, hh), (1, ff)):
            ex, ey, w, norm = self.sets[k]
            new = v.clone()
            for axis, e, dim in ((0, ex, 2), (1, ey, 1)):
                for up in (True, False):
                    part = (e > 0) if up else (e < 0)
                    b, nu = v[part], self.rate[axis] * e[part].abs().view(-1, 1, 1)
                    edge = v.select(dim, 0 if up else -1)
                    leaves = (e < 0) if up else (e > 0)
                    dens = (e[leaves].abs().view(-1, 1) * edge[leaves]).sum(0) / norm
                    along = (ey if axis == 0 else ex)[part].view(-1, 1)
                    u = self.ut if axis == 1 and not up else 0.0
                    ghost = w[part].view(-1, 1) * (dens * (1 + along * u) + along * (u / self.ut))
                    n = b.shape[dim]
                    seen = torch.cat([ghost.unsqueeze(dim), b.narrow(dim, 0, n - 1)] if up
                                     else [b.narrow(dim, 1, n - 1), ghost.unsqueeze(dim)], dim)
                    new[part] += nu * (seen - b)
            if k == 1:
                for axis, dim in ((0, 2), (1, 1)):
                    up_h, dn_h = self._flux(0, hh, axis, True), self._flux(0, hh, axis, False)
                    up_f, dn_f = self._flux(1, ff, axis, True), self._flux(1, ff, axis, False)
                    for lower in (True, False):        # the neighbour on the lower or the upper side
                        there = lambda a: a.roll(1 if lower else -1, a.dim() - 3 + dim)  # noqa: E731
                        face = ~half & half.roll(1 if lower else -1, dim - 1)
                        n = half.shape[dim - 1]
                        inside = torch.arange(n, device=half.device) != (0 if lower else n - 1)
                        face &= inside.view((1, -1) if dim == 2 else (-1, 1))
                        want = there(up_h) - dn_h if lower else there(dn_h) - up_h
                        have = there(up_f) - dn_f if lower else there(dn_f) - up_f
                        d = torch.where(face, self.rate[axis] * (want - have), 0.0)
                        new += w.view(-1, 1, 1) * (d[0] + ex.view(-1, 1, 1) * d[1] + ey.view(-1, 1, 1) * d[2])
            ex, ey, w = (q.view(-1, 1, 1) for q in (ex, ey, w))
            eq = w * (new.sum(0) + ex * (ex * new).sum(0) + ey * (ey * new).sum(0))
            out.append(new - self.omega * (new - eq))
        return out

    def velocity(self, h, f):
        u = []
        for k, v in ((0, h), (1, f)):
            rho = 1 + self.ut * v.sum(0)
            u.append([self.ut * (e.view(-1, 1, 1) * v).sum(0) / rho for e in self.sets[k][:2]])
        return torch.stack([torch.where(self.half, a, b) for a, b in zip(*u)])


def _network(params):
    out, at = [], 0
    for a, b in zip(WIDTHS[:-1], WIDTHS[1:]):
        out.append((params[at:at + a * b].view(b, a), params[at + a * b:at + a * b + b]))
        at += a * b + b
    return out


def _forward(params, x):
    for i, (w, b) in enumerate(_network(params)):
        x = x @ w.T + b
        if i + 2 < len(WIDTHS):
            x = 0.5 * x * (1 + torch.erf(x / math.sqrt(2.0)))
    return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        dtype = torch.float64 if case["prec"] == 64 else torch.float32
        rule = _rule(case["set"], case["n"])
        h = torch.empty((len(rule[0]) ** 2, case["ny"], case["nx"]), dtype=dtype, device="cuda")
        h = _initial_state(case, seed, dtype, h).double()
        h = _March(rule, case["geom"], case["nx"], case["ny"], case["kn"], *_walls(case), case["order"]).march(h, case["steps"])
        if not case["tiled"]:
            return h
        inner = h[:, :, 32:-32].unflatten(2, (-1, 64)).permute(2, 1, 0, 3)
        return h[None, :, :, :32].permute(0, 2, 1, 3), inner, h[None, :, :, -32:].permute(0, 2, 1, 3)
    if kind == "solve":
        rule = _rule("half", case["n"])
        f = torch.as_tensor(_moment_fields(case, seed), device="cuda")
        rho = f[0]
        f = torch.stack([rho - 1, rho * f[1], rho * f[2], f[3] - 1, f[4], f[5] - 1]) / 0.01
        # the correction march from the defect adds the steps the march itself would take
        return _March(rule, "cavity", case["nx"], case["ny"], case["kn"], 0.0, 0.01).march(_hermite(rule, f), 2 * case["steps"])
    if kind == "batch":
        rule = _rule("half", case["n"])
        inst, pairs = _instances(case), _batch_pairs(case, seed)
        out = []
        for (geom, nx, ny), (kn, uw) in zip(inst, pairs):
            m = _March(rule, geom, nx, ny, kn, *((uw, -uw) if geom == "couette" else (0.0, uw)))
            h = torch.zeros((4 * case["n"] ** 2, ny, nx), dtype=torch.float64, device="cuda")
            out.append(m.moments(m.march(h, case["steps"])).reshape(-1))
        rest, speed = _scales([nx * ny for _, nx, ny in inst], pairs)
        return (torch.cat(out) - rest) / speed
    if kind == "hybrid":
        m = _Hybrid(case["n"], case["nx"], case["ny"], case["layer"], case["kn"], 0.01)
        packed = _hybrid_state(case, seed)
        half = m.half_np.reshape(-1)
        sizes = np.where(half, 4 * case["n"] ** 2, case["n"] ** 2)
        at = np.concatenate([[0], np.cumsum(sizes)])[:-1]
        state = []
        for mask, n in ((half, 4 * case["n"] ** 2), (~half, case["n"] ** 2)):
            v = np.zeros((half.size, n))
            v[mask] = packed[at[mask][:, None] + np.arange(n)]
            state.append(torch.as_tensor(v.T.reshape(n, case["ny"], case["nx"]).copy(), device="cuda"))
        for _ in range(case["steps"]):
            state = m.step(*state)
        return m.velocity(*state)
    if kind == "train":
        p = torch.as_tensor(_mlp_params(seed), device="cuda").double().requires_grad_()
        opt = torch.optim.Adam([p], lr=1e-3, betas=(0.9, 0.999), eps=1e-8)
        for x, t in zip(*_rows(case, seed)):
            opt.zero_grad()
            (_forward(p, x.double()) - t.double()).square().mean().backward()
            opt.step()
        return p.detach()
    kn, uw = _pair(seed)
    nx, ny = case["nx"], case["ny"]
    gx = 2 * (torch.arange(nx, device="cuda", dtype=torch.float64) + 0.5) / nx - 1
    gy = 2 * (torch.arange(ny, device="cuda", dtype=torch.float64) + 0.5) / ny - 1
    x = torch.stack([gx.expand(ny, nx), gy.view(ny, 1).expand(ny, nx), torch.full((ny, nx), (2 * math.log10(kn) + 1) / 3, device="cuda", dtype=torch.float64),
                     torch.full((ny, nx), (uw - 0.0125) / 0.0075, device="cuda", dtype=torch.float64)], -1)
    f = _forward(torch.as_tensor(np.load(PARAMS), device="cuda").double(), x).permute(2, 0, 1)
    return _hermite(_rule("half", case["n"]), uw / 0.01 * f)
