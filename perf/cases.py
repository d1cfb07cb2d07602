"""What is timed: time steps of the B-char library over the range it is used in.

A step is what a time-stepping program calls per step: ``Mesh.set_velocity``
(device-resident face velocities times the step's time factor) and
``Mesh.step`` with the library's default tolerances; ``batch`` cases step
several handles at once, ``serve`` cases run a short request stream.  Meshes,
fields, porosities and initial concentrations follow the recipes of
``paper_1908_05834_gb300.inputs`` (sizes per axis may differ); the seed draws
the widths, the porosity, the position of c0 and the time factor.

``exact`` recomputes a step in 64 bits with plain torch: absolute coordinates,
one pass per candidate cell offset, dense normal equations.
"""
from __future__ import annotations

import math

import numpy as np
import torch

# ---------------------------------------------------------------- the cases


def listed():
    return [
        # the plain 32x32 configuration: FP64 throughout, the smallest call, latency alone
        {"name": "vortex32_fp64", "kind": "step", "dim": 2, "n0": 32, "n1": 32, "n2": 1, "mesh": "uniform",
         "precision": "fp64", "c": "f64", "cfl": 0.32},
        # the smallest 2D request of the serving stream
        {"name": "vortex64_split", "kind": "step", "dim": 2, "n0": 64, "n1": 64, "n2": 1, "mesh": "uniform",
         "precision": "split", "c": "f64", "cfl": 2.0},
        # an ordinary 2D request (the stream's sizes are log-uniform in 64..1024 per axis)
        {"name": "vortex160_split", "kind": "step", "dim": 2, "n0": 160, "n1": 160, "n2": 1, "mesh": "uniform",
         "precision": "split", "c": "f64", "cfl": 2.0},
        # the stretched single vortex (the flagship recipe) at a coarse resolution
        {"name": "stretched96_split", "kind": "step", "dim": 2, "n0": 96, "n1": 96, "n2": 1, "mesh": "stretched",
         "precision": "split", "c": "f64", "cfl": 1.0},
        # the same recipe on a ragged mesh at the flagship's CFL number
        {"name": "stretched131x117_split", "kind": "step", "dim": 2, "n0": 131, "n1": 117, "n2": 1,
         "mesh": "stretched", "precision": "split", "c": "f64", "cfl": 5.12},
        # a small porous 3D mesh, FP64 throughout (the parity configuration)
        {"name": "porous16_fp64", "kind": "step", "dim": 3, "n0": 16, "n1": 16, "n2": 16, "mesh": "uniform",
         "precision": "fp64", "c": "f64", "cfl": 2.0},
        # the smallest 3D request of the serving stream
        {"name": "porous32_split", "kind": "step", "dim": 3, "n0": 32, "n1": 32, "n2": 32, "mesh": "uniform",
         "precision": "split", "c": "f64", "cfl": 2.0},
        # the large 3D recipe (stretched, wide porosity range, c stored in FP32), small and ragged
        {"name": "stretched23x22x22_f32", "kind": "step", "dim": 3, "n0": 23, "n1": 22, "n2": 22,
         "mesh": "stretched", "precision": "split", "c": "f32", "cfl": 4.0},
        # several independent problems of uneven size stepped at once
        {"name": "batch_uneven", "kind": "batch", "count": 4, "cells": 2500, "precision": "split", "c": "f64",
         "cfl": 1.5},
        # a short request stream: admission, mesh set-up, steps, results back on the host
        {"name": "serve_short", "kind": "serve", "count": 3, "cells": 2000, "steps": 1, "precision": "split",
         "c": "f64", "cfl": 1.5},
        # the flagship mesh with the alternating scalings and the column fix only (no minimisation):
        # tracking, intersections, assembly, balancing, scalings and update at full size
        {"name": "scalings1024_split", "kind": "scalings", "dim": 2, "n0": 1024, "n1": 1024, "n2": 1,
         "mesh": "stretched", "precision": "split", "c": "f64", "cfl": 5.12},
        # the same for the porous 3D workload, c stored in FP32
        {"name": "scalings96x3d_f32", "kind": "scalings", "dim": 3, "n0": 96, "n1": 96, "n2": 96, "mesh": "uniform",
         "precision": "split", "c": "f32", "cfl": 19.2},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["2d", "2d", "2ds", "2ds", "3d", "3d", "3ds", "batch", "serve", "s2d", "s3d"])
    cfl = round(math.exp(rng.uniform(math.log(0.3), math.log(5.0))), 3)
    if kind in ("2d", "2ds"):
        n = _log_int(rng, 32, 140 if kind == "2d" else 90)
        return {"kind": "step", "dim": 2, "n0": n, "n1": max(24, int(n * rng.uniform(0.7, 1.0))), "n2": 1,
                "mesh": "uniform" if kind == "2d" else "stretched", "precision": rng.choice(["fp64", "split", "split"]),
                "c": "f64", "cfl": cfl}
    if kind in ("3d", "3ds"):
        n = _log_int(rng, 10, 25 if kind == "3d" else 20)
        # stretched: near-cubes, as the recipe has them (the widths alone vary by 1.3 / 0.7)
        n1, n2 = ((max(8, int(n * rng.uniform(0.7, 1.0))) for _ in range(2)) if kind == "3d"
                  else (n - (n >= 16) * rng.randint(0, 1) for _ in range(2)))
        return {"kind": "step", "dim": 3, "n0": n, "n1": n1, "n2": n2, "mesh": "uniform" if kind == "3d" else "stretched",
                "precision": rng.choice(["fp64", "split", "split"]) if kind == "3d" else "split",
                "c": "f64" if kind == "3d" else "f32", "cfl": min(cfl, 4.0)}
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(2, 4), "cells": _log_int(rng, 600, 2500),
                "precision": "split", "c": "f64", "cfl": min(cfl, 4.0)}
    if kind == "serve":
        return {"kind": "serve", "count": rng.randint(1, 3), "cells": _log_int(rng, 600, 2000),
                "steps": 1, "precision": "split", "c": "f64", "cfl": min(cfl, 4.0)}
    if kind == "s2d":
        n = _log_int(rng, 300, 1024)
        return {"kind": "scalings", "dim": 2, "n0": n, "n1": int(n * rng.uniform(0.7, 1.0)), "n2": 1,
                "mesh": rng.choice(["uniform", "stretched"]), "precision": "split", "c": rng.choice(["f64", "f32"]),
                "cfl": cfl}
    n = _log_int(rng, 40, 90)
    return {"kind": "scalings", "dim": 3, "n0": n, "n1": int(n * rng.uniform(0.7, 1.0)),
            "n2": int(n * rng.uniform(0.7, 1.0)), "mesh": "uniform", "precision": "split",
            "c": rng.choice(["f64", "f32"]), "cfl": round(rng.uniform(1.0, 19.0), 2)}


# ---------------------------------------------------------------- inputs


def _problem(dim, n, mesh, cfl, seed):
    """(coords, phi, face velocities, c0, dt, time factor) of one problem, host arrays."""
    from paper_1908_05834_gb300 import inputs
    rng = np.random.Generator(np.random.PCG64(seed))
    # 3D: a little narrower than the recipe's 0.7..1.3, because the mean of a few dozen widths strays from h
    # by several per cent and the cells' aspect ratio should stay the recipe's
    lo, hi = (0.5, 1.5) if dim == 2 else (0.76, 1.24)
    coords = [inputs.uniform_coords(k) if mesh == "uniform" else inputs.stretched_coords(rng, k, lo, hi) for k in n]
    nc = int(np.prod(n))
    h = 1.0 / max(n)
    centre = rng.uniform(0.3, 0.7, dim)
    if dim == 2:
        phi = np.ones(nc)
        faces = inputs.vortex2d_faces(coords)
        c0 = inputs.indicator_ball_average(coords, tuple(centre), 0.15, 4)
        dt = cfl * h
    else:
        phi_min = 0.1 if mesh == "uniform" else 0.05
        phi = inputs.log_uniform_phi(rng, nc, phi_min, 0.3)
        faces = inputs.deform3d_faces(coords)
        c0 = (inputs.indicator_ball_average(coords, tuple(centre), 0.15, 4) if mesh == "uniform"
              else inputs.gaussian_average(coords, tuple(centre), 0.01))
        dt = cfl * h * phi_min / 2.0
    g = math.cos(math.pi * rng.uniform(0.0, 0.35))  # the time factor cos(pi t / T) at some mid-step time
    return coords, phi, faces, c0, dt, g


def _members(case, seed):
    """The problems of a batch or serve case: (dim, n, amplitude factor) from the seed alone."""
    out = []
    rng = np.random.Generator(np.random.PCG64([case["cells"], case["count"]]))
    for i in range(case["count"]):
        dim = 3 if i % 3 == 2 else 2
        cells = case["cells"] * math.exp(-0.7 * rng.uniform())
        k = cells ** (1.0 / dim)
        n = [max(8, int(k * f)) for f in rng.uniform(0.9, 1.0, dim)]
        out.append((dim, n, seed * 1009 + i))
    return out


def _dims(case):
    return [case["n0"], case["n1"], case["n2"]][:case["dim"]]


def _options(case):
    from paper_1908_05834_gb300 import bchar
    kw = {"precision": bchar.FP64 if case["precision"] == "fp64" else bchar.FP32_SPLIT}
    if case["kind"] == "scalings":
        kw["qp_max_refine"] = 0
    return bchar.default_options(**kw)


def _handle(case, dim, n, mesh, seed, stream=None):
    from paper_1908_05834_gb300 import bchar
    coords, phi, faces, c0, dt, g = _problem(dim, n, mesh, case["cfl"], seed)
    m = bchar.Mesh(coords, phi, _options(case), stream=stream)
    dtype = torch.float64 if case["c"] == "f64" else torch.float32
    c = torch.tensor(np.asarray(c0, dtype=np.float64), device="cuda").to(dtype)
    fd = [torch.tensor(f.reshape(-1), device="cuda") for f in faces]
    return {"mesh": m, "faces": fd, "g": g, "dt": dt, "c": c, "out": torch.empty_like(c)}


def prepare(case, seed):
    if case["kind"] in ("step", "scalings"):
        return {"kind": "step", **_handle(case, case["dim"], _dims(case), case["mesh"], seed)}
    if case["kind"] == "batch":
        streams = [torch.cuda.Stream() for _ in range(case["count"])]
        hs = [_handle(case, dim, n, "uniform" if i % 2 else "stretched" if dim == 2 else "uniform", s,
                      streams[i].cuda_stream) for i, (dim, n, s) in enumerate(_members(case, seed))]
        torch.cuda.synchronize()
        return {"kind": "batch", "handles": hs, "streams": streams}
    from paper_1908_05834_gb300 import serve
    reqs, prepared = _requests(case, seed)
    opts = _options(case)
    return {"kind": "serve", "reqs": reqs, "executor": serve.GpuExecutor(prepared, opts),
            "estimator": serve.estimator_for(prepared, opts)}


class _Request:
    """A request in the server's terms (see paper_1908_05834_gb300.inputs.ServeRequest)."""

    def __init__(self, rid, nc, steps, dt, g):
        self.rid, self.arrival_s, self.nc, self.steps, self.dt, self._g = rid, 0.0, nc, steps, dt, g

    def time_factor(self, k):
        return self._g


def _requests(case, seed):
    reqs, prepared = [], {}
    for rid, (dim, n, s) in enumerate(_members(case, seed)):
        coords, phi, faces, c0, dt, g = _problem(dim, n, "uniform", case["cfl"], s)
        prepared[rid] = (coords, phi, faces, np.asarray(c0, dtype=np.float64))
        reqs.append(_Request(rid, int(np.prod(n)), case["steps"], dt, g))
    return reqs, prepared


def run(state):
    if state["kind"] == "step":
        m = state["mesh"]
        m.set_velocity(state["faces"], scale=state["g"])
        info = m.step(state["dt"], state["c"], state["out"])
        return {"c": state["out"], "mass": info["mass_after"], "nnz": info["nnz"]}
    if state["kind"] == "batch":
        from paper_1908_05834_gb300 import bchar
        hs = state["handles"]
        for h in hs:
            h["mesh"].set_velocity(h["faces"], scale=h["g"])
        bchar.step_batch([h["mesh"] for h in hs], [h["dt"] for h in hs], [h["c"] for h in hs], [h["out"] for h in hs])
        return [h["out"] for h in hs]
    from paper_1908_05834_gb300 import serve
    server = serve.Server(state["executor"], state["estimator"], max_active=8)
    return [r.c for r in server.run(state["reqs"])]


def _step_work(dim, n, mesh, c_bytes):
    nc = float(np.prod(n))
    faces = sum(nc / k * (k + 1) for k in n)
    balls = nc * (4 if dim == 2 else 8) * (1.0 if mesh == "uniform" else 1.3)
    entries = nc * (3.5 if dim == 2 else 7.0)
    # c in and out, the face velocities, the mesh's porosity, the matrix written and read once (index and value);
    # one RK4 substep per ball, the intersections of a ball with a cell neighbourhood, 21 products with the matrix
    return {"bytes": nc * (2 * c_bytes + 8) + 8 * faces + 24 * entries,
            "flops": balls * (4 * 12 * dim + 3 ** dim * 40.0) + 42 * entries}


def work(case):
    cb = 8 if case["c"] == "f64" else 4
    if case["kind"] in ("step", "scalings"):
        return _step_work(case["dim"], _dims(case), case["mesh"], cb)
    per = [_step_work(dim, n, "uniform", cb) for dim, n, _ in _members(case, 0)]
    k = case.get("steps", 1)
    return {"bytes": k * sum(w["bytes"] for w in per), "flops": k * sum(w["flops"] for w in per)}


# ---------------------------------------------------------------- the same in 64 bits

_MOST_DENSE = 4200  # cells up to which the minimisation's dense normal equations take a few seconds


def exact(case, seed):
    if case["kind"] in ("step", "scalings"):
        n = _dims(case)
        if case["kind"] == "step" and np.prod(n) > _MOST_DENSE:
            return None
        p = _problem(case["dim"], n, case["mesh"], case["cfl"], seed)
        c = torch.tensor(np.asarray(p[3], dtype=np.float64), device=_dev())
        if case["c"] == "f32":
            c = c.float().double()
        c, mass = _Exact(*p[:3], p[4], p[5]).step(c, case["kind"] == "step")
        return {"c": c, "mass": mass, "nnz": None}
    if case["cells"] > _MOST_DENSE or case["count"] > 4:
        return None
    out = []
    for i, (dim, n, s) in enumerate(_members(case, seed)):
        mesh = "uniform" if case["kind"] == "serve" or i % 2 or dim == 3 else "stretched"
        p = _problem(dim, n, mesh, case["cfl"], s)
        ex = _Exact(*p[:3], p[4], p[5])
        c = torch.tensor(np.asarray(p[3], dtype=np.float64), device=_dev())
        for _ in range(case.get("steps", 1)):
            c, _mass = ex.step(c, True)
        out.append(c)
    return out


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


class _Exact:
    """One step in FP64 (the method of the package's header, default options)."""

    NB, SCALINGS, DROP, EPS, DELTA, CFL = 2, 10, 1e-12, 1e-7, 1e-6, 0.5

    def __init__(self, coords, phi, faces, dt, g):
        d = self.dev = _dev()
        self.dim = len(coords)
        self.x = [torch.tensor(c, dtype=torch.float64, device=d) for c in coords]
        self.w = [x[1:] - x[:-1] for x in self.x]
        self.n = [len(c) - 1 for c in coords]
        self.nc = int(np.prod(self.n))
        self.phi = torch.tensor(phi, dtype=torch.float64, device=d)
        self.u = [torch.tensor(f.reshape(-1) * g, dtype=torch.float64, device=d) for f in faces]
        self.dt = dt
        self.const = bool((self.phi == self.phi[0]).all())
        k = torch.arange(self.nc, device=d)
        self.ijk = self._split(k)
        cw = [self.w[a][self.ijk[a]] for a in range(self.dim)]
        wmin = cw[0]
        vol = cw[0]
        for a in range(1, self.dim):
            wmin = torch.minimum(wmin, cw[a])
            vol = vol * cw[a]
        self.vp = vol * self.phi
        self.r = wmin / (2 * self.NB)
        self.cnt = [torch.clamp(torch.floor(self.NB * c / wmin + 1e-9).long(), min=self.NB) for c in cw]
        self.nk = self.cnt[0] * self.cnt[1] * (self.cnt[2] if self.dim == 3 else 1)
        ball = math.pi * self.r ** 2 if self.dim == 2 else 4.0 / 3.0 * math.pi * self.r ** 3
        self.rho = self.vp / (self.nk * ball)
        self.matrix = None

    def _split(self, k):
        out, rest = [], k
        for a in range(self.dim):
            out.append(rest % self.n[a])
            rest = rest // self.n[a]
        return out

    def _flat(self, c):
        k = c[-1]
        for a in range(self.dim - 2, -1, -1):
            k = c[a] + self.n[a] * k
        return k

    def _flow(self, p, c):
        out = []
        phi = self.phi[self._flat(c)]
        for a in range(self.dim):
            k = None
            for b in range(self.dim - 1, -1, -1):
                k = c[b] if k is None else c[b] + (self.n[b] + (b == a)) * k
            stride = 1
            for b in range(a):
                stride *= self.n[b]
            lo, hi = self.u[a][k], self.u[a][k + stride]
            xi = (p[a] - self.x[a][c[a]]) / self.w[a][c[a]]
            out.append((lo + xi * (hi - lo)) / phi)
        return out

    def _locate(self, p):
        return [torch.clamp(torch.searchsorted(self.x[a], p[a].contiguous(), right=True) - 1, 0, self.n[a] - 1)
                for a in range(self.dim)]

    def _move(self, p, k, h):
        return [torch.clamp(p[a] + h * k[a], float(self.x[a][0]), float(self.x[a][-1])) for a in range(self.dim)]

    def _track(self, p, c, sign):
        vmax = 0.0
        for a in range(self.dim):  # the largest |face velocity| / phi over the cells
            k = None
            for b in range(self.dim - 1, -1, -1):
                k = self.ijk[b] if k is None else self.ijk[b] + (self.n[b] + (b == a)) * k
            stride = int(np.prod(self.n[:a]))
            vmax = max(vmax, float((torch.maximum(self.u[a][k].abs(), self.u[a][k + stride].abs()) / self.phi).max()))
        hmin = min(float(w.min()) for w in self.w)
        s = max(1, math.ceil(self.dt * vmax / (self.CFL * hmin)))
        h = sign * self.dt / s
        for _ in range(s):
            k1 = self._flow(p, c)
            q = self._move(p, k1, h / 2)
            k2 = self._flow(q, self._locate(q))
            q = self._move(p, k2, h / 2)
            k3 = self._flow(q, self._locate(q))
            q = self._move(p, k3, h)
            k4 = self._flow(q, self._locate(q))
            p = self._move(p, [k1[a] + 2 * k2[a] + 2 * k3[a] + k4[a] for a in range(self.dim)], h / 6)
            c = self._locate(p)
        return p, c

    def _lens(self, d, r1, r2):
        t = r1 + r2 - d
        dd = torch.clamp(d, min=1e-300)
        s1, s2 = t * (d + r2 - r1) / (2 * dd), t * (d + r1 - r2) / (2 * dd)
        rmin = torch.minimum(r1, r2)
        if self.dim == 2:
            def seg(r, s):
                ph = 2 * torch.atan2(torch.sqrt(torch.clamp(s * (2 * r - s), min=0.0)), r - s)
                p2 = ph * ph
                small = ph * p2 / 6 * (1 - p2 / 20 * (1 - p2 / 42 * (1 - p2 / 72 * (1 - p2 / 110))))
                return 0.5 * r * r * torch.where(ph < 0.25, small, ph - torch.sin(ph))
            v, full = seg(r1, s1) + seg(r2, s2), math.pi * rmin ** 2
        else:
            v = math.pi / 3 * (s1 * s1 * (3 * r1 - s1) + s2 * s2 * (3 * r2 - s2))
            full = 4.0 / 3.0 * math.pi * rmin ** 3
        return torch.where(d >= r1 + r2, torch.zeros_like(d), torch.where(d <= (r1 - r2).abs(), full, v))

    def _rows(self, lo, hi):
        """Entries (row, column, value) of A^(0) for the cells lo..hi-1."""
        d = self.dev
        cells = torch.arange(lo, hi, device=d)
        K = torch.repeat_interleave(cells, self.nk[lo:hi])
        off = torch.cumsum(self.nk[lo:hi], 0) - self.nk[lo:hi]
        s = torch.arange(K.numel(), device=d) - torch.repeat_interleave(off, self.nk[lo:hi])
        p, c, rest = [], [], s
        for a in range(self.dim):
            ca = self.cnt[a][K]
            sub = rest % ca
            rest = rest // ca
            i = self.ijk[a][K]
            c.append(i)
            p.append(self.x[a][i] + (sub + 0.5) * self.w[a][i] / ca)
        rK = self.r[K]
        if self.const:
            p, c = self._track(p, c, -1.0)
            rh = rK
        else:
            pts = [torch.cat([p[b]] + [p[b] + sg * rK * (a == b) for a in range(self.dim) for sg in (-1.0, 1.0)])
                   for b in range(self.dim)]
            q, cq = self._track(pts, [v.repeat(1 + 2 * self.dim) for v in c], -1.0)
            m = K.numel()
            p, c = [v[:m] for v in q], [v[:m] for v in cq]
            rh = sum(torch.sqrt(sum((q[b][k * m:(k + 1) * m] - p[b]) ** 2 for b in range(self.dim)))
                     for k in range(1, 1 + 2 * self.dim)) / (2 * self.dim)
            del q, cq, pts
        reach = rh + self.r.max()
        first = [torch.clamp(torch.searchsorted(self.x[a], (p[a] - reach).contiguous(), right=True) - 1, 0, self.n[a] - 1)
                 for a in range(self.dim)]
        last = [torch.clamp(torch.searchsorted(self.x[a], (p[a] + reach).contiguous(), right=True) - 1, 0, self.n[a] - 1)
                for a in range(self.dim)]
        width = [int((last[a] - first[a]).max()) + 1 for a in range(self.dim)] + [1] * (3 - self.dim)
        den = torch.zeros_like(rh)
        found = []
        for oz in range(width[2]):
            for oy in range(width[1]):
                for ox in range(width[0]):
                    o = (ox, oy, oz)
                    ok = torch.ones_like(K, dtype=torch.bool)
                    for a in range(self.dim):
                        ok &= first[a] + o[a] <= last[a]
                    b = torch.nonzero(ok).reshape(-1)
                    if not b.numel():
                        continue
                    mc = [first[a][b] + o[a] for a in range(self.dim)]
                    M = self._flat(mc)
                    rM, rb = self.r[M], rh[b]
                    total = torch.zeros_like(rb)
                    cm = [self.cnt[a][M] for a in range(self.dim)]
                    most = [int(v.max()) for v in cm] + [1] * (3 - self.dim)
                    for sz in range(most[2]):
                        for sy in range(most[1]):
                            for sx in range(most[0]):
                                sub = (sx, sy, sz)
                                d2, has = torch.zeros_like(rb), torch.ones_like(M, dtype=torch.bool)
                                for a in range(self.dim):
                                    z = self.x[a][mc[a]] + (sub[a] + 0.5) * self.w[a][mc[a]] / cm[a] - p[a][b]
                                    d2 += z * z
                                    has &= sub[a] < cm[a]
                                total += torch.where(has, self._lens(torch.sqrt(d2), rb, rM), 0.0)
                    total *= self.rho[M]
                    den.index_add_(0, b, total)
                    keep = total > 0
                    found.append((b[keep], M[keep], total[keep]))
        mass = self.vp[K] / self.nk[K]
        b = torch.cat([f[0] for f in found])
        M = torch.cat([f[1] for f in found])
        v = torch.cat([f[2] for f in found]) / den[b] * mass[b]
        void = torch.nonzero(den == 0).reshape(-1)
        row, colm, val = torch.cat([K[b], K[void]]), torch.cat([M, self._flat(c)[void]]), torch.cat([v, mass[void]])
        key, inv = torch.unique(row * self.nc + colm, return_inverse=True)
        val = torch.zeros(key.numel(), dtype=torch.float64, device=d).index_add_(0, inv, val)
        keep = val >= self.DROP * self.vp[key // self.nc]
        return key[keep], val[keep]

    def _initial(self):
        parts = [self._rows(lo, min(self.nc, lo + (1 << 18))) for lo in range(0, self.nc, 1 << 18)]
        key, val = torch.cat([q[0] for q in parts]), torch.cat([q[1] for q in parts])
        have = torch.zeros(self.nc, dtype=torch.bool, device=self.dev)
        have[key % self.nc] = True
        empty = torch.nonzero(~have).reshape(-1)
        if empty.numel():  # a column nobody reaches goes to the cell its centre is carried into
            c = [v[empty] for v in self.ijk]
            p = [self.x[a][c[a]] + 0.5 * self.w[a][c[a]] for a in range(self.dim)]
            _, c = self._track(p, c, 1.0)
            key = torch.cat([key, self._flat(c) * self.nc + empty])
            val = torch.cat([val, self.vp[empty]])
            key, order = torch.sort(key)
            val = val[order]
        return key // self.nc, key % self.nc, val

    def _targets(self, row, col):
        """Row targets, consistent with the columns' on every connected component."""
        n = self.nc
        label = torch.arange(2 * n, device=self.dev)
        a, b = row, col + n
        while True:
            old = label.clone()
            low = torch.minimum(label[a], label[b])
            label.scatter_reduce_(0, label[a], low, "amin")
            label.scatter_reduce_(0, label[b], low, "amin")
            label.scatter_reduce_(0, a, low, "amin")
            label.scatter_reduce_(0, b, low, "amin")
            label = label[label]
            label = label[label]
            if torch.equal(label, old):
                break
        zero = torch.zeros(2 * n, dtype=torch.float64, device=self.dev)
        sr, sc = zero.clone().index_add_(0, label[:n], self.vp), zero.index_add_(0, label[n:], self.vp)
        sr, sc = sr[label[:n]], sc[label[:n]]
        return torch.where((sc - sr).abs() > 1e-11 * sr, self.vp * sc / sr, self.vp)

    def step(self, c, minimise):
        if self.matrix is None:
            row, col, a = self._initial()
            b = self._targets(row, col)

            def sums(i, v):
                return torch.zeros(self.nc, dtype=torch.float64, device=self.dev).index_add_(0, i, v)

            for _ in range(self.SCALINGS):
                a = a * (self.vp / sums(col, a))[col]
                a = a * (b / sums(row, a))[row]
            q = a * self._minimise(row, col, a, b) if minimise else a
            s = sums(col, q)
            dead = s == 0
            q = torch.where(dead[col], a, q)
            q = q * (self.vp / torch.where(dead, sums(col, a), s))[col]
            self.matrix = (row, col, q / self.vp[row])
        row, col, w = self.matrix
        out = torch.zeros(self.nc, dtype=torch.float64, device=self.dev).index_add_(0, row, w * c[col])
        return out, float((self.vp * out).sum())

    def _minimise(self, row, col, a, b):
        """1 + x of the bounded minimisation with the elastic penalty, by an interior point with
        dense solves of the normal equations (rows eliminated)."""
        n, dev = self.nc, self.dev
        gr, gc = a / b[row], a / self.vp[col]
        eps2, gamma = self.EPS ** 2, self.DELTA / self.EPS ** 2
        one = torch.ones(2 * n, dtype=torch.float64, device=dev)
        f = torch.ones_like(a)
        u, zl, zh = f.clone(), 0.1 * gamma * f, 0.1 * gamma * f
        p, q, zp, zq, y = 0.1 * one, 0.1 * one, gamma * one, gamma * one, 0.0 * one

        def G(v):
            return torch.cat([torch.zeros_like(b).index_add_(0, row, gr * v),
                              torch.zeros_like(b).index_add_(0, col, gc * v)])

        def GT(v):
            return gr * v[row] + gc * v[n + col]

        def boundary(pairs):
            return 1.0 / max(1.0, max(float((-dv / v).max()) for v, dv in pairs))

        pairs = 2 * a.numel() + 4 * n
        best = (math.inf, f)
        for _ in range(150):
            rd = f - 1 - GT(y) - zl + zh
            rdp, rdq = gamma - y - zp, gamma + y - zq
            rp = one - G(f) - eps2 * y - p + q
            ru = 2 - f - u
            mu = float(f @ zl + u @ zh + p @ zp + q @ zq) / pairs
            off = max(float(rp.abs().max()), 100 * mu)
            if mu < 1e-9 and off < best[0]:
                best = (off, f.clone())
            if float(rp.abs().max()) <= 1e-12 and mu <= 1e-14:
                break
            D = 1 / (1 + zl / f + zh / u)
            Dp, Dq = p / zp, q / zq
            sh = eps2 + Dp + Dq
            wr, wc, wx = D * gr * gr, D * gc * gc, D * gr * gc
            dr = sh[:n].index_add(0, row, wr)
            W = torch.zeros(n, n, dtype=torch.float64, device=dev)
            W[row, col] = wx
            S = -(W.t() @ (W / dr[:, None]))
            S.diagonal().add_(sh[n:].index_add(0, col, wc))
            L, bad = torch.linalg.cholesky_ex(S)
            if int(bad):
                L, _bad = torch.linalg.cholesky_ex(S + torch.diag(1e-13 * S.diagonal()))

            def normal(v):
                return torch.cat([dr * v[:n] + W @ v[n:], W.t() @ v[:n]]) + \
                    torch.cat([torch.zeros_like(b), (sh[n:].index_add(0, col, wc)) * v[n:]])

            def solve(r):
                v = torch.zeros_like(r)
                for _k in range(3):
                    e = r - normal(v)
                    yc = torch.cholesky_solve((e[n:] - W.t() @ (e[:n] / dr))[:, None], L)[:, 0]
                    v = v + torch.cat([(e[:n] - W @ yc) / dr, yc])
                return v

            def direction(cl, ch, cp, cq):
                t = -rd + cl / f - ch / u + (zh / u) * ru
                sp, sq = -rdp + cp / p, -rdq + cq / q
                dy = solve(rp - G(D * t) - Dp * sp + Dq * sq)
                df = D * (t + GT(dy))
                du = ru - df
                dp, dq = Dp * (sp + dy), Dq * (sq - dy)
                return (df, du, dp, dq, dy, (cl - zl * df) / f, (ch - zh * du) / u, (cp - zp * dp) / p,
                        (cq - zq * dq) / q)

            df, du, dp, dq, dy, dzl, dzh, dzp, dzq = direction(-f * zl, -u * zh, -p * zp, -q * zq)
            ap = boundary([(f, df), (u, du), (p, dp), (q, dq)])
            ad = boundary([(zl, dzl), (zh, dzh), (zp, dzp), (zq, dzq)])
            aff = float((f + ap * df) @ (zl + ad * dzl) + (u + ap * du) @ (zh + ad * dzh)
                        + (p + ap * dp) @ (zp + ad * dzp) + (q + ap * dq) @ (zq + ad * dzq)) / pairs
            sm = max(min(1.0, (aff / mu) ** 3) * mu, 1e-15)
            df, du, dp, dq, dy, dzl, dzh, dzp, dzq = direction(sm - f * zl - df * dzl, sm - u * zh - du * dzh,
                                                                sm - p * zp - dp * dzp, sm - q * zq - dq * dzq)
            ap = 0.99 * boundary([(f, df), (u, du), (p, dp), (q, dq)])
            ad = 0.99 * boundary([(zl, dzl), (zh, dzh), (zp, dzp), (zq, dzq)])
            f, u, p, q = f + ap * df, u + ap * du, p + ap * dp, q + ap * dq
            y, zl, zh, zp, zq = y + ad * dy, zl + ad * dzl, zh + ad * dzh, zp + ad * dzp, zq + ad * dzq
        return best[1].clamp(0.0, 2.0)
