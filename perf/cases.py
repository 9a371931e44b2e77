"""What the performance of this framework is measured on.

Each case is one call, or one short sequence of calls, that a program using
the package makes through its public entry points: chunks of graph-replayed
time steps on one grid (in the sizes, geometries and precision modes of the
configurations and tests), a batch of uneven grids, a monitored run, and a
whole small request from grid creation to the downloaded result.

Every case continues from a saved state, as a production run does: a Mach 1.4
jet that has started to entrain its surroundings (a weak co-flow, an inward
drift at the side boundaries, noise in the shear layer), uploaded in
``prepare``.  ``exact`` evaluates the same steps in 64 bits with plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2003_09926_gb300 import jz
from paper_2003_09926_gb300 import workloads as W

CFL = 0.5

# One stream for all grids: a program steps its grid on one stream, pass after pass.
_stream = None


def _one_stream():
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


# ---- the cases -------------------------------------------------------------------


def listed():
    return [
        # the smallest serving request (1.5e5 points, odd sizes), one 20-step chunk of the request loop
        dict(name="box_p32_69x47x46", kind="chunk", geom="box", ni=69, nj=47, nk=46, prec="p32", model="smag",
             map_amp=0.0, steps=20),
        # configuration 0: the plain FP64 method on the smallest grid
        dict(name="box_p64_48x32x32", kind="chunk", geom="box", ni=48, nj=32, nk=32, prec="p64", model="smag",
             map_amp=0.0, steps=20),
        # the paper's smallest mesh: the cylinder with its centreline treatment, a long thin azimuth
        dict(name="cyl_p32_32x32x361", kind="chunk", geom="cyl", ni=32, nj=32, nk=361, prec="p32", model="smag",
             map_amp=0.0, steps=20),
        # a small request as the serving loop handles it: create, set the state, step, diagnose, download, release
        dict(name="request_p32_96x64x64", kind="request", geom="box", ni=96, nj=64, nk=64, prec="p32", model="smag",
             map_amp=0.0, steps=20),
        # a medium run watched at every step (diagnostics formed by the steps), odd sizes
        dict(name="monitor_p32_181x121x121", kind="monitor", geom="box", ni=181, nj=121, nk=121, prec="p32",
             model="smag", map_amp=0.02, steps=8),
        # configuration 1, the headline: the mapped 9.4-million-point jet
        dict(name="box_p32_256x192x192", kind="chunk", geom="box", ni=256, nj=192, nk=192, prec="p32", model="smag",
             map_amp=0.02, steps=5),
        # the paper's mesh 6, its largest on one of its nodes' cores
        dict(name="cyl_p32_256x128x361", kind="chunk", geom="cyl", ni=256, nj=128, nk=361, prec="p32", model="smag",
             map_amp=0.0, steps=4),
        # a large run (3.2e7 points), the regime of the upper half of the mesh table
        dict(name="box_p32_384x288x288", kind="chunk", geom="box", ni=384, nj=288, nk=288, prec="p32", model="smag",
             map_amp=0.02, steps=2),
        # configuration 3: 64 uneven grids advanced together
        dict(name="batch_p32_64", kind="batch", geom="box", grids=64, grids_seed=3, prec="p32", model="smag",
             map_amp=0.0, steps=2),
        # the FP64 method at a size that fills the chip
        dict(name="box_p64_128x96x96", kind="chunk", geom="box", ni=128, nj=96, nk=96, prec="p64", model="smag",
             map_amp=0.02, steps=2),
        # FP64 state between FP32 steps (long runs whose increments fall below the FP32 spacing)
        dict(name="box_s64_160x128x128", kind="chunk", geom="box", ni=160, nj=128, nk=128, prec="s64", model="smag",
             map_amp=0.02, steps=5),
        # turbulence in a periodic mapped box: Vreman's model, a fixed time step
        dict(name="periodic_p32_128x96x97", kind="chunk", geom="periodic", ni=128, nj=96, nk=97, prec="p32",
             model="vreman", map_amp=0.1, steps=10, dt=2e-4),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["box", "box", "box", "cyl", "cyl", "p64", "s64", "periodic", "batch", "monitor", "request"])
    amp = rng.choice([0.0, 0.02])
    if kind == "batch":
        return dict(kind="batch", geom="box", grids=rng.randint(8, 64), grids_seed=rng.randint(0, 10 ** 6), prec="p32",
                    model="smag", map_amp=0.0, steps=rng.randint(1, 2))
    if kind == "cyl":  # the paper's meshes 1 to 6 and what lies between them, 361 azimuthal points or fewer
        ni, nj = int(_log(rng, 32, 256)), int(_log(rng, 24, 128))
        nk = rng.choice([361, 361, 2 * rng.randint(60, 180) + 1])
        return dict(kind="chunk", geom="cyl", ni=ni, nj=nj, nk=nk, prec="p32", model="smag", map_amp=0.0,
                    steps=max(1, min(20, int(4e7 / (ni * nj * nk)))))
    lo, hi, most = {"box": (1e5, 2e7, 4e7), "p64": (5e4, 1.2e6, 2e6), "s64": (1e5, 4e6, 1.2e7),
                    "periodic": (1e5, 4e6, 1.2e7), "monitor": (1e5, 4e6, 2e7), "request": (1e5, 1e6, 8e6)}[kind]
    # the shape of the serving trace's requests, 1.5 : 1 : 1, varied, odd sizes as they come
    pts = _log(rng, lo, hi)
    nj = max(8, int(round((pts / 1.5) ** (1.0 / 3.0) * rng.uniform(0.85, 1.15))))
    nk = max(8, int(round((pts / 1.5) ** (1.0 / 3.0) * rng.uniform(0.85, 1.15))))
    ni = max(8, int(round(pts / (nj * nk))))
    case = dict(kind=kind if kind in ("monitor", "request") else "chunk", geom="periodic" if kind == "periodic" else "box",
                ni=ni, nj=nj, nk=nk, prec=kind if kind in ("p64", "s64") else "p32", model="smag", map_amp=amp,
                steps=max(1, min(20, int(most / (ni * nj * nk)))))
    if kind == "periodic":
        case.update(model=rng.choice(["smag", "vreman", "euler"]), map_amp=0.1, dt=2e-4)
    return case


_PREC = {"p64": W.P64, "p32": W.P32, "s64": W.P32_S64}


def _grids(case):
    """(grid description, flow parameters) of every grid of a case."""
    prec = _PREC[case["prec"]]
    if case["kind"] == "batch":
        made = W.config3(case["grids"], seed=case["grids_seed"], precision=prec)["cases"]
        return [(c["grid"], c["flow"]) for c in made]
    sizes = (case["ni"], case["nj"], case["nk"])
    if case["geom"] == "cyl":
        return [(W.cyl_grid(*sizes, precision=prec), W.jet_flow())]
    if case["geom"] == "periodic":
        flow = {"smag": W.jet_flow(re=2e3), "vreman": W.jet_flow(re=5e3, sgs=W.SGS_VREMAN),
                "euler": W.jet_flow(re=0.0, cs=0.0)}[case["model"]]
        return [(W.periodic_grid(*sizes, hi=(2.0, 1.5, 1.2), map_amp=case["map_amp"], map_seed=5, precision=prec), flow)]
    return [(W.jet_grid(*sizes, map_amp=case["map_amp"], map_seed=1, precision=prec), W.jet_flow())]


# ---- the saved state that a case continues from -----------------------------------


def _base(d, a, idx):
    """Coordinate (radius, azimuth) along direction a at the indices idx, before the sinusoidal offset."""
    n, lo, hi, c, w, rc = (d["ni"], d["nj"], d["nk"])[a], d["lo"][a], d["hi"][a], d["stretch_c"], d["stretch_w"], d["cluster_r"]
    cyl = d.get("geom", 0) == W.GEOM_CYLINDER

    def g(H, s):
        if not torch.is_tensor(s):
            s = torch.tensor(s, dtype=torch.float64, device=idx.device)
        return s - (c / H) * (torch.tanh((H * s - rc) / w) + torch.tanh((H * s + rc) / w))

    if cyl and a == 2:
        return 2.0 * math.pi * torch.remainder(idx, n - 1) / (n - 1)
    if cyl and a == 1:
        s = idx / (n - 1)
        return hi * s if c == 0.0 else hi * g(hi, s) / g(hi, 1.0)
    if d["bc"][2 * a] == W.BC_PERIODIC:
        return lo + (hi - lo) * idx / n
    if a == 0 or c == 0.0:
        return lo + (hi - lo) * idx / (n - 1)
    H = 0.5 * (hi - lo)
    return 0.5 * (hi + lo) + H * g(H, -1.0 + 2.0 * idx / (n - 1)) / g(H, 1.0)


def _saved_state(d, flow, seed, device):
    """[5][nk][nj][ni] conserved variables in FP64."""
    gen = torch.Generator(device=device).manual_seed(int(seed) * 1000003 + d["ni"] * 7919 + d["nj"] * 104729 + d["nk"])
    f64 = dict(dtype=torch.float64, device=device)
    x, y, z = (_base(d, a, torch.arange(n, **f64)) for a, n in enumerate((d["ni"], d["nj"], d["nk"])))
    x, y, z = x[None, None, :], y[None, :, None], z[:, None, None]
    shape = (d["nk"], d["nj"], d["ni"])

    def noise():
        return 2.0 * torch.rand(shape, generator=gen, **f64) - 1.0

    gamma = flow["gamma"]
    if d["bc"][0] == W.BC_PERIODIC:  # smooth waves plus white noise
        ph = 2.0 * math.pi * torch.rand(5, generator=gen, **f64)
        kx, ky, kz = (2.0 * math.pi / (h - l) for l, h in zip(d["lo"], d["hi"]))
        wave = lambda q, a, b, c: torch.sin(a * kx * x + b * ky * y + c * kz * z + ph[q])  # noqa: E731
        rho = 1.0 + 0.05 * wave(0, 1, 1, 0) + 0.002 * noise()
        u = 0.5 + 0.1 * wave(1, 1, 2, 1) + 0.002 * noise()
        v = 0.1 * wave(2, 2, 1, 1) + 0.002 * noise()
        w = 0.1 * wave(3, 1, 1, 2) + 0.002 * noise()
        p = (1.0 + 0.03 * wave(4, 1, 1, 1) + 0.002 * noise()) / gamma
    else:
        if d.get("geom", 0) == W.GEOM_CYLINDER:
            y, z = y * torch.cos(z), y * torch.sin(z)
        r = torch.sqrt(y * y + z * z)
        near = torch.exp(-(r / 2.0) ** 2)  # the disturbances sit in and around the jet
        jet = 0.5 * flow["mach"] * (1.0 - torch.tanh((r - flow["r0"]) / (2.0 * flow["theta"])))
        u = jet + 0.05 + 0.01 * flow["mach"] * near * noise()
        v = -0.03 * torch.tanh(y) + 0.01 * flow["mach"] * near * noise()
        w = -0.03 * torch.tanh(z) + 0.01 * flow["mach"] * near * noise()
        rho = 1.0 + 0.001 * near * noise()
        p = (1.0 + 0.001 * near * noise()) / gamma
    full = lambda a: a.expand(shape)  # noqa: E731
    rho, u, v, w, p = full(rho), full(u), full(v), full(w), full(p)
    Q = torch.stack([rho, rho * u, rho * v, rho * w, p / (gamma - 1.0) + 0.5 * rho * (u * u + v * v + w * w)])
    if d.get("geom", 0) == W.GEOM_CYLINDER:
        Q[:, -1] = Q[:, 0]  # the last azimuthal plane repeats the first
    return Q


# ---- one pass ------------------------------------------------------------------------


def _state_view(g):
    """The grid's state where it lives in the caller's buffer: field[var][k][j][i], two ghost layers, rows padded to
    32 elements; the three state copies are followed by the metrics (and, in the FP64-state mode, its FP64 copy)."""
    prec = g.desc["precision"]
    size, msize = (8 if prec == W.P64 else 4), (8 if prec in (W.P64, W.P32_M64) else 4)
    _, nk, nj, ni = g.shape
    pitch = (ni + 4 + 31) // 32 * 32
    plane = pitch * (nj + 4)
    npad = plane * (nk + 4)
    up = lambda n: (n + 255) // 256 * 256  # noqa: E731
    tail = 3 * up(5 * npad * size) + up(10 * npad * msize) + (up(5 * npad * 8) if prec == W.P32_S64 else 0)
    at = g.ptr - g.buf.data_ptr() + g.nbytes - tail
    flat = g.buf[at:at + 5 * npad * size].view(torch.float64 if size == 8 else torch.float32)
    return flat.as_strided((5, nk, nj, ni), (npad, plane, pitch, 1), flat.storage_offset() + 2 * plane + 2 * pitch + 2)


def _grid_at(desc, flow, Q):
    g = jz.Grid(desc, stream=_one_stream()).init(flow, 0)
    g.upload(Q)
    return g


def prepare(case, seed):
    grids = _grids(case)
    saved = [_saved_state(d, f, seed + 7 * k, "cuda").cpu().numpy() for k, (d, f) in enumerate(grids)]
    s = dict(case=case)
    if case["kind"] == "request":
        (s["desc"], s["flow"]), = grids
        s["Q"] = saved[0]
        return s
    s["grids"] = [_grid_at(d, f, Q) for (d, f), Q in zip(grids, saved)]
    s["views"] = [_state_view(g) for g in s["grids"]]
    if case["kind"] == "batch":
        s["batch"] = jz.Batch(s["grids"], stream=_one_stream())
    if case["kind"] == "monitor":
        s["grids"][0].set_step_diagnostics(True)
        s["records"] = [jz.PinnedDiag() for _ in range(case["steps"])]
    return s


_NAMES = ("time", "dt", "rho_min", "rho_max", "p_min", "p_max", "mach_max")


def _numbers(records):
    """The columns of a list of diagnostics records; numbers of FP32 grids in FP32."""
    return {**{k: np.asarray([d[k] for d in records], dtype=np.float32) for k in _NAMES + ("sum",)},
            **{k: np.asarray([d[k] for d in records], dtype=np.int64) for k in ("step", "nonfinite")}}


def run(s):
    case = s["case"]
    if case["kind"] == "batch":
        s["batch"].nsteps(case["steps"], cfl=CFL)
        return s["views"]
    if case["kind"] == "request":
        g = _grid_at(s["desc"], s["flow"], s["Q"])
        g.nsteps(case["steps"], cfl=CFL)
        d = g.diagnostics()
        Q = g.download().astype(np.float32)  # the grid's own precision is kept
        g.close()
        return [Q, _numbers([d])]
    g = s["grids"][0]
    if case["kind"] == "monitor":
        for rec in s["records"]:
            g.nsteps(1, cfl=CFL)
            g.step_diagnostics_async(rec)
        last = g.diagnostics()  # waits: every record has been copied
        return [s["views"][0], _numbers([rec.read() for rec in s["records"]] + [last])]
    if "dt" in case:
        g.nsteps(case["steps"], dt=case["dt"])
    else:
        g.nsteps(case["steps"], cfl=CFL)
    return s["views"]


def work(case):
    """Every Runge-Kutta stage reads the state it starts from, the step's first state (the first stage: one state) and
    the ten metric terms, and writes one state; the time step reads the state and the metrics once more; 556
    operations a point and stage (each face flux formed once), 60 for the time step."""
    pts = sum(d["ni"] * d["nj"] * d["nk"] for d, _ in _grids(case))
    state, metrics = {"p64": (40, 80), "p32": (20, 40), "s64": (20, 40)}[case["prec"]]
    wide = 40 if case["prec"] == "s64" else state  # what is kept between steps
    stages = (state + metrics + state) + 4 * (state + wide + metrics + state) + (40 if case["prec"] == "s64" else 0)
    step = stages + (state + metrics if "dt" not in case else 0)
    return {"bytes": float(pts * step * case["steps"]), "flops": float(pts * case["steps"] * (5 * 556 + 60))}


# ---- the same steps in 64 bits, plain torch --------------------------------------------


def _sinusoid(d, seed_words):
    m = [1 + int(seed_words[2 * c] % 3) for c in range(9)]
    th = [2.0 * math.pi * float(seed_words[2 * c + 1] >> 11) / 2.0 ** 53 for c in range(9)]
    return m, th


def _splitmix64(x):
    z = (x + 0x9E3779B97F4A7C15) & (2 ** 64 - 1)
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & (2 ** 64 - 1)
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & (2 ** 64 - 1)
    return z ^ (z >> 31)


class _Reference:
    """One grid: geometry, boundary conditions, fluxes and the five-stage step on whole arrays [k][j][i]."""

    def __init__(self, d, flow, device):
        self.d, self.f = d, flow
        self.n = n = (d["ni"], d["nj"], d["nk"])
        self.cyl = d.get("geom", 0) == W.GEOM_CYLINDER
        self.per = [d["bc"][2 * a] == W.BC_PERIODIC for a in range(3)]
        self.pn = [n[0], n[1], n[2] - 1 if self.cyl else n[2]]
        self.lo = [0 if p else 1 for p in self.per]
        self.hi = [self.pn[a] - 1 if self.per[a] else n[a] - 2 for a in range(3)]
        self.dev = device
        self._metrics()

    def _index(self, a, lo, hi):
        idx = torch.arange(lo, hi + 1, device=self.dev)
        return torch.remainder(idx, self.pn[a]) if self.per[a] else idx.clamp(0, self.n[a] - 1)

    def pad(self, A):
        """Two ghost layers on every face: wrapped, clamped, or from across the centreline."""
        n = self.n
        if self.cyl:
            across = torch.remainder(torch.arange(n[2], device=self.dev) + self.pn[2] // 2, self.pn[2])
            low = A.index_select(-3, across)[..., 1:3, :].flip(-2)
            A = torch.cat([low, A, A[..., -1:, :], A[..., -1:, :]], dim=-2)
        else:
            A = A.index_select(-2, self._index(1, -2, n[1] + 1))
        return A.index_select(-1, self._index(0, -2, n[0] + 1)).index_select(-3, self._index(2, -2, n[2] + 1))

    def _metrics(self):
        d, n = self.d, self.n
        f64 = dict(dtype=torch.float64, device=self.dev)
        idx = [torch.arange(-1, n[a] + 1, **f64) for a in range(3)]
        base = [_base(d, a, idx[a]) for a in range(3)]
        shp = [(1, 1, -1), (1, -1, 1), (-1, 1, 1)]
        if self.cyl:
            r, th = base[1].view(shp[1]), base[2].view(shp[2])
            X = [base[0].view(shp[0]) + 0 * r * th, r * torch.cos(th) + 0 * base[0].view(shp[0]),
                 r * torch.sin(th) + 0 * base[0].view(shp[0])]
        else:
            words = [_splitmix64(d["map_seed"] ^ c) for c in range(18)]
            m, ph = _sinusoid(d, words)
            one = torch.ones(n[2] + 2, n[1] + 2, n[0] + 2, **f64)
            X = []
            for a in range(3):
                x = base[a].view(shp[a]) * one
                if d["map_amp"] != 0.0:
                    h = 0.5 * (_base(d, a, idx[a] + 1) - _base(d, a, idx[a] - 1))
                    off = d["map_amp"] * h.view(shp[a])
                    for e in range(3):
                        P = n[e] if self.per[e] else n[e] - 1
                        off = off * torch.sin(2.0 * math.pi * m[3 * a + e] * idx[e] / P + ph[3 * a + e]).view(shp[e])
                    x = x + off
                X.append(x)
        self.y0, self.z0 = X[1][1:-1, 1:-1, 1], X[2][1:-1, 1:-1, 1]  # of the x- face

        def at(A, o):
            return A[1 + o[2]:1 + o[2] + n[2], 1 + o[1]:1 + o[1] + n[1], 1 + o[0]:1 + o[0] + n[0]]

        E = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
        add = lambda a, b, s: tuple(p + s * q for p, q in zip(a, b))  # noqa: E731
        D = lambda p, b, o: 0.5 * (at(X[p], add(o, E[b], 1)) - at(X[p], add(o, E[b], -1)))  # noqa: E731
        zero = (0, 0, 0)
        S = torch.empty((3, 3) + at(X[0], zero).shape, **f64)
        for k in range(3):
            b, c = (k + 1) % 3, (k + 2) % 3
            for mm in range(3):
                p, q = (mm + 1) % 3, (mm + 2) % 3
                up, dn = E[c], add(zero, E[c], -1)
                t1 = 0.5 * (D(p, b, up) * at(X[q], up) - D(p, b, dn) * at(X[q], dn))
                up, dn = E[b], add(zero, E[b], -1)
                t2 = 0.5 * (D(p, c, up) * at(X[q], up) - D(p, c, dn) * at(X[q], dn))
                S[k, mm] = t1 - t2
        A = [[D(mm, k, zero) for k in range(3)] for mm in range(3)]
        det = (A[0][0] * (A[1][1] * A[2][2] - A[1][2] * A[2][1]) - A[0][1] * (A[1][0] * A[2][2] - A[1][2] * A[2][0])
               + A[0][2] * (A[1][0] * A[2][1] - A[1][1] * A[2][0]))
        if self.cyl:
            det[:, 0] = det[:, 1]  # zero volume on the centreline: the adjacent radial node's
        self.S, self.J = S, 1.0 / det
        self.Sp, self.Jp = self.pad(S)[..., 1:-1, 1:-1, 1:-1], self.pad(self.J)[1:-1, 1:-1, 1:-1]

    # -- boundary nodes: the face latest in the order y-, y+, z-, z+, x+, x- decides
    def boundary(self, Q):
        d, f, n = self.d, self.f, self.n
        gam = f["gamma"]
        gm1 = gam - 1.0
        done = Q.clone()
        for face in (2, 3, 4, 5, 1, 0):
            a, side, kind = face // 2, face % 2, d["bc"][face]
            if kind == W.BC_PERIODIC:
                continue
            ax = -1 - a
            spot = n[a] - 1 if side else 0
            if kind == W.BC_AXIS:
                done[..., 0, :] = Q[:, :self.pn[2], 1, :].mean(dim=1, keepdim=True)
                continue
            if kind == W.BC_INFLOW:
                r = torch.sqrt(self.y0 * self.y0 + self.z0 * self.z0)
                u = 0.5 * f["mach"] * (1.0 - torch.tanh((r - f["r0"]) / (2.0 * f["theta"])))
                done[0, ..., 0], done[1, ..., 0], done[2, ..., 0], done[3, ..., 0] = 1.0, u, 0.0, 0.0
                done[4, ..., 0] = 1.0 / gam / gm1 + 0.5 * u * u
                continue
            q = Q.select(ax, self.hi[a] if side else self.lo[a])
            rest = [e for e in (2, 1, 0) if e != a]  # the remaining dimensions, slowest first
            for dim, e in zip((-2, -1), rest):
                q = q.index_select(dim, torch.arange(n[e], device=self.dev).clamp(self.lo[e], self.hi[e]))
            s = self.S[a].select(ax, spot)
            if self.cyl and a != 1:  # vanishing face metric on the centreline: the adjacent radial node's normal
                s = s.clone()
                jd = 1 + rest.index(1)
                s.select(jd, 0).copy_(s.select(jd, 1))
            nn = (1.0 if side else -1.0) * s / torch.sqrt((s * s).sum(0))
            vel = q[1:4] / q[0]
            p = gm1 * (q[4] - 0.5 * q[0] * (vel * vel).sum(0))
            c = torch.sqrt(gam * p / q[0])
            un = (vel * nn).sum(0)
            Rp, Rm = un + 2.0 * c / gm1, -2.0 / gm1
            ub, cb = 0.5 * (Rp + Rm), 0.25 * gm1 * (Rp - Rm)
            out = ub > 0
            ent = torch.where(out, p / q[0] ** gam, torch.full_like(p, 1.0 / gam))
            tang = torch.where(out, vel - un * nn, torch.zeros_like(vel))
            rb = (cb * cb / (gam * ent)) ** (1.0 / gm1)
            pb = rb * cb * cb / gam
            vb = tang + ub * nn
            b = torch.cat([rb[None], rb * vb, (pb / gm1 + 0.5 * rb * (vb * vb).sum(0))[None]])
            still = torch.zeros_like(q)
            still[0], still[4] = 1.0, 1.0 / gam / gm1
            b = torch.where(un >= c, q, torch.where(un <= -c, still, b))
            done.select(ax, spot).copy_(b)
        if self.cyl:
            done[:, -1] = done[:, 0]
        return done

    def prim(self, Q):
        gam = self.f["gamma"]
        vel = Q[1:4] / Q[0]
        p = (gam - 1.0) * (Q[4] - 0.5 * Q[0] * (vel * vel).sum(0))
        return vel, p, gam * p / Q[0]

    def viscosity(self, T):
        f = self.f
        return (f["mach"] / f["re"] if f["re"] > 0 else 0.0) * T * torch.sqrt(T) * (1.0 + f["s1"]) / (T + f["s1"])

    def time_step(self, Q, cfl):
        f = self.f
        vel, p, T = self.prim(Q)
        s2 = (self.S * self.S).sum(1)
        rate = 0.0
        for k in range(3):
            rate = rate + self.J * (((self.S[k] * vel).sum(0)).abs() + torch.sqrt(T) * torch.sqrt(s2[k]))
        nu = max(4.0 / 3.0, f["gamma"] / f["pr"]) * self.viscosity(T) / Q[0]
        return cfl / float((rate + 2.0 * nu * self.J * self.J * s2.sum(0)).max())

    def residual(self, Q):
        f, n = self.f, self.n
        gam = f["gamma"]
        P = self.pad(Q)
        vel, p, T = self.prim(P)
        V = torch.cat([vel, T[None]])
        mid = (slice(1, -1),) * 3
        S, J = self.Sp, self.Jp

        def step(A, a, o):  # A on the padded box, shifted by o along direction a, on the box with one layer less
            s = [slice(1, -1)] * 3
            s[2 - a] = slice(1 + o, A.shape[-1 - a] - 1 + o)
            return A[(Ellipsis,) + tuple(s)]

        v0, p0, T0, q0 = vel[(slice(None),) + mid], p[mid], T[mid], P[(slice(None),) + mid]
        Fv = None
        if f["re"] > 0 or f["cs"] > 0:
            diff = [0.5 * J * (step(V, a, 1) - step(V, a, -1)) for a in range(3)]
            g = [[S[0, m] * diff[0][q] + S[1, m] * diff[1][q] + S[2, m] * diff[2][q] for m in range(3)] for q in range(4)]
            del diff
            mu = self.viscosity(T0)
            mut = torch.zeros_like(mu)
            delta2 = J ** (-2.0 / 3.0)
            if f["cs"] > 0 and f.get("sgs", 0) == W.SGS_VREMAN:
                b = [[sum(g[x][m] * g[y][m] for m in range(3)) for y in range(3)] for x in range(3)]
                aa = b[0][0] + b[1][1] + b[2][2]
                B = (b[0][0] * b[1][1] - b[0][1] ** 2 + b[0][0] * b[2][2] - b[0][2] ** 2 + b[1][1] * b[2][2] - b[1][2] ** 2)
                ratio = torch.where(aa > 0, B.clamp(min=0.0) / torch.where(aa > 0, aa, torch.ones_like(aa)), torch.zeros_like(aa))
                mut = q0[0] * 2.5 * f["cs"] ** 2 * delta2 * torch.sqrt(ratio)
            elif f["cs"] > 0:
                s12, s13, s23 = (0.5 * (g[x][y] + g[y][x]) for x, y in ((0, 1), (0, 2), (1, 2)))
                ss = g[0][0] ** 2 + g[1][1] ** 2 + g[2][2] ** 2 + 2.0 * (s12 ** 2 + s13 ** 2 + s23 ** 2)
                mut = q0[0] * f["cs"] ** 2 * delta2 * torch.sqrt(2.0 * ss)
            mue, kap = mu + mut, (mu / f["pr"] + mut / f["prt"]) / (gam - 1.0)
            div = g[0][0] + g[1][1] + g[2][2]
            Fv = [[mue * (g[q][m] + g[m][q] - (2.0 / 3.0 * div if q == m else 0.0)) for q in range(3)] for m in range(3)]
            for m in range(3):
                Fv[m].append(v0[0] * Fv[m][0] + v0[1] * Fv[m][1] + v0[2] * Fv[m][2] + kap * g[3][m])
            del g
        U = [(S[k] * v0).sum(0) for k in range(3)]
        lam = [U[k].abs() + torch.sqrt(T0) * torch.sqrt((S[k] * S[k]).sum(0)) for k in range(3)]
        R = torch.zeros_like(Q)
        for k in range(3):
            G = q0 * U[k]
            for m in range(3):
                G[1 + m] += S[k, m] * p0
            G[4] += p0 * U[k]
            if Fv is not None:
                for c in range(4):
                    G[1 + c] -= S[k, 0] * Fv[0][c] + S[k, 1] * Fv[1][c] + S[k, 2] * Fv[2][c]
            a, b = lam[(k + 1) % 3], lam[(k + 2) % 3]
            pos = lam[k] > 0
            safe = torch.where(pos, lam[k], torch.ones_like(lam[k]))
            lt = torch.where(pos, lam[k] * (1.0 + (a / safe) ** f["sigma"] + (b / safe) ** f["sigma"]), torch.zeros_like(safe))
            pp, pm = step(p, k, 1), step(p, k, -1)
            nu = (pp - 2.0 * p0 + pm).abs() / (pp + 2.0 * p0 + pm)
            ax = -1 - k

            def line(A, lead, first, count):  # `count` nodes along k from `first`, own nodes across; `lead` ghost layers
                for e in range(3):
                    A = A.narrow(-1 - e, first + lead if e == k else lead, count if e == k else n[e])
                return A

            N = n[k] + 1  # faces -1/2 .. n-1/2
            Ga, Gb = line(G, 1, -1, N), line(G, 1, 0, N)
            l = 0.5 * (line(lt, 1, -1, N) + line(lt, 1, 0, N))
            e2 = f["k2"] * torch.maximum(line(nu, 1, -1, N), line(nu, 1, 0, N))
            e4 = (f["k4"] - e2).clamp(min=0.0)
            qm, qa, qb, qp = (line(P, 2, o, N) for o in (-2, -1, 0, 1))
            h = 0.5 * (Ga + Gb) - l * (e2 * (qb - qa) - e4 * (qp - 3.0 * qb + 3.0 * qa - qm))
            R += h.narrow(ax, 1, n[k]) - h.narrow(ax, 0, n[k])
        return R

    def advance(self, Q, cfl=None, dt=None):
        if dt is None:
            dt = self.time_step(Q, cfl)
        inner = (slice(None),) + tuple(slice(self.lo[a], self.hi[a] + 1) for a in (2, 1, 0))
        Ql = Q
        for alpha in (0.25, 1.0 / 6.0, 0.375, 0.5, 1.0):
            new = Q.clone()
            new[inner] = (Q - alpha * dt * self.J * self.residual(Ql))[inner]
            Ql = self.boundary(new)
        return Ql, dt

    def diagnose(self, Q, time, dt):
        vel, p, T = self.prim(Q)
        return {"time": time, "dt": dt, "rho_min": float(Q[0].min()), "rho_max": float(Q[0].max()), "p_min": float(p.min()),
                "p_max": float(p.max()), "mach_max": float(torch.sqrt((vel * vel).sum(0) / T).max()),
                "sum": [float(x) for x in (Q / self.J).flatten(1).sum(1)]}


def exact(case, seed):
    device = "cuda" if torch.cuda.is_available() else "cpu"
    out = []
    for k, (d, f) in enumerate(_grids(case)):
        ref = _Reference(d, f, device)
        Q = ref.boundary(_saved_state(d, f, seed + 7 * k, device))
        time, dt, log = 0.0, 0.0, []
        for _ in range(case["steps"]):
            if case["kind"] == "monitor":
                log.append(ref.diagnose(Q, time, dt))
            Q, dt = ref.advance(Q, None if "dt" in case else CFL, case.get("dt"))
            time += dt
        log.append(ref.diagnose(Q, time, dt))
        out.append(Q)
        del ref
    if case["kind"] in ("request", "monitor"):
        columns = {k: np.asarray([r[k] for r in log]) for k in _NAMES + ("sum",)}
        return [out[0], {**columns, "step": None, "nonfinite": None}]
    return out
