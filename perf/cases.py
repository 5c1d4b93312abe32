"""What a user of this solver has it do, as measurable cases.

Each case is a dict of plain values; `prepare` builds what a program has in
hand before the call (grid, bodies, context, start fields), `run` is one pass
through the public entry points, `exact` the same outputs from plain torch in
64 bits (its own classification, ghost rows and linear solves; none of the
library's code).

Kinds of pass:
  step      restart from a saved state and advance `steps` fractional steps:
            the way every simulation spends its time. A pass starts from the
            impulsive state with a bump in the wake, an empty guess history
            and step 0, so that every pass does the same work.
  poisson   one pressure solve from a zero guess to the default 1e-10.
  move      the body pitches up and back: move, step, move, step.
  ensemble  several 2D cases resident on their own streams, their captured
            steps enqueued together and waited for.
  serve     requests through the server: grid, bodies, classification, steps
            and results back on the host, several at a time.
"""
import math
import os

# a process-wide setting of programs that run many cases at once: their
# streams map to separate hardware queues (read when CUDA starts)
os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")

import numpy as np
import torch

from paper_2505_17287_gb300 import ibm, synth

F64 = torch.float64
BC = (0, 1, 2, 2, 2, 2)   # inflow, outflow, free-slip sides


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest 2D study: latency of one host-driven step
        dict(name="step_2d_small", kind="step", body="ellipse", nx=128, ny=64, nz=1, prec="fp64", graph=1, steps=4),
        # the 2D cylinder workload, each step one captured graph
        dict(name="step_2d_cylinder", kind="step", body="ellipse", nx=256, ny=128, nz=1, prec="mixed", graph=2, steps=4),
        # a 2D grid at the top of the ensemble's range
        dict(name="step_2d_large", kind="step", body="ellipse", nx=1024, ny=512, nz=1, prec="mixed", graph=1, steps=2),
        # a ragged 3D grid (no extent divides by 4) in full FP64
        dict(name="step_3d_odd", kind="step", body="spheres", nx=129, ny=85, nz=77, prec="fp64", graph=1, steps=2),
        # an ordinary 3D request: uniform box with a few spheres
        dict(name="step_3d_spheres", kind="step", body="spheres", nx=160, ny=160, nz=160, prec="mixed", graph=1, steps=2),
        # the wing in full FP64
        dict(name="step_wing_fp64", kind="step", body="wing", nx=192, ny=128, nz=128, prec="fp64", graph=1, steps=2),
        # the wing on its reference grid, mixed precision
        dict(name="step_wing_mixed", kind="step", body="wing", nx=384, ny=256, nz=256, prec="mixed", graph=1, steps=2),
        # the largest of which three fit the card beside each other
        dict(name="step_wing_large", kind="step", body="wing", nx=512, ny=384, nz=320, prec="mixed", graph=1, steps=1),
        # a pressure solve on its own, odd 2D extents
        dict(name="poisson_2d_odd", kind="poisson", body="ellipse", nx=601, ny=301, nz=1, prec="mixed", graph=1, steps=0),
        # a body in motion: reclassified, tables and multigrid rebuilt every step
        dict(name="move_wing", kind="move", body="wing", nx=192, ny=128, nz=128, prec="mixed", graph=1, steps=2),
        # a parameter study: uneven 2D cases at once
        dict(name="ensemble_2d", kind="ensemble", body="ellipse", nx=512, ny=256, nz=1, prec="mixed", graph=2, steps=4,
             count=12),
        # the request loop, from inputs on the host to results on the host
        dict(name="serve_spheres", kind="serve", body="spheres", nx=96, ny=96, nz=96, prec="mixed", graph=1, steps=2,
             count=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "step", "poisson", "poisson", "move", "ensemble", "serve"])
    prec = rng.choice(["mixed", "mixed", "fp64"])
    graph = rng.choice([1, 1, 2])
    c = dict(kind=kind, prec=prec, graph=graph, steps=rng.choice([2, 4]) if graph == 2 else rng.choice([1, 2, 3]))
    if kind in ("ensemble", "serve"):
        if kind == "ensemble":
            nx = _log(rng, 160, 640)
            c.update(body="ellipse", nx=nx, ny=nx // 2, nz=1, graph=2, steps=rng.choice([2, 4]), count=rng.randint(4, 16))
        else:
            n = _log(rng, 48, 112)
            c.update(body="spheres", nx=n, ny=n, nz=n, graph=1, steps=rng.choice([1, 2]), count=rng.randint(2, 5))
        return c
    body = "wing" if kind == "move" else rng.choice(["ellipse", "spheres", "wing"])
    if body == "ellipse":
        nx = _log(rng, 110, 1300)
        c.update(body=body, nx=nx, ny=max(50, int(nx * rng.uniform(0.4, 0.6))), nz=1)
    elif body == "spheres":
        nx = _log(rng, 72, 260)
        c.update(body=body, nx=nx, ny=max(56, int(nx * rng.uniform(0.7, 1.1))), nz=max(56, int(nx * rng.uniform(0.7, 1.1))))
    else:
        nx = _log(rng, 120, 240 if kind == "move" else 440)
        c.update(body=body, nx=nx, ny=int(nx * rng.uniform(0.6, 0.75)), nz=int(nx * rng.uniform(0.6, 0.75)))
    if rng.random() < 0.5:   # half of them in whole multiples, as users pick sizes
        for k in ("nx", "ny", "nz"):
            c[k] = max(1, c[k] // 8 * 8) if c[k] > 1 else 1
    if kind == "poisson":
        c["steps"] = 0
    if kind == "move":
        c["steps"], c["graph"] = 2, 1
    return c


def _parts(case):
    """The single cases that a pass works on: uneven sizes for an ensemble or a request stream."""
    n = case.get("count", 1)
    out = []
    for q in range(n):
        c = dict(case)
        if n > 1:   # from 60% to 100% of the named size
            f = 1.0 - 0.4 * q / max(1, n - 1)
            for k in ("nx", "ny", "nz"):
                c[k] = max(32, int(case[k] * f) // 8 * 8 + (q % 3 == 2)) if case[k] > 1 else 1
        out.append(c)
    return out


def _problem(case, seed):
    """Grid, bodies and flow parameters of a single case: a synth.Case."""
    r = np.random.default_rng([int(seed) & 0x7FFFFFFF, case["nx"], case["ny"], case["nz"]])
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if case["body"] == "ellipse":
        a = r.uniform(0.4, 0.9)
        v, e = synth.ellipse_polyline(a, a * r.uniform(0.6, 1.0), r.uniform(0.1, 3.0), 256, r.uniform(-0.3, 0.3),
                                      r.uniform(-0.3, 0.3))
        xf, yf, zf = synth.uniform_faces(-8.0, 24.0, nx), synth.uniform_faces(-8.0, 8.0, ny), np.array([0.0, 1.0])
        bodies, Re, dt = [(v, e)], r.uniform(60.0, 200.0), 0.2 * min(32.0 / nx, 16.0 / ny)
    elif case["body"] == "spheres":
        spheres = [(r.uniform(0.45, 0.6), (x + r.uniform(-0.2, 0.2), y + r.uniform(-0.2, 0.2), r.uniform(-0.8, 0.8)))
                   for x, y in ((-0.5, -1.0), (1.5, 0.9), (3.6, -0.6))]
        bodies = [synth.icosphere(3, rad, c) for rad, c in spheres]
        xf, yf, zf = synth.uniform_faces(-4.0, 8.0, nx), synth.uniform_faces(-3.0, 3.0, ny), synth.uniform_faces(-3.0, 3.0, nz)
        Re, dt = r.uniform(100.0, 500.0), 0.2 * min(12.0 / nx, 6.0 / ny, 6.0 / nz)
    else:
        base = synth.wing_case(nx, ny, nz)
        v, e = synth.naca_wing(100, 50, 2.0, r.uniform(12.0, 18.0))
        xf, yf, zf, bodies, Re, dt = base.xf, base.yf, base.zf, [(v, e)], 1000.0, 0.002 * min(1.0, 384.0 / nx)
    return synth.Case("case", 2 if nz == 1 else 3, xf, yf, zf, bodies[0][0], bodies[0][1], float(Re), float(dt),
                      case["steps"], meta={"bodies": bodies})


def _centres(f, dev):
    f = torch.as_tensor(f, dtype=F64, device=dev)
    return 0.5 * (f[1:] + f[:-1])


def _bump(p, seed, dev):
    """A smooth bump in the wake per velocity component (sums of separable
    Gaussians): breaks the symmetry of the impulsive start."""
    r = np.random.default_rng([int(seed) & 0x7FFFFFFF, 17])
    x, y, z = (_centres(f, dev) for f in (p.xf, p.yf, p.zf))
    out = []
    for _ in range(p.ndim):
        t = 0.0
        for _ in range(3):
            c = (r.uniform(0.8, 3.0), r.uniform(-0.8, 0.8), r.uniform(-0.8, 0.8) if p.ndim == 3 else 0.5)
            w = r.uniform(0.2, 0.6)
            gx, gy, gz = (torch.exp(-((q - q0) ** 2) / w) for q, q0 in zip((x, y, z), c))
            t = t + r.uniform(-0.2, 0.2) * gz[:, None, None] * gy[None, :, None] * gx[None, None, :]
        out.append(t)
    return out


def _rhs(p, seed, dev):
    """A pressure right-hand side: waves over the box and noise near the body."""
    r = np.random.default_rng([int(seed) & 0x7FFFFFFF, 23])
    x, y, z = (_centres(f, dev) for f in (p.xf, p.yf, p.zf))
    t = 0.0
    for _ in range(4):
        k = r.uniform(0.2, 2.0, 3)
        f = r.uniform(0.0, 6.28, 3)
        gx, gy, gz = (torch.cos(a * q + b) for a, q, b in zip(k, (x, y, z), f))
        t = t + gz[:, None, None] * gy[None, :, None] * gx[None, None, :]
    g = torch.Generator(device=dev).manual_seed(int(seed) & 0x7FFFFFFF)
    noise = torch.rand(t.shape, dtype=F64, device=dev, generator=g) * 2.0 - 1.0
    near = (torch.exp(-z ** 2) if p.ndim == 3 else torch.ones_like(z))[:, None, None] * torch.exp(-y ** 2)[None, :, None] \
        * torch.exp(-x ** 2)[None, None, :]
    return t + 20.0 * noise * near


def _pitch(p, degrees):
    """The wing's vertices pitched about the span axis through the quarter chord."""
    v = np.array(p.verts)
    a = math.radians(degrees)
    x, y = v[:, 0] - 0.25, v[:, 1].copy()
    v[:, 0], v[:, 1] = 0.25 + math.cos(a) * x + math.sin(a) * y, -math.sin(a) * x + math.cos(a) * y
    return v


PITCH = 0.25   # degrees between the two positions of a moving wing


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------

def _velocities(p):
    return ["u", "v", "w"][:p.ndim]


def _get(s, name, out):
    ibm.ibm_get_field(s.ctx, ibm.FIELDS[name], out.data_ptr(), 1, out.numel() * 8)
    return out


def _set(s, name, src):
    ibm.ibm_set_field(s.ctx, ibm.FIELDS[name], src.data_ptr(), 1, src.numel() * 8)


def _solver(case, p):
    prec = ibm.IBM_MIXED if case["prec"] == "mixed" else ibm.IBM_FP64
    s = ibm.Solver(p, precision=prec, bc=BC, stream=torch.cuda.Stream())
    s.set_opts(precision=prec, graph=case["graph"])
    for v, e in synth.case_bodies(p):
        s.set_body(v, e)
    s.classify()
    return s


def _start(case, p, seed):
    """A classified context, its start fields on the device and room for its results."""
    s = _solver(case, p)
    start = {}
    with torch.cuda.stream(s.stream):   # the tensors belong to the stream that the library copies on
        fluid = torch.as_tensor(s.get("type"), device="cuda") == ibm.IBM_FLUID
        for n, d in zip(_velocities(p), _bump(p, seed, "cuda")):
            t = _get(s, n, torch.empty(s.shape, dtype=F64, device="cuda"))
            start[n] = t + torch.where(fluid, d, 0.0)
        for n in _velocities(p):
            start["face_" + n] = _get(s, "face_" + n, torch.empty(s.field_size("face_" + n), dtype=F64, device="cuda"))
        start["p"] = torch.zeros(s.shape, dtype=F64, device="cuda")
        outs = {n: torch.empty(s.shape, dtype=F64, device="cuda") for n in _velocities(p) + ["p"]}
    torch.cuda.synchronize()
    return dict(s=s, start=start, outs=outs, steps=case["steps"])


def _restart(one):
    """Back to the saved start: the fields, step 0 and an empty guess history."""
    s = one["s"]
    for n, t in one["start"].items():
        _set(s, n, t)
    s.set("step", 0)
    ctl = np.zeros(s.field_size("p_hist_ctl"))
    ibm.ibm_set_field(s.ctx, ibm.FIELDS["p_hist_ctl"], ctl.ctypes.data, 0, ctl.nbytes)


def _results(one):
    return {n: _get(one["s"], n, t) for n, t in one["outs"].items()}


def _checked(r):
    if r["status"] != ibm.IBM_OK:
        raise RuntimeError("the solver did not converge: %r" % (r,))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "serve":
        return dict(kind=kind, case=case, srv=ibm.Server(max_slots=4),
                    parts=[_problem(c, seed + 31 * q) for q, c in enumerate(_parts(case))])
    if kind == "ensemble":
        all_ = [_start(c, _problem(c, seed + 31 * q), seed + 31 * q) for q, c in enumerate(_parts(case))]
        for one in all_:
            one["s"].step_prepare()
        torch.cuda.synchronize()
        return dict(kind=kind, all=all_)
    p = _problem(case, seed)
    if kind == "poisson":
        s = _solver(case, p)
        rhs = _rhs(p, seed, "cuda").contiguous()
        torch.cuda.synchronize()
        return dict(kind=kind, s=s, rhs=rhs)
    one = _start(case, p, seed)
    one["kind"] = kind
    if kind == "move":
        one["up"], one["back"], one["dt"] = _pitch(p, PITCH), np.array(p.verts), p.dt
    elif case["graph"] == 2:
        one["s"].step_prepare()
        torch.cuda.synchronize()
    return one


def run(st):
    kind = st["kind"]
    if kind == "serve":
        c, srv = st["case"], st["srv"]
        prec = ibm.IBM_MIXED if c["prec"] == "mixed" else ibm.IBM_FP64
        ids = [srv.submit(p, nsteps=c["steps"], precision=prec, outputs=True, bc=BC) for p in st["parts"]]
        res = [srv.wait(i) for i in ids]
        for r in res:
            _checked(r)
        return [r["outputs"] for r in res]
    if kind == "ensemble":
        for one in st["all"]:
            _restart(one)
        for one in st["all"]:
            one["s"].step_async(one["steps"])
        for one in st["all"]:
            _checked(one["s"].step_wait())
        return [_results(one) for one in st["all"]]
    s = st["s"]
    if kind == "poisson":
        with torch.cuda.stream(s.stream):
            phi = torch.zeros(s.shape, dtype=F64, device="cuda")
            _checked(s.poisson_solve(st["rhs"], phi))
        return phi
    _restart(st)
    if kind == "move":
        w = math.radians(PITCH) / st["dt"]
        for verts, sign in ((st["up"], -1.0), (st["back"], 1.0)):
            s.move_body(verts, omega=(0.0, 0.0, sign * w), centre=(0.25, 0.0, 0.0))
            _checked(s.step(1))
    else:
        _checked(s.step(st["steps"]))
    return _results(st)


def work(case):
    """State in and out once a step (velocities, face velocities, convective
    term, pressure); operations: a few hundred a cell for the operators of a
    step and its two linear solves at the least."""
    by = fl = 0.0
    for c in _parts(case):
        n = float(c["nx"]) * c["ny"] * c["nz"]
        d = 2 if c["nz"] == 1 else 3
        if case["kind"] == "poisson":
            by, fl = by + 16.0 * n, fl + 100.0 * n
        else:
            by, fl = by + case["steps"] * n * 16.0 * (3 * d + 1), fl + case["steps"] * n * 100.0 * (d + 1)
    return {"bytes": by, "flops": fl}


def tolerance(case):
    # Both linear solves stop at a relative residual (pressure 1e-10, velocity
    # 1e-12), so a correct run is off by that times the conditioning of its
    # operators. Measured against `exact` over 90 cases of these ranges: up to
    # 7e-8 in 2D (the pressure) and 6e-9 in 3D; single cells next to a wing up
    # to 2.4e-6 of their component's root mean square, 2D ones 1e-7.
    if case["nz"] == 1:
        return {"rel": 3e-7, "max": 2e-6}
    return {"rel": 2.5e-8, "max": 1e-5}


# ---------------------------------------------------------------------------
# the same in plain torch, 64 bits
# ---------------------------------------------------------------------------

FLUID, GHOST, DEAD = 0, 1, 2


def _sl(a, lo, hi):
    s = [slice(None)] * 3
    s[2 - a] = slice(lo, hi)
    return tuple(s)


class _Flow:
    """The discrete flow problem on a device: the grid, then per body position
    the cell types and ghost rows."""

    def __init__(self, p, dev):
        self.p, self.dev, self.nd = p, dev, p.ndim
        f = [p.xf, p.yf, p.zf if p.ndim == 3 else np.array([0.0, 1.0])]
        self.f = [torch.as_tensor(np.asarray(a), dtype=F64, device=dev) for a in f]
        self.h = [a[1:] - a[:-1] for a in self.f]
        self.c = [0.5 * (a[1:] + a[:-1]) for a in self.f]
        self.hc = [a[1:] - a[:-1] for a in self.c]
        self.n = [len(a) for a in self.h]
        self.shape = (self.n[2], self.n[1], self.n[0])
        self.N = self.n[0] * self.n[1] * self.n[2]
        self.vol = self.h[2][:, None, None] * self.h[1][None, :, None] * self.h[0][None, None, :]
        self.eig = None

    def bc1(self, t, a):
        return t.reshape([(1, 1, -1), (1, -1, 1), (-1, 1, 1)][a])

    # geometry ---------------------------------------------------------------

    def classify(self, bodies):
        off, V, E = 0, [], []
        for v, e in bodies:
            V.append(v)
            E.append(e.astype(np.int64) + off)
            off += len(v)
        V = torch.as_tensor(np.concatenate(V), dtype=F64, device=self.dev)
        self.el = V[torch.as_tensor(np.concatenate(E), device=self.dev)][..., :self.nd]   # (ne, nd vertices, nd)
        ins = self._inside()
        near = torch.zeros_like(ins)
        for a in range(self.nd):
            near[_sl(a, 0, -1)] |= ~ins[_sl(a, 1, None)]
            near[_sl(a, 1, None)] |= ~ins[_sl(a, 0, -1)]
        self.type = torch.where(ins, torch.where(near, GHOST, DEAD), FLUID)
        self.fl, self.dead = self.type == FLUID, self.type == DEAD
        self.vf = torch.where(self.fl, self.vol, 0.0)
        self.vsum = self.vf.sum()
        self.gi = (self.type == GHOST).flatten().nonzero()[:, 0]
        self._ghost_rows()
        self.ubi = torch.zeros(len(self.gi), 3, dtype=F64, device=self.dev)

    def _inside(self):
        """Parity of the surface crossings above each centre along the last axis."""
        a = self.nd - 1   # the ray's axis
        el = self.el
        lo, hi = el.amin((0, 1)), el.amax((0, 1))
        cx = self.c[0]
        cy = self.c[1] if self.nd == 3 else torch.zeros(1, dtype=F64, device=self.dev)
        ix = ((cx >= lo[0]) & (cx <= hi[0])).nonzero()[:, 0]
        iy = ((cy >= lo[1]) & (cy <= hi[1])).nonzero()[:, 0] if self.nd == 3 else torch.zeros(1, dtype=torch.int64, device=self.dev)
        X, Y = cx[ix].repeat(len(iy)), cy[iy].repeat_interleave(len(ix))
        col = ix.repeat(len(iy)) + self.n[0] * iy.repeat_interleave(len(ix))
        marks = torch.zeros((self.n[a] + 1) * self.n[0] * (self.n[1] if self.nd == 3 else 1), dtype=torch.int32, device=self.dev)
        ncol = marks.numel() // (self.n[a] + 1)
        step = max(1, int(4e7 // len(el)))
        for s in range(0, len(X), step):
            x, y = X[s:s + step, None], Y[s:s + step, None]
            if self.nd == 2:
                A, B = el[None, :, 0], el[None, :, 1]
                hit = (A[..., 0] > x) != (B[..., 0] > x)
                q, t = hit.nonzero(as_tuple=True)
                A, B, x = el[t, 0], el[t, 1], x[q, 0]
                top = A[:, 1] + (x - A[:, 0]) / (B[:, 0] - A[:, 0]) * (B[:, 1] - A[:, 1])
            else:
                P = el[None]
                w = []
                for m in range(3):
                    A, B = P[:, :, m], P[:, :, (m + 1) % 3]
                    w.append((B[..., 0] - A[..., 0]) * (y - A[..., 1]) - (B[..., 1] - A[..., 1]) * (x - A[..., 0]))
                hit = ((w[0] > 0) & (w[1] > 0) & (w[2] > 0)) | ((w[0] < 0) & (w[1] < 0) & (w[2] < 0))
                q, t = hit.nonzero(as_tuple=True)
                w = [k[q, t] for k in w]
                z = el[t, :, 2]
                top = (w[1] * z[:, 0] + w[2] * z[:, 1] + w[0] * z[:, 2]) / (w[0] + w[1] + w[2])
            marks.index_add_(0, torch.searchsorted(self.c[a], top) * ncol + col[s:s + step][q], torch.ones_like(q, dtype=torch.int32))
        above = marks.reshape(self.n[a] + 1, ncol).flip(0).cumsum(0).flip(0)[1:]   # crossings above centre k
        return ((above & 1) == 1).reshape(self.shape)

    def _closest(self, P):
        """The closest surface point to each point of P (lowest element on ties)."""
        el, out = self.el, torch.empty_like(P)

        def seg(p, A, B):
            d = B - A
            t = (((p - A) * d).sum(-1) / (d * d).sum(-1)).clamp(0.0, 1.0)
            return A + t[..., None] * d

        step = max(1, int((4e6 if self.nd == 3 else 2e7) // len(el)))
        for s in range(0, len(P), step):
            p = P[s:s + step, None]
            if self.nd == 2:
                q = seg(p, el[None, :, 0], el[None, :, 1])
            else:
                A, B, C = el[None, :, 0], el[None, :, 1], el[None, :, 2]
                n = torch.linalg.cross(B - A, C - A)
                proj = p - ((p - A) * n).sum(-1, keepdim=True) / (n * n).sum(-1, keepdim=True) * n
                ok = torch.ones(p.shape[0], len(el), dtype=torch.bool, device=self.dev)
                for U, W in ((A, B), (B, C), (C, A)):
                    ok &= (torch.linalg.cross((W - U).expand_as(proj), proj - U) * n).sum(-1) >= 0
                q, best = seg(p, A, B), None
                best = ((q - p) ** 2).sum(-1)
                for U, W in ((B, C), (C, A)):
                    r = seg(p, U, W)
                    d = ((r - p) ** 2).sum(-1)
                    q, best = torch.where((d < best)[..., None], r, q), torch.minimum(d, best)
                q = torch.where(ok[..., None], proj, q)
            k = ((q - p) ** 2).sum(-1).argmin(1)
            out[s:s + step] = q[torch.arange(len(k), device=self.dev), k]
        return out

    def _ijk(self, idx):
        return [idx % self.n[0], idx // self.n[0] % self.n[1], idx // (self.n[0] * self.n[1])][:self.nd]

    def _basis(self, x):
        one = torch.ones_like(x[0])
        if self.nd == 2:
            return torch.stack([one, x[0], x[1], x[0] * x[1]], -1)
        return torch.stack([one, x[0], x[1], x[2], x[0] * x[1], x[1] * x[2], x[2] * x[0], x[0] * x[1] * x[2]], -1)

    def _corners(self, base):
        nc = 2 ** self.nd
        d = [torch.tensor([(m >> a) & 1 for m in range(nc)], device=self.dev) for a in range(self.nd)]
        ijk = [b[:, None] + q[None] for b, q in zip(base, d)]
        st = [1, self.n[0], self.n[0] * self.n[1]]
        return sum(s * q for s, q in zip(st, ijk)), ijk, self._basis([q.to(F64) for q in d])

    @staticmethod
    def _solve(rows, rhs):
        """w with rows^T w = rhs, and whether a pivot vanished."""
        M = rows.transpose(1, 2)
        LU, piv, _ = torch.linalg.lu_factor_ex(M)
        bad = LU.diagonal(dim1=1, dim2=2).abs().amin(1) < 1e-12 * M.abs().amax((1, 2))
        return torch.linalg.lu_solve(LU, piv, rhs[..., None])[..., 0], bad

    def _hmin(self, ijk):
        return torch.stack([self.h[a][ijk[a]] for a in range(self.nd)]).amin(0)

    def _ghost_rows(self):
        nd, t = self.nd, self.type.flatten()
        ijk = self._ijk(self.gi)
        P = torch.stack([self.c[a][ijk[a]] for a in range(nd)], -1)
        q = self._closest(P) if len(P) else P
        self.bi = q
        d = q - P
        dist = (d * d).sum(-1).sqrt()
        degen = ~(dist >= 1e-9 * self._hmin(ijk))
        nrm = torch.where(degen[:, None], 0.0, d / dist[:, None])
        ip = torch.where(degen[:, None], P, 2.0 * q - P)
        base = [(torch.searchsorted(self.c[a], ip[:, a].contiguous(), right=True) - 1).clamp(0, self.n[a] - 2) for a in range(nd)]
        cidx, cijk, corner = self._corners(base)
        ct = t[cidx]
        selfm = cidx == self.gi[:, None]
        one = selfm.any(1)
        kind2 = degen | ((ct == DEAD) & ~selfm).any(1)
        hb = [self.hc[a][base[a]] for a in range(nd)]
        loc = lambda x: [(x[:, a] - self.c[a][base[a]]) / hb[a] for a in range(nd)]  # noqa: E731
        bIP, xb = self._basis(loc(ip)), loc(q)
        bBI = self._basis(xb)
        g = [nrm[:, a] / hb[a] for a in range(nd)]
        z = torch.zeros_like(g[0])
        if nd == 2:
            gBI = torch.stack([z, g[0], g[1], g[0] * xb[1] + g[1] * xb[0]], -1)
        else:
            gBI = torch.stack([z, g[0], g[1], g[2], g[0] * xb[1] + g[1] * xb[0], g[1] * xb[2] + g[2] * xb[1],
                               g[0] * xb[2] + g[2] * xb[0],
                               g[0] * xb[1] * xb[2] + g[1] * xb[0] * xb[2] + g[2] * xb[0] * xb[1]], -1)
        rows = corner[None].expand(len(P), -1, -1)
        wv, b1 = self._solve(torch.where(selfm[..., None], bBI[:, None], rows), bIP)
        wp, b2 = self._solve(torch.where(selfm[..., None], gBI[:, None], rows), bIP)
        kind2 = kind2 | b1 | b2
        self.bv = torch.where(kind2 | ~one, 0.0, torch.where(selfm, wv, 0.0).sum(1))
        # fallback: the nearest FLUID corner, else the first FLUID face neighbour
        far = sum((self.c[a][cijk[a]] - ip[:, a, None]) ** 2 for a in range(nd))
        far = torch.where(ct == FLUID, far, math.inf)
        pick = cidx.gather(1, far.argmin(1, keepdim=True))[:, 0]
        none = ~torch.isfinite(far.amin(1))
        for a in reversed(range(nd)):
            st = [1, self.n[0], self.n[0] * self.n[1]][a]
            for sgn, ok in ((1, ijk[a] < self.n[a] - 1), (-1, ijk[a] > 0)):
                nb = torch.where(ok, self.gi + sgn * st, self.gi)
                pick = torch.where(none & ok & (t[nb] == FLUID), nb, pick)
        first = torch.zeros_like(wv)
        first[:, 0] = 1.0
        k2 = kind2[:, None]
        self.sidx = torch.where(k2, pick[:, None], torch.where(selfm, self.gi[:, None], cidx))
        self.wv = torch.where(k2, first, torch.where(selfm, 0.0, wv))
        self.wp = torch.where(k2, first, torch.where(selfm, 0.0, wp))

    def body_velocity(self, pts, omega_z, centre):
        out = torch.zeros(len(pts), 3, dtype=F64, device=self.dev)
        out[:, 0], out[:, 1] = -omega_z * (pts[:, 1] - centre[1]), omega_z * (pts[:, 0] - centre[0])
        return out

    def move(self, bodies, omega_z, centre, u, F):
        """The fields after the bodies moved: fresh cells, dead cells, ghosts, faces next to changed cells."""
        old, nd = self.type, self.nd
        self.classify(bodies)
        self.ubi = self.body_velocity(self.bi, omega_z, centre)
        fresh = self.fl & (old != FLUID)
        fi = fresh.flatten().nonzero()[:, 0]
        u = [torch.where(self.dead, 0.0, t) for t in u]
        if len(fi):
            ijk = self._ijk(fi)
            P = torch.stack([self.c[a][ijk[a]] for a in range(nd)], -1)
            q = self._closest(P)
            d = P - q
            dist = (d * d).sum(-1).sqrt()
            bad = ~(dist >= 1e-9 * self._hmin(ijk))
            base = [torch.where(bad | (d[:, a] >= 0), ijk[a], ijk[a] - 1).clamp(0, self.n[a] - 2) for a in range(nd)]
            cidx, _, corner = self._corners(base)
            selfm = cidx == fi[:, None]
            bad = bad | ((self.type.flatten()[cidx] != FLUID) & ~selfm).any(1)
            loc = [(q[:, a] - self.c[a][base[a]]) / self.hc[a][base[a]] for a in range(nd)]
            rows = torch.where(selfm[..., None], self._basis(loc)[:, None], corner[None])
            w, sing = self._solve(rows, (corner[None] * selfm[..., None]).sum(1))
            bad = (bad | sing)[:, None]
            wb = torch.where(bad[:, 0], 1.0, torch.where(selfm, w, 0.0).sum(1))
            w = torch.where(bad | selfm, 0.0, w)
            ub = self.body_velocity(q, omega_z, centre)
            for m in range(nd):
                t = u[m].flatten()
                t[fi] = ub[:, m]
                for _ in range(400):
                    new = (w * t[cidx]).sum(1) + wb * ub[:, m]
                    gap = (new - t[fi]).abs().max()
                    t[fi] = new
                    if float(gap) <= 1e-16:
                        break
                u[m] = t.reshape(self.shape)
        u = self.refresh(u)
        F = [t.clone() for t in F]
        for a in range(nd):
            ch = (self.type != old)
            ch = ch[_sl(a, 0, -1)] | ch[_sl(a, 1, None)]
            F[a][_sl(a, 1, -1)] = torch.where(ch, self.mean_faces(u[a], a), F[a][_sl(a, 1, -1)])
        return u, F, fresh

    # operators ----------------------------------------------------------------

    def refresh(self, u):
        """Dirichlet ghost rows solved for the ghost values (Jacobi passes)."""
        out = []
        for m, t in enumerate(u):
            t = t.flatten().clone()
            for _ in range(120 if len(self.gi) else 0):
                new = (2.0 - self.bv) * self.ubi[:, m] - (self.wv * t[self.sidx]).sum(1)
                gap = (new - t[self.gi]).abs().max()
                t[self.gi] = new
                if float(gap) <= 1e-16:
                    break
            out.append(t.reshape(self.shape))
        return out

    def dirichlet(self, a, side, m):
        code = BC[2 * a + side]
        if code == 0:
            return True, self.p.u_inf[m]
        return (True, 0.0) if code == 2 and m == a else (False, 0.0)

    def mean_faces(self, u, a):
        L, R = self.type[_sl(a, 0, -1)], self.type[_sl(a, 1, None)]
        ok = (L != DEAD) & (R != DEAD) & ((L == FLUID) | (R == FLUID))
        return torch.where(ok, 0.5 * (u[_sl(a, 0, -1)] + u[_sl(a, 1, None)]), 0.0)

    def ends(self, a):
        return ((0, _sl(a, 0, 1)), (1, _sl(a, -1, None)))

    def area(self, a):
        h = list(self.h)
        h[a] = torch.ones(1, dtype=F64, device=self.dev)
        return h[2][:, None, None] * h[1][None, :, None] * h[0][None, None, :]

    def faces(self, u):
        F, net, out = [], 0.0, 0.0
        for a in range(self.nd):
            sh = list(self.shape)
            sh[2 - a] += 1
            t = torch.zeros(sh, dtype=F64, device=self.dev)
            t[_sl(a, 1, -1)] = self.mean_faces(u[a], a)
            A = self.area(a)
            for side, e in self.ends(a):
                code = BC[2 * a + side]
                t[e] = self.p.u_inf[a] if code == 0 else 0.0 if code == 2 else torch.where(self.fl[e], u[a][e], 0.0)
                if code == 1:
                    out = out + torch.where(self.fl[e], A.expand_as(t[e]), 0.0).sum()
                net = net + (1.0 if side == 0 else -1.0) * (A * t[e]).sum()
            F.append(t)
        for a in range(self.nd):
            for side, e in self.ends(a):
                if BC[2 * a + side] == 1:
                    F[a][e] += torch.where(self.fl[e], (-1.0 if side == 0 else 1.0) * net / out, 0.0)
        return F

    def conv(self, u, F, m):
        """Convective term of component m (before the FLUID mask)."""
        acc = torch.zeros(self.shape, dtype=F64, device=self.dev)
        for a in range(self.nd):
            t = torch.empty_like(F[a])
            t[_sl(a, 1, -1)] = 0.5 * (u[_sl(a, 0, -1)] + u[_sl(a, 1, None)])
            for side, e in self.ends(a):
                isd, val = self.dirichlet(a, side, m)
                t[e] = val if isd else u[e]
            t = t * F[a]
            acc += (t[_sl(a, 1, None)] - t[_sl(a, 0, -1)]) / self.bc1(self.h[a], a)
        return torch.where(self.fl, acc, 0.0)

    def viscous(self, u, m, alpha):
        """(alpha sum c u_nb + Dirichlet values, alpha sum c) of component m."""
        off = torch.zeros(self.shape, dtype=F64, device=self.dev)
        D = torch.zeros(self.shape, dtype=F64, device=self.dev)
        wall = torch.zeros(self.shape, dtype=F64, device=self.dev)
        for a in range(self.nd):
            lo = self.bc1(1.0 / (self.hc[a] * self.h[a][:-1]), a)
            hi = self.bc1(1.0 / (self.hc[a] * self.h[a][1:]), a)
            off[_sl(a, 0, -1)] += lo * u[_sl(a, 1, None)]
            off[_sl(a, 1, None)] += hi * u[_sl(a, 0, -1)]
            D[_sl(a, 0, -1)] += lo
            D[_sl(a, 1, None)] += hi
            for side, e in self.ends(a):
                isd, val = self.dirichlet(a, side, m)
                if isd:
                    w2 = 2.0 / self.h[a][0 if side == 0 else -1] ** 2
                    D[e] += w2
                    wall[e] += w2 * val
        return alpha * off, alpha * D, alpha * wall

    def helmholtz(self, rhs, u, m, alpha):
        _, D, _ = self.viscous(u, m, alpha)
        u = torch.where(self.dead, 0.0, u)
        bcs = (2.0 - self.bv) * self.ubi[:, m]
        for _ in range(400):
            off = self.viscous(u, m, alpha)[0]
            new = torch.where(self.fl, (rhs + off) / (1.0 + D), u).flatten()
            if len(self.gi):
                new[self.gi] = bcs - (self.wv * new[self.sidx]).sum(1)
            new = new.reshape(self.shape)
            gap = float((new - u).abs().max())
            u = new
            if gap <= 4e-16:
                break
        return u

    def A(self, x):
        """FLUID rows div grad, GHOST rows x_G - sum wp x_m, DEAD rows 0."""
        y = torch.zeros_like(x)
        for a in range(self.nd):
            g = (x[_sl(a, 1, None)] - x[_sl(a, 0, -1)]) / self.bc1(self.hc[a], a)
            y[_sl(a, 0, -1)] += g / self.bc1(self.h[a][:-1], a)
            y[_sl(a, 1, None)] -= g / self.bc1(self.h[a][1:], a)
        y = torch.where(self.fl, y, 0.0).flatten()
        xf = x.flatten()
        y[self.gi] = xf[self.gi] - (self.wp * xf[self.sidx]).sum(1)
        return y.reshape(self.shape)

    def mean(self, x):
        return (self.vf * x).sum() / self.vsum

    def proj(self, x):
        return torch.where(self.fl, x - self.mean(x), torch.where(self.dead, 0.0, x))

    def _along(self, t, M, a):
        """Contraction of axis a (0 = x) with M's first index."""
        if a == 0:
            return t @ M
        if a == 1:
            return torch.matmul(M.t(), t)
        return (M.t() @ t.reshape(t.shape[0], -1)).reshape(t.shape)

    def separable(self, r):
        """The body-free operator's inverse by the eigenpairs of its 1D parts."""
        if self.eig is None:
            V, mu = [], []
            for a in range(3):
                n = self.n[a]
                K = torch.zeros(n, n, dtype=F64)
                if n > 1:
                    i = torch.arange(n - 1)
                    tt = (1.0 / self.hc[a]).cpu()
                    K[i, i + 1] = tt
                    K[i + 1, i] = tt
                    K[i, i] -= tt
                    K[i + 1, i + 1] -= tt
                s = self.h[a].cpu().rsqrt()
                e, W = torch.linalg.eigh(s[:, None] * K * s[None])
                V.append((s[:, None] * W).to(self.dev))
                mu.append(e.to(self.dev))
            L = mu[2][:, None, None] + mu[1][None, :, None] + mu[0][None, None, :]
            keep = L.abs() > 1e-12 * L.abs().max()
            self.eig = V, torch.where(keep, 1.0 / torch.where(keep, L, 1.0), 0.0)
        V, inv = self.eig
        t = self.vol * r
        for a in range(self.nd):
            t = self._along(t, V[a], a)
        t = t * inv
        for a in range(self.nd):
            t = self._along(t, V[a].t().contiguous(), a)
        if self.nd == 2:
            t = t / self.h[2][0]
        return t

    def pressure(self, b):
        """P A x = P b by BiCGStab; zero FLUID mean, DEAD cells 0."""
        def K(r):
            z = torch.where(self.dead, 0.0, self.separable(torch.where(self.fl, r, 0.0))).flatten()
            z[self.gi] = r.flatten()[self.gi] + (self.wp * z[self.sidx]).sum(1)
            return z.reshape(self.shape)

        def M(x):
            return self.proj(self.A(x))

        dot = lambda x, y: (x * y).sum()  # noqa: E731
        b = self.proj(torch.where(self.fl, b, 0.0))
        x, r = torch.zeros_like(b), b.clone()
        bn = float(dot(b, b).sqrt())
        best = (math.inf, x)
        for _ in range(6):   # restarts from the true residual
            rh, p, v = r.clone(), torch.zeros_like(b), torch.zeros_like(b)
            rho = al = om = torch.ones((), dtype=F64, device=self.dev)
            for _ in range(14):
                rho, old = dot(rh, r), rho
                p = r + rho / old * (al / om) * (p - om * v)
                ph = K(p)
                v = M(ph)
                al = rho / dot(rh, v)
                s = r - al * v
                sh = K(s)
                t = M(sh)
                om = dot(t, s) / dot(t, t)
                x = x + al * ph + om * sh
                r = s - om * t
                if not float(dot(r, r).sqrt()) > 1e-14 * bn:
                    break
            r = b - M(x)
            rel = float(dot(r, r).sqrt()) / bn
            if rel < best[0]:
                best = (rel, x)
            if rel <= 1e-13 or not math.isfinite(rel):
                break
        x = best[1]
        return torch.where(self.dead, 0.0, x - self.mean(x))

    # steps ----------------------------------------------------------------------

    def start(self, seed):
        """(state before the first step): the impulsive start and the bump."""
        u = [torch.where(self.fl, self.p.u_inf[m], 0.0).to(F64) for m in range(self.nd)]
        u = self.refresh(u)
        F = self.faces(u)
        return [t + torch.where(self.fl, d, 0.0) for t, d in zip(u, _bump(self.p, seed, self.dev))], F, None

    def step(self, u, F, Nold, fresh=None):
        dt, alpha = self.p.dt, 0.5 * self.p.dt / self.p.Re
        N = [self.conv(u[m], F, m) for m in range(self.nd)]
        us = []
        for m in range(self.nd):
            old = N[m] if Nold is None else Nold[m]
            if fresh is not None:
                old = torch.where(fresh, N[m], old)
            off, D, wall = self.viscous(u[m], m, alpha)
            rhs = u[m] - dt * (1.5 * N[m] - 0.5 * old) + (off - D * u[m] + 2.0 * wall)
            us.append(self.helmholtz(torch.where(self.fl, rhs, 0.0), u[m], m, alpha))
        F = self.faces(us)
        div = sum((F[a][_sl(a, 1, None)] - F[a][_sl(a, 0, -1)]) / self.bc1(self.h[a], a) for a in range(self.nd))
        phi = self.pressure(torch.where(self.fl, div / dt, 0.0))
        un = []
        for a in range(self.nd):
            g = (phi[_sl(a, 1, None)] - phi[_sl(a, 0, -1)]) / self.bc1(self.hc[a], a)
            some = self.fl[_sl(a, 0, -1)] | self.fl[_sl(a, 1, None)]
            F[a][_sl(a, 1, -1)] -= torch.where(some, dt * g, 0.0)
            half = torch.zeros(self.shape, dtype=F64, device=self.dev)
            half[_sl(a, 0, -1)] += 0.5 * g
            half[_sl(a, 1, None)] += 0.5 * g
            un.append(torch.where(self.fl, us[a] - dt * half, us[a]))
        return self.refresh(un), F, N, phi


def _exact_one(case, seed, dev, bump=True):
    p = _problem(case, seed)
    f = _Flow(p, dev)
    bodies = synth.case_bodies(p)
    f.classify(bodies)
    if case["kind"] == "poisson":
        return f.pressure(_rhs(p, seed, dev))
    u, F, N = f.start(seed)
    if not bump:
        u = f.refresh([torch.where(f.fl, p.u_inf[m], 0.0).to(F64) for m in range(f.nd)])
    phi = None
    for q in range(case["steps"]):
        fresh = None
        if case["kind"] == "move":
            w = math.radians(PITCH) / p.dt * (-1.0 if q == 0 else 1.0)
            verts = _pitch(p, PITCH) if q == 0 else np.array(p.verts)
            u, F, fresh = f.move([(verts, p.elems)], w, (0.25, 0.0), u, F)
        u, F, N, phi = f.step(u, F, N, fresh)
    return {**dict(zip(_velocities(p), u)), "p": phi}


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["nx"] * case["ny"] * case["nz"] > 50_000_000:
        return None   # over 20 seconds
    if case["kind"] == "serve":
        return [{k: v.cpu().numpy() for k, v in _exact_one(c, seed + 31 * q, dev, bump=False).items()}
                for q, c in enumerate(_parts(case))]
    if case["kind"] == "ensemble":
        return [_exact_one(c, seed + 31 * q, dev) for q, c in enumerate(_parts(case))]
    return _exact_one(case, seed, dev)
