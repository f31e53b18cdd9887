"""The calls whose speed matters to a user of the library, as data.

``listed()`` holds one case per kind of work, from the smallest call to the
largest; ``draw()`` gives further cases of the same kinds over the same ranges.
``prepare`` makes what a program has in hand before the call (the handle of its
geometry, the hierarchy, the fields), ``run`` is one pass through the public
entry points, ``work`` the bytes and operations the pass cannot do without and
``exact`` the same outputs from plain torch in 64 bits.

Kinds

* ``apply``     one matrix-free operator application (eb_apply), the call inside
                a user's own iteration: small 2D grids, where only latency
                counts, up to 256^3.
* ``wave``      a run of leapfrog steps (wave_step), FP32 and FP64.
* ``poisson``   one AMG-PCG solve on a hierarchy that is kept (pcg_solve): the
                small FP64 parity grid, 2D stars and the 256^3 ellipsoid with
                the FP32 V-cycle and the FP64 or double-float outer iteration.
* ``heat``      one Crank-Nicolson step with a variable coefficient (heat_step).
* ``batch``     one backward-Euler step of many stars of uneven size at once
                (batch_heat_step).
* ``geometry``  a new domain from scratch: build, right-hand side, hierarchy,
                solve (what a sweep over shapes pays for each of them).
* ``forward``   the learned stage's network on an image (nn_forward).
* ``backward``  its parameter gradient on a training batch (nn_backward).
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import numpy as np
import torch

import paper_2204_06083_gb300 as eb
from paper_2204_06083_gb300 import learned

DTYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
PRECS = {"f64": eb.EB_F64, "f32": eb.EB_F32, "bf16": eb.EB_BF16, "df": eb.EB_DF64}
SIZE = {"f64": 8, "f32": 4, "bf16": 2}


def listed():
    return [
        # one apply on the smallest grid of the tests and the benchmark: launch and call latency
        dict(name="apply_f64_128", kind="apply", dim=2, n0=128, n1=127, n2=1, dtype="f64"),
        # the operator on the benchmark's 3D grid in the V-cycle's precision
        dict(name="apply_f32_256c", kind="apply", dim=3, n0=256, n1=256, n2=256, dtype="f32"),
        # the wave workload's grid and data type
        dict(name="wave_f32_4096", kind="wave", n0=4096, n1=4096, dtype="f32", steps=256),
        # the same scheme in FP64 on a ragged middle-sized grid, a run that is no multiple of a graph's chunk
        dict(name="wave_f64_1530", kind="wave", n0=1530, n1=1501, dtype="f64", steps=100),
        # the small FP64 Poisson solve (latency-bound)
        dict(name="poisson_f64_128", kind="poisson", dim=2, n0=128, n1=128, n2=1, vcycle="f64", outer="f64"),
        # an ordinary 2D solve with the mixed-precision V-cycle
        dict(name="poisson_f32_1022", kind="poisson", dim=2, n0=1022, n1=1027, n2=1, vcycle="f32", outer="f64"),
        # the benchmark's headline solve
        dict(name="poisson_df_256c", kind="poisson", dim=3, n0=256, n1=256, n2=256, vcycle="f32", outer="df"),
        # a Crank-Nicolson step with a variable coefficient on a middle-sized grid
        dict(name="heat_beta_1200", kind="heat", n0=1200, n1=1187, vcycle="f32", outer="df"),
        # the batched workload: 64 stars of 128..1024 nodes per axis
        dict(name="batch_64", kind="batch", count=64, nmin=128, nmax=1024, layout=0, vcycle="f32", outer="df"),
        # a new domain from scratch, as in a sweep over shapes
        dict(name="geometry_514", kind="geometry", dim=2, n0=514, n1=501, n2=1, vcycle="f32", outer="f64"),
        # the learned stage on the image of the learned workload
        dict(name="forward_2048", kind="forward", images=1, h=2048, w=2048),
        # the gradient of one training batch of the learned workload
        dict(name="backward_16x512", kind="backward", images=16, h=512, w=512),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _even(v):
    return 2 * int(round(v / 2))


def draw(rng):
    kind = rng.choice(["apply", "wave", "poisson", "heat", "batch", "geometry", "forward", "backward"])
    if kind in ("apply", "poisson", "geometry"):
        dim = rng.choice([2, 3])
        top = {"apply": (2048, 254), "poisson": (1200, 200), "geometry": (1000, 128)}[kind][dim - 2]
        n0 = _even(_log(rng, 96 if dim == 2 else 40, top))
        near = lambda: int(round(n0 * rng.uniform(0.92, 1.0)))
        n1, n2 = near(), near() if dim == 3 else 1
        c = dict(kind=kind, dim=dim, n0=n0, n1=n1, n2=n2)
        if kind == "apply":
            return dict(c, dtype=rng.choice(["f64", "f32", "bf16"]))
        vcycle, outer = rng.choice([("f32", "df"), ("f32", "f64"), ("f64", "f64")])
        return dict(c, vcycle=vcycle, outer=outer)
    if kind == "wave":
        n0 = _even(_log(rng, 128, 4096))
        return dict(kind=kind, n0=n0, n1=int(n0 * rng.uniform(0.9, 1.0)), dtype=rng.choice(["f32", "f64"]),
                    steps=int(_log(rng, 8, 256)))
    if kind == "heat":
        n0 = _even(_log(rng, 200, 1200))
        return dict(kind=kind, n0=n0, n1=int(n0 * rng.uniform(0.92, 1.0)), vcycle="f32",
                    outer=rng.choice(["df", "f64"]))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 48), nmin=100, nmax=_even(_log(rng, 200, 1000)),
                    layout=rng.randint(1, 1 << 20), vcycle="f32", outer=rng.choice(["df", "f64"]))
    if kind == "forward":
        return dict(kind=kind, images=rng.randint(1, 3), h=int(_log(rng, 33, 1150)), w=int(_log(rng, 33, 1150)))
    return dict(kind=kind, images=rng.randint(1, 12), h=int(_log(rng, 48, 560)), w=int(_log(rng, 48, 560)))


# ------------------------------------------------------------------ geometries

def _grid(dim, n0, n1, n2, half=1.0):
    """A box with n0 nodes over [-half, half] and the same h on the other axes, centred."""
    h = 2.0 * half / (n0 - 1)
    n = (n0, n1, n2 if dim == 3 else 1)
    lo = tuple(-0.5 * h * (k - 1) if k > 1 else 0.0 for k in n)
    return SimpleNamespace(dim=dim, n=n, lo=lo, h=h)


def _star(rng):
    """The benchmark's random stars: r = 0.5 + sum_{k=2..6} a_k sin(k phi + p_k) about (0.02, 0.01)."""
    return SimpleNamespace(kind=eb.EB_LS_STAR2D, center=(0.02, 0.01, 0.0), semi=(1.0, 1.0, 1.0),
                           rot=(1.0, 0.0, 0.0, 0.0, 1.0, 0.0, 0.0, 0.0, 1.0), r0=0.5, ks=[2, 3, 4, 5, 6],
                           amps=[rng.uniform(0.0, 0.05) for _ in range(5)],
                           phases=[rng.uniform(0.0, 2.0 * math.pi) for _ in range(5)], psi=None)


def _quadric(rng, dim):
    """Circle of radius 0.5 (2D) or the ellipsoid (0.7, 0.5, 0.4) in a seeded rotation (3D)."""
    if dim == 2:
        return SimpleNamespace(kind=eb.EB_LS_QUADRIC, semi=(0.5, 0.5, 1.0),
                               center=(0.02 * rng.uniform(-1.0, 1.0), 0.02 * rng.uniform(-1.0, 1.0), 0.0),
                               rot=(1.0, 0.0, 0.0, 0.0, 1.0, 0.0, 0.0, 0.0, 1.0), r0=0.5, ks=[], amps=[], phases=[],
                               psi=None)
    q, r = np.linalg.qr(np.array([[rng.gauss(0.0, 1.0) for _ in range(3)] for _ in range(3)]))
    q = q * np.sign(np.diag(r))[None, :]
    if np.linalg.det(q) < 0:
        q[:, 0] = -q[:, 0]
    return SimpleNamespace(kind=eb.EB_LS_QUADRIC, center=(0.0, 0.0, 0.0), semi=(0.7, 0.5, 0.4),
                           rot=tuple(float(v) for v in q.ravel()), r0=0.5, ks=[], amps=[], phases=[], psi=None)


def _domain(case, seed):
    """(grid, level set, generator of plain random numbers) of a single-grid case."""
    rng = random.Random(1000003 * seed + case["n0"])
    dim = case.get("dim", 2)
    g = _grid(dim, case["n0"], case["n1"], case.get("n2", 1))
    quadric = dim == 3 or case["n0"] <= 128
    return g, (_quadric(rng, dim) if quadric else _star(rng)), rng


def _shape(g):
    return (g.n[1], g.n[0]) if g.dim == 2 else (g.n[2], g.n[1], g.n[0])


def _coords(g):
    """Coordinates of the nodes, broadcastable over the grid's shape (x fastest)."""
    out = []
    for a in range(g.dim):
        v = g.lo[a] + torch.arange(g.n[a], dtype=torch.float64, device="cuda") * g.h
        out.append(v.view([-1 if g.dim - 1 - a == k else 1 for k in range(g.dim)]))
    return out


def _solution(coefs, pts, t=0.0):
    """Manufactured solution at the points (seeded wave numbers and phases)."""
    (kx, px, ky, py) = coefs
    u = torch.sin(kx * pts[0] + px) * torch.cos(ky * pts[1] + py)
    if len(pts) == 3:
        u = u * torch.exp(pts[2])
    return math.exp(-t) * u


def _source(coefs, pts):
    """Its Laplacian."""
    (kx, _, ky, _) = coefs
    return ((1.0 if len(pts) == 3 else 0.0) - kx * kx - ky * ky) * _solution(coefs, pts)


def _heat_f(coefs, pts, t):
    """-F of the heat equation u_t = Lap u + F with the manufactured solution."""
    return _solution(coefs, pts, t) + math.exp(-t) * _source(coefs, pts)


def _coefs(rng):
    return rng.uniform(1.5, 2.5), rng.uniform(0.0, 1.0), rng.uniform(2.5, 3.5), rng.uniform(0.0, 1.0)


def _columns(xg):
    return [xg[:, a] for a in range(xg.shape[1])]


def _beta(pts):
    return 2.0 + torch.sin(pts[0] * pts[1])


def _half_betas(g):
    pts = _coords(g)
    return [_beta([p + (0.5 * g.h if b == a else 0.0) for b, p in enumerate(pts)]).expand(_shape(g)).contiguous()
            for a in range(g.dim)]


def _rhs(handle, g, coefs, scale=1.0):
    f = (scale * _source(coefs, _coords(g))).expand(_shape(g)).contiguous()
    ug = _solution(coefs, _columns(handle.cuts()[3])).contiguous()
    return handle.rhs(f, ug)


def _stars(case, seed):
    """Grids and stars of a batch case: uneven even widths, some grids shorter than wide.  The sizes are the case's
    own, so that every seed has the same amount of work; the shapes are the seed's."""
    sizes = random.Random(case["layout"])
    rng = random.Random(1000003 * seed + case["count"])
    out = []
    for _ in range(case["count"]):
        n0 = _even(sizes.uniform(case["nmin"], case["nmax"]))
        out.append((_grid(2, n0, n0 - sizes.randint(0, n0 // 16), 1), _star(rng)))
    return out, rng


def _pulse(pts, rng):
    rr, th, w = 0.25 * math.sqrt(rng.random()), rng.uniform(0.0, 2.0 * math.pi), rng.uniform(0.02, 0.05)
    cx, cy = 0.02 + rr * math.cos(th), 0.01 + rr * math.sin(th)
    return torch.exp(-((pts[0] - cx) ** 2 + (pts[1] - cy) ** 2) / (w * w))


RTOL = {"poisson": 1e-12, "heat": 1e-12, "batch": 1e-12, "geometry": 1e-12}


def _params(seed):
    """Network parameters of ordinary size (the initialisation of training, all layers alive, nonzero biases)."""
    p = learned.init_params(seed % 1000, last_scale=0.5)
    rng = np.random.default_rng(seed % 1000 + 1)
    return (p + (p == 0) * rng.uniform(-0.05, 0.05, size=p.shape)).astype(np.float32)


def _image(case, seed):
    """(s_hat, m): residuals of unit rms on the CPs, m the mask of a disk-like domain in every image."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n, h, w = case["images"], case["h"], case["w"]
    s = torch.randn((n, h, w), generator=gen, device="cuda", dtype=torch.float32)
    y = torch.linspace(-1.0, 1.0, h, device="cuda").view(1, h, 1)
    x = torch.linspace(-1.0, 1.0, w, device="cuda").view(1, 1, w)
    r = 0.6 + 0.2 * torch.rand((n, 1, 1), generator=gen, device="cuda")
    m = ((x * x + y * y) < r * r).float()
    d = torch.randn((n, h, w), generator=gen, device="cuda", dtype=torch.float32)
    return torch.stack([s * m, m.expand(n, h, w)], dim=-1).contiguous(), d * m


# ----------------------------------------------------------------- prepare, run

def prepare(case, seed):
    kind = case["kind"]
    if kind in ("forward", "backward"):
        inp, dout = _image(case, seed)
        return SimpleNamespace(kind=kind, net=eb.Net(_params(seed)), inp=inp, dout=dout)
    if kind == "batch":
        geos, rng = _stars(case, seed)
        b = eb.Batch([g for g, _ in geos], [l for _, l in geos])
        coefs = _coefs(rng)
        f, u0, ug, dts = b.zeros(), b.zeros(), torch.zeros(b.num_cut, dtype=torch.float64, device="cuda"), []
        for k, (g, _) in enumerate(geos):
            dts.append(g.h)
            geo, pts = b.geometry(k), _coords(g)
            b.view(f, k).copy_(_heat_f(coefs, pts, g.h))
            b.view(u0, k).copy_(_solution(coefs, pts) * ((geo.classes() & eb.CODE_CP) != 0))
            ug[b.cut_off[k]:b.cut_off[k + 1]] = _solution(coefs, _columns(geo.cuts()[3]), g.h)
        b.heat_setup(dts, theta=1.0, vcycle_prec=PRECS[case["vcycle"]])
        b.set_outer(PRECS[case["outer"]])
        return SimpleNamespace(kind=kind, batch=b, u0=u0, b1=b.rhs(f, ug))
    g, ls, rng = _domain(case, seed)
    if kind == "geometry":
        coefs = _coefs(rng)
        f = _source(coefs, _coords(g)).expand(_shape(g)).contiguous()
        return SimpleNamespace(kind=kind, g=g, ls=ls, f=f, coefs=coefs, vcycle=PRECS[case["vcycle"]],
                               outer=PRECS[case["outer"]])
    h = eb.EB(g, ls)
    if kind == "apply":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn(_shape(g), generator=gen, device="cuda", dtype=torch.float64).to(DTYPES[case["dtype"]])
        return SimpleNamespace(kind=kind, h=h, x=x, out=torch.zeros_like(x))
    if kind == "wave":
        dt = 0.9 * g.h / math.sqrt(2.0)
        u0 = _pulse(_coords(g), rng) * ((h.classes() & eb.CODE_CP) != 0)
        u1 = u0 - 0.5 * dt * dt * h.apply(u0)
        t = DTYPES[case["dtype"]]
        return SimpleNamespace(kind=kind, h=h, dt=dt, steps=case["steps"], up=u0.to(t), uc=u1.to(t))
    coefs = _coefs(rng)
    if kind == "heat":
        h.set_beta(_half_betas(g))
        amg = eb.AMG(h, 1.0 / (0.5 * g.h), vcycle_prec=PRECS[case["vcycle"]])
        amg.set_outer(PRECS[case["outer"]])
        u0 = _solution(coefs, _coords(g)) * ((h.classes() & eb.CODE_CP) != 0)
        return SimpleNamespace(kind=kind, h=h, amg=amg, dt=g.h, u0=u0, b0=_rhs(h, g, coefs),
                               b1=_rhs(h, g, coefs, 0.9))
    amg = eb.AMG(h, vcycle_prec=PRECS[case["vcycle"]])
    return SimpleNamespace(kind=kind, h=h, amg=amg, b=_rhs(h, g, coefs), outer=PRECS[case["outer"]])


def run(state):
    kind = state.kind
    if kind == "apply":
        return state.h.apply(state.x, state.out)
    if kind == "wave":
        state.h.wave_step(state.up, state.uc, state.dt, state.steps)
        return state.up, state.uc
    if kind == "poisson":
        return state.amg.solve(state.b, rtol=RTOL[kind], outer=state.outer)[0]
    if kind == "heat":
        u = state.u0.clone()
        state.amg.heat_step(u, state.b1, state.dt, theta=0.5, b0=state.b0, rtol=RTOL[kind])
        return u
    if kind == "batch":
        u = state.u0.clone()
        state.batch.heat_step(u, state.b1, rtol=RTOL[kind])
        return u
    if kind == "geometry":
        h = eb.EB(state.g, state.ls)
        b = h.rhs(state.f, _solution(state.coefs, _columns(h.cuts()[3])).contiguous())
        amg = eb.AMG(h, vcycle_prec=state.vcycle)
        return {"code": h.classes(), "x": amg.solve(b, rtol=RTOL[kind], outer=state.outer)[0]}
    if kind == "forward":
        return state.net.forward(state.inp)
    state.net.backward(state.inp, state.dout)
    return state.net.params()[1]


# ------------------------------------------------------------------------- work

def _unknowns(dim, n0):
    h = 2.0 / (n0 - 1)
    return math.pi * 0.25 / h ** 2 if dim == 2 else 4.0 / 3.0 * math.pi * 0.14 / h ** 3


def work(case):
    kind = case["kind"]
    if kind in ("forward", "backward"):
        px = case["images"] * case["h"] * case["w"]
        fl = px * 2 * 9 * (2 * 32 + 4 * 32 * 32 + 32)
        # forward: two floats in, one out.  backward: the same inputs and the output gradient; forward, the
        # activation gradients of layers 2-6 and the weight gradients of all six.
        if kind == "forward":
            return {"bytes": px * 12, "flops": fl}
        return {"bytes": px * 12, "flops": 2 * fl + px * 2 * 9 * (4 * 32 * 32 + 32)}
    if kind == "batch":
        n = sum(_unknowns(2, g.n[0]) for g, _ in _stars(case, 0)[0])
        return {"bytes": n * 24, "flops": n * 100}
    n = _unknowns(case.get("dim", 2), case["n0"])
    if kind == "apply":
        return {"bytes": n * (2 * SIZE[case["dtype"]] + 1), "flops": n * (2 * case["dim"] + 2)}
    if kind == "wave":  # both fields in and out once, whatever the number of steps; the arithmetic of every step
        return {"bytes": n * (4 * SIZE[case["dtype"]] + 1), "flops": n * 8 * case["steps"]}
    # solves: b (and u) in, x out; at least some ten operator and preconditioner applications
    return {"bytes": n * (32 if kind == "heat" else 16), "flops": n * 10 * 60}


# ------------------------------------------------------------------------ exact

def _psi(ls, pts):
    """The level set at points given by their coordinates."""
    d = [p - ls.center[a] for a, p in enumerate(pts)]
    if ls.kind == eb.EB_LS_STAR2D:
        phi = torch.atan2(d[1], d[0])
        r = ls.r0
        for k, a, p in zip(ls.ks, ls.amps, ls.phases):
            r = r + a * torch.sin(k * phi + p)
        return torch.sqrt(d[0] * d[0] + d[1] * d[1]) - r
    n = len(pts)
    return sum((sum(ls.rot[3 * b + a] * d[b] for b in range(n)) / ls.semi[a]) ** 2 for a in range(n)) - 1.0


def _shift(v, axis, way):
    """The neighbour's value in direction (axis, way) at every node; axis 0 is x, the last dimension."""
    return torch.roll(v, -way, v.dim() - 1 - axis)


class _Plain:
    """Algorithm 1 in plain torch: the CPs, h^2 A and the boundary terms of h^2 b."""

    def __init__(self, g, ls, beta=None):
        self.g, pts = g, _coords(g)
        inside = (_psi(ls, pts) < 0).expand(_shape(g))
        dirs = [(a, w) for a in range(g.dim) for w in (-1, 1)]
        bp = torch.zeros_like(inside)
        for a, w in dirs:
            bp = bp | (inside & ~_shift(inside, a, w))
        cp = inside & ~bp
        self.inside, self.bp, self.cp, self.m = inside, bp, cp, cp.double()
        self.diag, self.cuts, self.nb = torch.zeros_like(self.m), [], []
        betas = _half_betas(g) if beta else None
        for a, w in dirs:
            bt = 1.0 if betas is None else (betas[a] if w > 0 else _shift(betas[a], a, -1))
            self.nb.append((a, w, bt))
            c = torch.ones_like(self.m)
            idx = torch.nonzero(cp & _shift(bp, a, w))
            # walk outward from the BP to the last inside node, then bisect to the crossing
            at = idx.clone()
            ax = g.dim - 1 - a
            at[:, ax] += w
            steps = torch.zeros(idx.shape[0], dtype=torch.float64, device="cuda")
            while True:
                nxt = at.clone()
                nxt[:, ax] += w
                go = inside[tuple(nxt.t())]
                if not bool(go.any()):
                    break
                at[go] = nxt[go]
                steps += go
            base = [g.lo[b] + at[:, g.dim - 1 - b].double() * g.h for b in range(g.dim)]
            lo, hi = torch.zeros_like(steps), torch.full_like(steps, g.h)
            for _ in range(60):
                mid = 0.5 * (lo + hi)
                neg = _psi(ls, [p + (w * mid if b == a else 0.0) for b, p in enumerate(base)]) < 0
                lo, hi = torch.where(neg, mid, lo), torch.where(neg, hi, mid)
            t = 0.5 * (lo + hi)
            cut = g.h / (g.h + steps * g.h + t)
            where = tuple(idx.t())
            c[where] = cut
            b_at = bt if betas is None else bt[where]
            self.cuts.append((where, b_at * cut, [p + (w * t if b == a else 0.0) for b, p in enumerate(base)]))
            self.diag += c * bt
        self.diag *= self.m

    def apply(self, x):
        """h^2 A x for x that is 0 off the CPs."""
        y = self.diag * x
        for a, w, bt in self.nb:
            y = y - bt * _shift(x, a, w)
        return y * self.m

    def rhs(self, f, coefs, t=0.0):
        """h^2 b of A u = b for div(beta grad u) = f."""
        b = -self.g.h ** 2 * f * self.m
        for where, c, pts in self.cuts:
            b[where] += c * _solution(coefs, pts, t)
        return b

    def solve(self, b, shift=0.0, x=None):
        """(shift h^2 I + h^2 A) x = b by CG with the diagonal, down to rounding; then once more from the residual."""
        s = shift * self.g.h ** 2
        x = torch.zeros_like(b) if x is None else x
        di = self.m / torch.where(self.cp, self.diag + s, torch.ones_like(self.m))
        for _ in range(2):
            r = b - self.apply(x) - s * x
            z = di * r
            p, rz, e, best = z, torch.sum(r * z), torch.zeros_like(b), None
            for k in range(20000):
                q = self.apply(p) + s * p
                al = rz / torch.sum(p * q)
                e = e + al * p
                r = r - al * q
                z = di * r
                new = torch.sum(r * z)
                p = z + (new / rz) * p
                rz = new
                if k % 50 == 0:
                    now = float(rz)
                    best = now if best is None else best
                    if not now > 1e-30 * best:
                        break
            x = x + e
        return x


def exact(case, seed):
    kind = case["kind"]
    if kind == "backward":
        return None  # sums with heavy cancellation of activations that are stored in 16 bits by design
    if kind == "forward":
        inp, _ = _image(case, seed)
        p = torch.tensor(_params(seed), dtype=torch.float64, device="cuda")
        outs = []
        for k in range(case["images"]):
            v, at = inp[k].double().permute(2, 0, 1), 0
            h, w = v.shape[1:]
            for layer, (ci, co) in enumerate([(2, 32)] + 4 * [(32, 32)] + [(32, 1)]):
                W = p[at:at + co * 9 * ci].view(co, 3, 3, ci)
                bias = p[at + co * 9 * ci:at + co * 9 * ci + co]
                at += co * 9 * ci + co
                pad = torch.nn.functional.pad(v, (1, 1, 1, 1))
                acc = bias.view(co, 1).expand(co, h * w).clone()
                for dy in range(3):
                    for dx in range(3):
                        acc += W[:, dy, dx, :] @ pad[:, dy:dy + h, dx:dx + w].reshape(ci, h * w)
                v = acc.view(co, h, w)
                if layer < 5:
                    v = torch.relu(v)
            outs.append(v[0] * inp[k, :, :, 1])
        return torch.stack(outs)
    if kind == "batch":
        geos, rng = _stars(case, seed)
        coefs = _coefs(rng)
        stride = max(g.n[0] for g, _ in geos)
        parts = []
        for g, ls in geos:
            o, pts = _Plain(g, ls), _coords(g)
            f = _heat_f(coefs, pts, g.h)
            u0 = _solution(coefs, pts) * o.m
            u = o.solve(g.h * u0 + o.rhs(f, coefs, g.h), 1.0 / g.h, u0)
            parts.append(torch.nn.functional.pad(u, (0, stride - g.n[0])).reshape(-1))
        return torch.cat(parts)
    g, ls, rng = _domain(case, seed)
    if kind == "apply":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        x = torch.randn(_shape(g), generator=gen, device="cuda", dtype=torch.float64).to(DTYPES[case["dtype"]])
        o = _Plain(g, ls)
        return o.apply(x.double() * o.m) / g.h ** 2
    if kind == "wave":
        o, t = _Plain(g, ls), DTYPES[case["dtype"]]
        lam = (0.9 / math.sqrt(2.0)) ** 2
        u0 = _pulse(_coords(g), rng) * o.m
        up, uc = u0.to(t).double(), (u0 - 0.5 * lam * o.apply(u0)).to(t).double()
        for _ in range(case["steps"]):
            up, uc = uc, 2.0 * uc - up - lam * o.apply(uc)
        return up, uc
    coefs = _coefs(rng)
    pts = _coords(g)
    if kind == "heat":
        o, h2, th = _Plain(g, ls, beta=True), g.h ** 2, 0.5
        u0 = _solution(coefs, pts) * o.m
        b0, b1 = o.rhs(_source(coefs, pts), coefs), o.rhs(0.9 * _source(coefs, pts), coefs)
        s = 1.0 / (th * g.h)
        b = s * h2 * u0 - (1 - th) / th * o.apply(u0) + b1 + (1 - th) / th * b0
        return o.solve(b, s, u0)
    o = _Plain(g, ls)
    x = o.solve(o.rhs(_source(coefs, pts), coefs))
    if kind == "poisson":
        return x
    code = torch.zeros(_shape(g), dtype=torch.uint8, device="cuda")
    code[o.bp] = eb.CODE_BP
    code[o.cp] = eb.CODE_CP
    for s, (a, w, _) in enumerate(o.nb):
        code[o.cp & _shift(o.bp, a, w)] |= 1 << s
    return {"code": code, "x": x}
