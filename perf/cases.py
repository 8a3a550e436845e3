"""The work that users of this solver have it do, as timed cases.

A case is one pass of a program through the public entry points:

  march    a solver handle takes `steps` time steps; the program then reads the
           state and the moments (bz_step, bz_get_state, bz_moments).  Passes
           go on from one another; every few of them the next realisation of
           the same unsteady flow begins (bz_set_state)
  adjoint  a backward sweep of `steps` adjoint steps over stored states
           (bz_adjoint_step), as a gradient computation takes them
  rollout  gradients of a wall-shear objective through `steps` steps
           (autodiff.rollout and its backward pass)
  batch    many uneven cavities advanced together (bz_batch_step)
  collide  the relaxation of a state that the caller owns (bz_collide_noalloc)

The moments, the lid shear and the lid gradient are doubles in the interface;
a program with an FP32 state keeps them with the accuracy they carry, as FP32.

`exact` computes the same passes in 64-bit PyTorch from the equations of the
method (Philox sampling, upwind streaming with diffuse walls, the Monte Carlo
collision sum, the conservation correction), the gradients by autograd.
"""
import math
import random

import numpy as np
import torch

from paper_1005_5405_gb300 import autodiff, binding, workloads

# A march starts over from its initial state after this many steps, with the
# samples of the steps that follow (one more realisation of an ensemble).
_WINDOW = 48

# Keys of a march, adjoint, rollout or collide case that may be left out.
_DEFAULTS = dict(kn=1.0, vmax=4.0, nt=1000, dtype="f32", u0=0.1, amp=0.0, period=0.0, profile=False,
                 per_cell=False, rv=0.0, rx=0.0, ry=0.0, steps=10)


def listed():
    return [
        # The smallest grid in use, in double precision: a validation run,
        # where a step is a handful of short launches.
        dict(name="cavity16_v12_f64", kind="march", nx=16, ny=16, nv=12, vmax=4.0, nt=1000, dtype="f64"),
        # A double-precision run on an odd, ragged grid with stretched cells.
        dict(name="ragged33x47_v14_f64", kind="march", nx=33, ny=47, nv=14, vmax=3.0, nt=3000, dtype="f64",
             kn=0.5, u0=0.05, rv=0.96, rx=0.99, ry=0.995),
        # An ordinary single-precision cavity.
        dict(name="cavity64_v24", kind="march", nx=64, ny=64, nv=24, vmax=4.5, nt=10000, kn=0.1),
        # The largest cavity: oscillating lid, 8.6 GB per state.
        dict(name="cavity256_v32", kind="march", nx=256, ny=256, nv=32, vmax=5.0, nt=20000, kn=0.05, u0=0.0,
             amp=0.05, period=50.0),
        # The paper's own production setups: transitional flow and near-continuum
        # flow on stretched grids (20 and 18 nodes per axis).
        dict(name="paper_delta1", kind="march", nx=160, ny=160, nv=20, vmax=3.0, nt=6144, kn=1.0, u0=0.01,
             rv=0.945, rx=0.996, ry=0.998),
        dict(name="paper_delta10", kind="march", nx=192, ny=192, nv=18, vmax=3.0, nt=8192, kn=0.1, u0=0.01,
             rv=0.970, rx=0.990, ry=0.995),
        # A ragged single-precision grid that no kernel is specialised for.
        dict(name="ragged97x61_v28", kind="march", nx=97, ny=61, nv=28, vmax=5.0, nt=12000, kn=0.3, u0=0.2),
        # Independent sample sets in every cell (no noise shared by cells).
        dict(name="percell64_v24", kind="march", nx=64, ny=64, nv=24, vmax=4.5, nt=10000, kn=0.1, per_cell=True,
             steps=4),
        # A backward sweep over stored states with a lid profile.
        dict(name="adjoint128_v20", kind="adjoint", nx=128, ny=128, nv=20, vmax=4.5, nt=5000, kn=0.2, profile=True,
             steps=4),
        # Optimisation of a lid profile: checkpointed forward and backward pass.
        dict(name="rollout64_v16", kind="rollout", nx=64, ny=64, nv=16, vmax=4.0, nt=4000, kn=0.5, profile=True,
             steps=8, every=4),
        # A parameter study: uneven cavities advanced as one batch.
        dict(name="batch16", kind="batch", n=16, nt=5000, first=100, steps=6),
        # The relaxation alone on memory that belongs to the caller.
        dict(name="collide64_v24", kind="collide", nx=64, ny=64, nv=24, vmax=4.5, nt=10000, steps=1),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def vbox(nv):
        return 3.0 if nv <= 10 else 4.0 if nv <= 18 else 4.5 if nv <= 26 else 5.0

    def grid(lo, hi, nv, most, kind="march", **more):
        # Cells of at most 0.2 mean free paths, samples in proportion to the
        # velocity nodes, as in the setups above.
        nx, ny = log(lo, hi), log(lo, hi)
        kn = max(math.exp(rng.uniform(math.log(0.05), math.log(5.0))), 5.0 / min(nx, ny))
        nt = min(most, int(nv ** 3 * math.exp(rng.uniform(math.log(0.15), math.log(1.2)))))
        return dict(kind=kind, nx=nx, ny=ny, nv=nv, vmax=vbox(nv), nt=max(200, nt), kn=round(kn, 4),
                    u0=round(rng.uniform(0.01, 0.2), 4), **more)

    what = rng.choice(["march", "march", "march", "stretched", "f64", "per_cell", "adjoint", "rollout", "batch",
                       "collide"])
    if what == "batch":
        return dict(kind="batch", n=rng.randint(3, 16), nt=log(2000, 8000), first=rng.randint(200, 900),
                    steps=rng.randint(3, 8))
    if what == "march":
        return grid(12, 220, rng.choice([12, 14, 16, 18, 20, 22, 24, 26, 28, 30, 32]), 20000,
                    steps=rng.randint(6, 14))
    if what == "stretched":
        c = grid(16, 190, rng.choice([14, 16, 18, 20, 24]), 9000, steps=rng.randint(6, 14))
        return dict(c, vmax=3.0, rv=round(rng.uniform(0.94, 0.98), 3), rx=round(rng.uniform(0.985, 0.998), 3),
                    ry=round(rng.uniform(0.985, 0.998), 3))
    if what == "f64":
        return grid(8, 64, rng.choice([8, 9, 10, 11, 12, 14, 15, 16, 18]), 5000, dtype="f64",
                    steps=rng.randint(6, 12))
    if what == "per_cell":
        return grid(12, 80, rng.choice([12, 15, 16, 18, 20, 24]), 10000, per_cell=True, steps=rng.randint(2, 5))
    if what == "adjoint":
        return grid(16, 128, rng.choice([12, 14, 16, 18, 20, 24]), 6000, kind="adjoint", profile=True,
                    steps=rng.randint(2, 5))
    if what == "rollout":
        return grid(10, 64, rng.choice([12, 16, 20]), 5000, kind="rollout", profile=True, steps=rng.randint(4, 10),
                    every=rng.randint(2, 5))
    return grid(12, 96, rng.choice([10, 12, 16, 18, 20, 24]), 12000, kind="collide", steps=1)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _full(case):
    return {**_DEFAULTS, **case}


def _problem(case, seed):
    """The problem statement of a march, adjoint, rollout or collide case."""
    c = _full(case)
    prof = c["u0"] + 0.1 * c["u0"] * np.random.default_rng(seed).standard_normal(c["nx"]) if c["profile"] else None
    return workloads.Problem("case", c["nx"], c["ny"], c["kn"], c["nv"], c["vmax"], c["nt"], seed % 2**32,
                             dtype=c["dtype"], lid_u0=c["u0"], lid_amp=c["amp"], lid_period=c["period"],
                             lid_profile=prof, eps=0.1 if c["kind"] == "collide" else 0.0, per_cell=c["per_cell"],
                             rv=c["rv"], rx=c["rx"], ry=c["ry"])


def _batch_problems(case, seed):
    """n uneven cavities: square grids of 32 to 128 cells a side, 16, 20 or 24
    velocity nodes per axis, Kn log-uniform, the sizes fixed by the case."""
    out = []
    for k in range(case["n"]):
        r = random.Random(case["first"] + k)
        side, nv = r.choice([32, 48, 64, 96, 128]), r.choice([16, 20, 24])
        kn = max(math.exp(r.uniform(math.log(0.05), math.log(5.0))), 5.0 / side)
        out.append(workloads.Problem("case", side, side, kn, nv,
                                     4.0 if nv == 16 else 4.5, case["nt"], (seed + k) % 2**32,
                                     lid_u0=r.uniform(0.01, 0.2), instance=k))
    return out


def _nodes(p):
    """Node velocities along one axis, their widths and the cell edges (float64)."""
    n, m = p.nv, p.nv // 2
    if p.rv > 0 and p.rv != 1:
        q = 1.0 / p.rv
        d0 = p.vmax * (q - 1.0) / (q ** m - 1.0)
        pos = [d0 * (q ** i - 1.0) / (q - 1.0) for i in range(m + 1)]
        e = np.array([-x for x in pos[:0:-1]] + pos)
        return 0.5 * (e[1:] + e[:-1]), e[1:] - e[:-1], e
    dv = 2.0 * p.vmax / n
    return -p.vmax + (np.arange(n) + 0.5) * dv, np.full(n, dv), -p.vmax + np.arange(n + 1) * dv


def _state(p, seed, noise=0.01):
    """A flow in progress: smooth density, velocity, temperature and shear
    fields over the cavity (a few random modes) and noise per node."""
    dt = torch.float64 if p.dtype == "f64" else torch.float32
    rng = np.random.default_rng(seed)
    x, y = (np.arange(p.nx) + 0.5) / p.nx, (np.arange(p.ny) + 0.5) / p.ny
    f = np.zeros((6, p.ny, p.nx))
    for k in range(6):
        for a in range(3):
            for b in range(3):
                ph = rng.uniform(0, 2 * math.pi, 2)
                f[k] += rng.standard_normal() * 0.2 / (1 + a + b) * np.outer(np.cos(math.pi * b * y + ph[0]),
                                                                            np.cos(math.pi * a * x + ph[1]))
    coef = torch.from_numpy(f.reshape(6, -1).T.copy()).cuda()
    a = torch.from_numpy(_nodes(p)[0]).cuda()
    vx, vy, vz = (v.reshape(-1) for v in torch.meshgrid(a, a, a, indexing="ij"))
    basis = torch.stack([torch.ones_like(vx), 2 * vx, 2 * vy, 2 * vz, vx * vx + vy * vy + vz * vz - 1.5, 2 * vx * vy])
    gen = torch.Generator(device="cuda").manual_seed(seed)
    h = torch.randn((p.nr, p.nvt), generator=gen, device="cuda", dtype=dt).mul_(noise)
    step = max(1, (1 << 28) // p.nvt)
    for c in range(0, p.nr, step):
        h[c:c + step] += (coef[c:c + step] @ basis).to(dt)
    return h


def _kept(p, x):
    """Results that the interface gives as doubles, with the accuracy of the state."""
    return x if p.dtype == "f64" else x.float()


def prepare(case, seed):
    c = _full(case)
    kind = c["kind"]
    s = dict(kind=kind, steps=c["steps"])
    if kind == "batch":
        probs = _batch_problems(case, seed)
        b = binding.Batch(probs)
        h0 = [_state(p, seed + i) for i, p in enumerate(probs)]
        for i, h in enumerate(h0):
            b.set_state(i, h, step=0)
        b.tune(1)
        return dict(s, probs=probs, batch=b, h0=h0, n=0, begun=0)
    p = _problem(case, seed)
    s["p"] = p
    if kind == "collide":
        h = _state(p, seed)
        return dict(s, h=h, out=torch.empty_like(h), n=0,
                    mom=torch.empty((p.nr, 11), dtype=torch.float64, device="cuda"))
    cav = binding.Cavity(p)
    s["cav"] = cav
    if kind == "march":
        h0 = _state(p, seed)
        cav.set_state(h0, step=0)
        return dict(s, h0=h0, n=0, begun=0, out=torch.empty((p.nr, p.nvt), dtype=cav.torch_dtype, device="cuda"),
                    mom=torch.empty((p.nr, 11), dtype=torch.float64, device="cuda"))
    if kind == "adjoint":
        # Two stored states, visited in turn, and the cotangent of the last one.
        lam = 0.01 * _state(p, seed + 2)
        return dict(s, h=[_state(p, seed), _state(p, seed + 1)], lam=lam, out=torch.empty_like(lam),
                    n=1_000_000)
    lid = torch.from_numpy(p.lid_profile).cuda().float().requires_grad_()
    return dict(s, lid=lid, h0=_state(p, seed).requires_grad_(), cot=0.01 * _state(p, seed + 1), every=c["every"])


def _next_realisation(state):
    """Counts the steps of a pass; true when a new realisation begins before it."""
    new = state["n"] + state["steps"] - state["begun"] > _WINDOW
    if new:
        state["begun"] = state["n"]
    state["n"] += state["steps"]
    return new


def run(state):
    kind = state["kind"]
    if kind == "march":
        p, cav = state["p"], state["cav"]
        if _next_realisation(state):
            cav.set_state(state["h0"], step=state["begun"])
        cav.step(state["steps"])
        h, _ = cav.get_state(out=state["out"])
        return {"h": h, "moments": _kept(p, cav.moments(out=state["mom"]))}
    if kind == "batch":
        b, probs = state["batch"], state["probs"]
        if _next_realisation(state):
            for i, h in enumerate(state["h0"]):
                b.set_state(i, h, step=state["begun"])
        b.step(state["steps"])
        return {"h": [b.get_state(i)[0] for i in range(len(probs))],
                "moments": [_kept(p, b.moments(i)) for i, p in enumerate(probs)]}
    if kind == "collide":
        p = state["p"]
        binding.collide_noalloc(p, state["n"], state["h"], state["out"], state["mom"])
        state["n"] += 1
        return {"h": state["out"], "moments": _kept(p, state["mom"])}
    if kind == "adjoint":
        p, cav, n = state["p"], state["cav"], state["n"]
        grad = torch.zeros(p.nx, dtype=torch.float64, device="cuda")
        lam = state["lam"]
        for k in range(state["steps"]):
            lam = cav.adjoint_step(n - k, state["h"][k % 2], lam, state["out"], grad, wD=1.0 / state["steps"])
        state["n"] = n - state["steps"]
        return {"lam": lam, "grad_lid": _kept(p, grad)}
    h, d = autodiff.rollout(state["cav"], state["lid"], state["h0"], state["steps"], every=state["every"])
    g_lid, g_h0 = torch.autograd.grad((h, d), (state["lid"], state["h0"]),
                                      (state["cot"], torch.ones_like(d)))
    return {"h": h.detach(), "D": d.detach().float(), "grad_lid": g_lid, "grad_h0": g_h0}


def work(case):
    """Bytes and operations of one pass: per step the state is read and
    written once; per node the streaming and the moments of the correction,
    per cell and sample its product, weight and four additions."""
    c = _full(case)

    def one(p, steps):
        el = 8 if p.dtype == "f64" else 4
        return dict(bytes=steps * 2 * p.nodes * el + p.nr * 88.0, flops=steps * (p.nodes * 36.0 + p.nr * p.nt * 9.0))

    if c["kind"] == "batch":
        w = [one(p, c["steps"]) for p in _batch_problems(case, 0)]
        out = sum(p.nodes * 4.0 for p in _batch_problems(case, 0))
        return dict(bytes=sum(x["bytes"] for x in w) + 2 * out, flops=sum(x["flops"] for x in w))
    p = _problem(case, 0)
    el = 8 if p.dtype == "f64" else 4
    w = one(p, c["steps"])
    if c["kind"] == "march":
        w["bytes"] += 2.0 * p.nodes * el            # the state copied out
    elif c["kind"] == "adjoint":
        w = dict(bytes=c["steps"] * 3.0 * p.nodes * el, flops=2 * w["flops"])
    elif c["kind"] == "rollout":
        # Forward steps, the replayed ones, and the adjoint steps.
        w = dict(bytes=2 * w["bytes"] + c["steps"] * 3.0 * p.nodes * el, flops=4 * w["flops"])
    return w


# ---------------------------------------------------------------------------
# The same passes in 64 bits
# ---------------------------------------------------------------------------
def _mul_hi(a, b):
    return ((a >> 16) * b + (((a & 0xFFFF) * b) >> 16)) >> 16


def _philox(c, k0, k1):
    """Philox4x32-10 of Salmon et al. (SC'11) on int64 tensors holding 32-bit words."""
    m = 0xFFFFFFFF
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
        h0, l0 = _mul_hi(c[0], 0xD2511F53), (c[0] * 0xD2511F53) & m
        h1, l1 = _mul_hi(c[2], 0xCD9E8D57), (c[2] * 0xCD9E8D57) & m
        c = (h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0)
    return c


class _Exact:
    """One cavity in float64: the step of the method as PyTorch operations."""

    def __init__(self, p):
        self.p = p
        t = lambda x: torch.as_tensor(x, dtype=torch.float64, device="cuda")  # noqa: E731
        v, d, e = _nodes(p)
        self.v, self.e, self.dv = t(v), t(e), 2.0 * p.vmax / p.nv
        L = 1.0 / p.kn

        def widths(n, r, lid):
            if not (r > 0 and r != 1):
                return np.full(n, L / n)
            i = np.arange(n)
            w = (1.0 / r) ** (n - 1 - i if lid else np.minimum(i, n - 1 - i)).astype(float)
            return L * w / w.sum()

        dx, dy = widths(p.nx, p.rx, False), widths(p.ny, p.ry, True)
        self.dt = p.cfl * min(dx.min(), dy.min()) / v[-1]
        self.dx, self.dy = t(dx), t(dy)
        self.kcoll = 5.0 * 1.016034 / 16.0 * math.sqrt(2.0 / math.pi)
        self.cw = math.pi * self.kcoll * self.dt / p.nt
        base = np.full(p.nx, p.lid_u0) if p.lid_profile is None else p.lid_profile
        self.base = t(base)
        if p.eps > 0:
            self.eps = p.eps
        else:
            self.eps = float(np.abs(base).max() + (abs(p.lid_amp) if p.lid_period > 0 else 0.0)) or 1.0
        n = p.nv
        vx, vy, vz = (x.reshape(-1) for x in torch.meshgrid(self.v, self.v, self.v, indexing="ij"))
        self.vx, self.vy, self.vz = vx, vy, vz
        self.ax1 = t(d) * math.pi ** -0.5 * torch.exp(-self.v * self.v)
        self.w = (self.ax1[:, None, None] * self.ax1[:, None] * self.ax1).reshape(-1)
        self.d1 = t(d)
        self.psi = torch.stack([torch.ones_like(vx), vx, vy, vz, vx * vx + vy * vy + vz * vz])
        iu = [(a, b) for a in range(5) for b in range(a, 5)]
        self.iu = iu
        self.pp = torch.stack([self.psi[a] * self.psi[b] for a, b in iu])
        self.m2 = torch.stack([vx * vx, vy * vy, vz * vz, vx * vy, vx * vz, vy * vz])
        self.n = n

    # -- samples --------------------------------------------------------------
    def _axis(self, x):
        p = self.p
        if p.rv > 0 and p.rv != 1:
            k = torch.searchsorted(self.e, x.contiguous(), right=True) - 1
        else:
            k = torch.floor((x + p.vmax) / self.dv).to(torch.int64)
        return k, (k >= 0) & (k < p.nv)

    def samples(self, step, cells=None):
        """Node indices (4, ..., nt; -1 outside) and weights of the step's set(s)."""
        p = self.p
        l = torch.arange(p.nt, device="cuda", dtype=torch.int64)
        if cells is None:
            word = torch.full_like(l, 0xFFFFFFFF)
        else:
            word = cells[:, None].expand(-1, p.nt)
            l = l.expand_as(word)
        one = torch.ones_like(l)
        u = []
        for d in range(2):
            u += list(_philox((l, one * (step & 0xFFFFFFFF), word, one * d), p.seed, p.instance))
        u = [(x.to(torch.float64) + 0.5) / 4294967296.0 for x in u]
        r = [torch.sqrt(-torch.log(u[i])) for i in (0, 2, 4)]
        th = [2 * math.pi * u[i] for i in (1, 3, 5)]
        v = [r[0] * torch.cos(th[0]), r[0] * torch.sin(th[0]), r[1] * torch.cos(th[1])]
        v1 = [r[1] * torch.sin(th[1]), r[2] * torch.cos(th[2]), r[2] * torch.sin(th[2])]
        kz = 1.0 - 2.0 * u[6]
        st, ph = torch.sqrt(1.0 - kz * kz), 2 * math.pi * u[7]
        k = [st * torch.cos(ph), st * torch.sin(ph), kz]
        s = sum((b - a) * q for a, b, q in zip(v, v1, k))
        idx = []
        for w in (v, v1, [a + s * q for a, q in zip(v, k)], [b - s * q for b, q in zip(v1, k)]):
            j, ok = torch.zeros_like(l), torch.ones_like(l, dtype=torch.bool)
            for x in w:
                kk, inside = self._axis(x)
                j, ok = j * p.nv + kk, ok & inside
            idx.append(torch.where(ok, j, torch.full_like(j, -1)))
        return torch.stack(idx), self.cw * s.abs()

    # -- streaming with diffuse walls -------------------------------------------
    def lid(self, step):
        p = self.p
        if p.lid_period > 0:
            return self.base + p.lid_amp * math.sin(2 * math.pi * step * self.dt / p.lid_period)
        return self.base

    def _emitted(self, hb, axis, sign, U):
        """Ghost values (faces, n tangential) of a wall: hb (faces, n, n, n) the
        boundary cells, the inward normal sign * e_axis, U the faces' x speed."""
        v = self.v
        wn = torch.where(sign * v < 0, -sign * v * self.ax1, torch.zeros_like(v))
        f = hb.moveaxis(axis + 1, 1)
        out = torch.einsum("fabc,a,b,c->f", f, wn, self.ax1, self.ax1)
        cout = wn.sum() * self.ax1.sum() ** 2
        hn = torch.where(sign * v > 0, sign * v * self.ax1, torch.zeros_like(v)).sum()
        d = v[None, :] - U[:, None]
        tang = (self.d1 * math.pi ** -0.5 * torch.exp(-d * d)).sum(1)
        nw = (cout + self.eps * out) / (hn * tang * self.ax1.sum())
        return (nw[:, None] * torch.exp(2 * v[None, :] * U[:, None] - (U * U)[:, None]) - 1.0) / self.eps

    def ghosts(self, h, U):
        p, n = self.p, self.n
        g = h.view(p.ny, p.nx, n, n, n)
        z = torch.zeros(p.ny, dtype=torch.float64, device="cuda")
        zx = torch.zeros(p.nx, dtype=torch.float64, device="cuda")
        return (self._emitted(g[:, 0], 0, 1, z), self._emitted(g[:, -1], 0, -1, z),
                self._emitted(g[0], 1, 1, zx), self._emitted(g[-1], 1, -1, U))

    def stream(self, h, U):
        p, n = self.p, self.n
        left, right, bottom, top = self.ghosts(h, U)
        g = h.view(p.ny, p.nx, n, n, n)
        out = g.clone()
        neg, pos = int((self.v < 0).sum()), int((self.v <= 0).sum())
        ax = (self.v.abs()[None, :] * self.dt / self.dx[:, None])[None, :, :, None, None]
        ay = (self.v.abs()[None, :] * self.dt / self.dy[:, None])[:, None, None, :, None]

        def move(at, src, inner, outer, face, frac_in, frac_out):
            # out -= frac (g - upwind source), the wall's ghost values at the edge
            out[inner + at] -= frac_in * (g[inner + at] - g[src + at])
            out[outer + at] -= frac_out * (g[outer + at] - face)

        a, lo, hi = slice(None), slice(0, neg), slice(pos, n)
        # x direction: v_x > 0 from the left cell, v_x < 0 from the right one
        move((hi,), (a, slice(0, p.nx - 1)), (a, slice(1, p.nx)), (a, slice(0, 1)),
             left[:, None, None, :, None].expand(-1, 1, n - pos, -1, n), ax[:, 1:, hi], ax[:, :1, hi])
        move((lo,), (a, slice(1, p.nx)), (a, slice(0, p.nx - 1)), (a, slice(p.nx - 1, p.nx)),
             right[:, None, None, :, None].expand(-1, 1, neg, -1, n), ax[:, :-1, lo], ax[:, -1:, lo])
        # y direction: v_y > 0 from the cell below, v_y < 0 from the one above
        move((a, hi), (slice(0, p.ny - 1), a), (slice(1, p.ny), a), (slice(0, 1), a),
             bottom[None, :, :, None, None].expand(1, -1, -1, n - pos, n), ay[1:, :, :, hi], ay[:1, :, :, hi])
        move((a, lo), (slice(1, p.ny), a), (slice(0, p.ny - 1), a), (slice(p.ny - 1, p.ny), a),
             top[None, :, :, None, None].expand(1, -1, -1, neg, n), ay[:-1, :, :, lo], ay[-1:, :, :, lo])
        return out.view(p.nr, p.nvt)

    def shear(self, h, U):
        """Mean lid shear D of a state."""
        p, n = self.p, self.n
        top = self.ghosts(h, U)[3]
        g = h.view(p.ny, p.nx, n, n, n)[-1]
        up = torch.where(self.v > 0, self.v, torch.zeros_like(self.v)) * self.ax1
        dn = torch.where(self.v < 0, self.v, torch.zeros_like(self.v)) * self.ax1
        xs = self.v * self.ax1
        cell = torch.einsum("fabc,a,b,c->f", g, xs, up, self.ax1)
        wall = (top * xs).sum(1) * dn.sum() * self.ax1.sum()
        return (2.0 * (cell + wall) * self.dx).sum() * p.kn

    # -- relaxation -----------------------------------------------------------
    def _solve(self, h, dn):
        """h_c and its corrected value from h~ and the collision sum dn (cells, nodes)."""
        hc = h + dn / self.w
        G = (self.w * (1.0 + self.eps * hc)) @ self.pp.T
        M = torch.zeros((h.shape[0], 5, 5), dtype=torch.float64, device="cuda")
        for q, (a, b) in enumerate(self.iu):
            M[:, a, b] = G[:, q]
            M[:, b, a] = G[:, q]
        rhs = -(dn @ self.psi.T)
        mu = torch.linalg.solve(M, rhs)
        return hc + (1.0 + self.eps * hc) * (mu @ self.psi)

    def collide(self, ht, step, in_place=False):
        p = self.p
        out = ht if in_place else torch.empty_like(ht)
        parts = []
        width = max(1, (1 << 27) // max(p.nvt, p.nt)) if not p.per_cell else max(1, (1 << 23) // p.nt)
        if not p.per_cell:
            idx, W = self.samples(step)
            safe = idx.clamp_min(0)
            keep = (idx >= 0).to(torch.float64)
        for c in range(0, p.nr, width):
            h = ht[c:c + width]
            if p.per_cell:
                idx, W = self.samples(step, torch.arange(c, min(p.nr, c + width), device="cuda"))
                safe, keep = idx.clamp_min(0), (idx >= 0).to(torch.float64)
                a, b = (h.gather(1, safe[q]) * keep[q] for q in (0, 1))
                r = W * (a + b + self.eps * a * b)
                dn = torch.zeros_like(h)
                for q in range(4):
                    dn.scatter_add_(1, safe[q], (r if q > 1 else -r) * keep[q])
            else:
                x = h.t().contiguous()
                a, b = (x[safe[q]] * keep[q][:, None] for q in (0, 1))
                r = W[:, None] * (a + b + self.eps * a * b)
                del a, b
                dn = torch.zeros_like(x)
                for q in range(4):
                    dn = dn.index_add(0, safe[q], r * ((1.0 if q > 1 else -1.0) * keep[q])[:, None])
                dn = dn.t()
            new = self._solve(h, dn)
            if torch.is_grad_enabled() and new.requires_grad:
                parts.append(new)
            else:
                out[c:c + width] = new
        return torch.cat(parts) if parts else out

    def step(self, h, n, U=None):
        return self.collide(self.stream(h, self.lid(n) if U is None else U), n, in_place=not torch.is_grad_enabled())

    def moments(self, h):
        e, rows = self.eps, []
        width = max(1, (1 << 27) // self.p.nvt)
        for c in range(0, self.p.nr, width):
            wh = h[c:c + width] * self.w
            rho = wh.sum(1)
            n = 1.0 + e * rho
            u = (wh @ self.psi[1:4].T) / n[:, None]
            m = wh @ self.m2.T
            th = ((2.0 / 3.0) * m[:, :3].sum(1) - rho) / n - (2.0 * e / 3.0) * (u * u).sum(1)
            uu = torch.stack([u[:, a] * u[:, b] for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))], 1)
            rows.append(torch.cat([rho[:, None], u, th[:, None], 2.0 * m - 2.0 * e * n[:, None] * uu], 1))
        return torch.cat(rows)


def _stored(x):
    return x.detach().double()


def exact(case, seed):
    c = _full(case)
    kind, steps = c["kind"], c["steps"]
    if kind == "batch":
        hs, ms = [], []
        for i, p in enumerate(_batch_problems(case, seed)):
            with torch.no_grad():
                e, h = _Exact(p), _stored(_state(p, seed + i))
                for n in range(steps):
                    h = e.step(h, n)
                hs.append(h)
                ms.append(e.moments(h))
        return {"h": hs, "moments": ms}
    p = _problem(case, seed)
    e = _Exact(p)
    if kind in ("march", "collide"):
        with torch.no_grad():
            h = _stored(_state(p, seed))
            for n in range(steps):
                h = e.step(h, n) if kind == "march" else e.collide(h, n)
            return {"h": h, "moments": e.moments(h)}
    if kind == "adjoint":
        hs = [_stored(_state(p, seed)), _stored(_state(p, seed + 1))]
        lam = _stored(0.01 * _state(p, seed + 2))
        grad = torch.zeros(p.nx, dtype=torch.float64, device="cuda")
        for k in range(steps):
            with torch.enable_grad():
                h, U = hs[k % 2].clone().requires_grad_(), e.base.clone().requires_grad_()
                out, D = e.step(h, 1_000_000 - k, U), e.shear(h, U)
                lam, g = torch.autograd.grad((out, D), (h, U), (lam, torch.full_like(D, 1.0 / steps)))
            grad += g
        return {"lam": lam, "grad_lid": grad}
    with torch.enable_grad():
        # The handle's eps is that of its problem; the lid speeds are the FP32 ones.
        U = torch.from_numpy(p.lid_profile).cuda().float().double().requires_grad_()
        h0 = _stored(_state(p, seed)).requires_grad_()
        h, D = h0, 0.0
        for n in range(steps):
            D = D + e.shear(h, U) / steps
            h = e.step(h, n, U)
        g_lid, g_h0 = torch.autograd.grad((h, D), (U, h0), (_stored(0.01 * _state(p, seed + 1)), torch.ones_like(D)))
    return {"h": h.detach(), "D": D.detach(), "grad_lid": g_lid, "grad_h0": g_h0}
