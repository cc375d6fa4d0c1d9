"""What a user of this library has it do, as cases that can be timed and checked.

A case is one call pattern of the public entry points (``native.Domain``,
``native.Batch``): a number of coarse steps, then the results a program reads
at that point -- the force history of the steps, and for the runs whose field
is looked at a snapshot of the levels that a dense array can hold.  Results
are returned in the precision the populations are stored in (what such a
program keeps or writes out).

  one_step_D10      a coupled loop: one coarse step of a small refined
                    cylinder, then its forces (the smallest call)
  tgv_128_f64       the Taylor-Green validation run, FP64, with its field
  cylinder_D40_f32  the refined cylinder of the benchmark, forces and field
  wing_c64_f32      the flapping ellipse: a moving body whose refinement follows
  naca_c64_f16      a pitching section with an inflow, 16-bit storage
  table1_D128_f32   the paper's cylinder study: four levels, a large level 0
  cavity_solid_f32  the lid-driven cavity, its cylinder by bounce-back
  cavity_ibm_f32    the same with the cylinder as an immersed body
  sweep_4096_f32    a large uniform grid, beyond the L2 cache
  sweep_4096_bf16   the same in 16-bit storage
  les_2960_f32      a ragged large grid with the LES collision
  batch64_bf16      64 uneven instances stepped together, every force history
                    read and the coarse field of the one that is watched
"""
from __future__ import annotations

import math
from dataclasses import replace

import numpy as np
import torch

from paper_2402_04606_gb300 import native
from paper_2402_04606_gb300 import workloads as wl

STORAGE = {"f64": wl.F64, "f32": wl.F32, "f16": wl.F16DEV, "bf16": wl.BF16DEV}
BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
RESULT = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
# arithmetic of one cell update: moments, equilibrium and relaxation (with the
# moment transforms of MRT, or the stress and eddy viscosity of LES)
FLOPS = {"bgk": 100, "mrt": 130, "les": 125}


def listed():
    return [
        dict(name="one_step_D10", kind="cylinder", size=10, levels=3, block=8, storage="f32", coll="bgk", steps=1,
             snapshot=0),
        dict(name="tgv_128_f64", kind="sweep", nx=128, ny=128, block=16, storage="f64", coll="bgk", steps=1000,
             snapshot=1),
        dict(name="cylinder_D40_f32", kind="cylinder", size=40, levels=3, block=16, storage="f32", coll="bgk",
             steps=500, snapshot=3),
        dict(name="wing_c64_f32", kind="wing", size=64, levels=4, block=16, storage="f32", coll="bgk", steps=200,
             chords=50, snapshot=1),
        dict(name="naca_c64_f16", kind="naca", size=64, levels=3, block=16, storage="f16", coll="bgk", steps=500,
             snapshot=1),
        dict(name="table1_D128_f32", kind="table1", size=128, levels=4, block=16, storage="f32", coll="bgk", steps=200,
             snapshot=1),
        dict(name="cavity_solid_f32", kind="cavity", size=304, mode="bounce", block=16, storage="f32", coll="bgk",
             steps=1000, snapshot=1),
        dict(name="cavity_ibm_f32", kind="cavity", size=304, mode="ibm", block=16, storage="f32", coll="bgk",
             steps=1000, snapshot=1),
        dict(name="sweep_4096_f32", kind="sweep", nx=4096, ny=4096, block=16, storage="f32", coll="bgk", steps=1000,
             snapshot=1),
        dict(name="sweep_4096_bf16", kind="sweep", nx=4096, ny=4096, block=16, storage="bf16", coll="bgk", steps=1000,
             snapshot=1),
        dict(name="les_2960_f32", kind="sweep", nx=2960, ny=1488, block=16, storage="f32", coll="les", steps=1000,
             snapshot=1),
        dict(name="batch64_bf16", kind="batch", instances=64, scale=1.0, block=16, storage="bf16", coll="bgk",
             steps=32, snapshot=1),
    ]


def draw(rng):
    """One more case: the kind first, then sizes over the range the listed ones span."""
    for _ in range(1000):
        c = _draw(rng)
        if _valid(c):
            return c
    raise RuntimeError("no case drawn")


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw(rng):
    kind = rng.choice(["cylinder", "cylinder", "wing", "plate", "naca", "cavity", "sweep", "sweep", "sweep", "batch"])
    coll = rng.choice(["bgk", "bgk", "mrt", "les"])
    storage = rng.choice(["f32", "f32", "f32", "f64", "f16", "bf16"])
    if kind == "sweep":
        block = rng.choice([8, 16, 16, 32])
        nx = max(block, int(_log(rng, 48, 4096)) // block * block)
        ny = max(block, int(_log(rng, 48, 4096)) // block * block)
        # about as many cell updates as the listed grids take, fewer in FP64
        most = (2.0e9 if storage == "f64" else 1.2e10) / (nx * ny)
        steps = max(1, min(int(_log(rng, 10, 2000)), int(most)))
        return dict(kind=kind, nx=nx, ny=ny, block=block, storage=storage, coll=coll, steps=steps, snapshot=1)
    steps = int(_log(rng, 1, 300))
    if kind == "cylinder":
        size, levels = int(_log(rng, 10, 64)), rng.choice([1, 2, 3])
        return dict(kind=kind, size=size, levels=levels, block=8 if size < 24 else rng.choice([8, 16]),
                    storage=storage, coll=coll, steps=steps, snapshot=rng.choice([0, levels]))
    if kind == "wing":
        return dict(kind=kind, size=int(_log(rng, 24, 72)), levels=rng.choice([3, 4]), block=16, storage=storage,
                    coll=coll, steps=steps, chords=rng.choice([20, 30, 50]), snapshot=rng.choice([0, 1]))
    if kind in ("plate", "naca"):
        return dict(kind=kind, size=int(_log(rng, 24, 72)), levels=rng.choice([2, 3]), block=16, storage=storage,
                    coll=coll, steps=steps, snapshot=rng.choice([0, 1]))
    if kind == "cavity":
        return dict(kind=kind, size=max(64, int(_log(rng, 64, 768)) // 16 * 16), mode=rng.choice(["bounce", "ibm"]),
                    block=16, storage=storage, coll=coll, steps=int(_log(rng, 10, 1000)), snapshot=1)
    return dict(kind=kind, instances=int(_log(rng, 4, 48)), scale=1.0, block=16,
                storage=rng.choice(["f32", "f16", "bf16"]), coll=rng.choice(["bgk", "mrt"]),
                steps=int(_log(rng, 1, 24)), snapshot=1)


def _valid(c):
    """a refinement that stays clear of the sides, a body that fits one thread block's memory, FP64 work in bounds"""
    if c["kind"] in ("sweep", "batch"):
        return True
    spec = _specs(c, 0)[0]
    states = _plan(spec, _boxes(spec))
    if states is None:
        return False
    if c["storage"] == "f64" and (_updates(spec, states) * c["steps"] > 2.0e9):
        return False
    return not (c["kind"] == "cavity" and c["mode"] == "ibm" and spec.body.a > (40 if c["storage"] == "f64" else 64))


def _collision(spec, coll):
    return wl.with_mrt(spec) if coll == "mrt" else wl.with_les(spec) if coll == "les" else spec


def _specs(c, seed):
    """The case's domains; the seed gives the physical parameters a study varies."""
    rng = np.random.default_rng([7, seed])
    st, kind = STORAGE[c["storage"]], c["kind"]
    if kind == "sweep":
        spec = wl.DomainSpec(name="sweep", nx0=c["nx"], ny0=c["ny"], levels=1, block=c["block"],
                             tau_finest=float(rng.uniform(0.53, 0.8)), storage=st)
    elif kind == "cylinder":
        spec = wl.cylinder(D=c["size"], levels=c["levels"], re=float(rng.uniform(60, 180)), storage=st,
                           block=c["block"], n_markers=int(round(math.pi * c["size"])))
    elif kind == "table1":
        spec = wl.cylinder_table1(D=c["size"], levels=c["levels"], re=float(rng.uniform(100, 550)), storage=st)
    elif kind == "wing":
        spec = wl.wing(c=c["size"], levels=c["levels"], re=float(rng.uniform(100, 200)),
                       amp_deg=float(rng.uniform(30, 60)), storage=st, domain_chords=c["chords"],
                       n_markers=int(round(3.125 * c["size"])))
    elif kind == "plate":
        spec = wl.pitch_up(c=c["size"], levels=c["levels"], re=float(rng.uniform(500, 1000)), storage=st)
    elif kind == "naca":
        spec = wl.pitching_airfoil(c=c["size"], levels=c["levels"], re=float(rng.uniform(500, 1000)),
                                   amp_deg=float(rng.uniform(32, 64)), storage=st)
    elif kind == "cavity":
        spec = wl.cavity(L=c["size"], re=float(rng.uniform(100, 1000)), mode=c["mode"], storage=st)
    else:
        specs = wl.batch(c["instances"], seed=0, storage=st, block=c["block"], scale=c["scale"])
        out = []
        for s in specs:  # the mix of the serving loop, each run with its own parameters
            re = float(rng.uniform(50.0, 400.0))
            s = replace(s, tau_finest=wl.tau_from_re(s.body.u_ref, s.body.l_ref, re))
            if s.body.motion != 0:
                s.body.alpha_amp = math.radians(float(rng.uniform(16.0, 64.0)))
            out.append(_collision(s, c["coll"]))
        return out
    return [_collision(spec, c["coll"])]


def _initial(c, seed):
    """rho, ux, uy of a uniform grid: a vortex with smooth disturbances, periodic (sums of products of one
    cosine in x and one in y)"""
    rng = np.random.default_rng([11, seed])
    x, y = 2 * np.pi * np.arange(c["nx"]) / c["nx"], 2 * np.pi * np.arange(c["ny"]) / c["ny"]
    out = []
    for base, amp in ((1.0, 2e-4), (0.0, 0.02), (0.0, 0.02)):
        f = np.full((c["ny"], c["nx"]), base)
        for _ in range(3):
            kx, ky = rng.integers(1, 5, size=2)
            px, py = rng.uniform(0, 2 * np.pi, size=2)
            f += np.outer(amp * rng.uniform(0.3, 1.0) * np.cos(ky * y + py), np.cos(kx * x + px))
        out.append(f)
    return out


def prepare(case, seed):
    specs = _specs(case, seed)
    if case["kind"] == "batch":
        b = native.Batch(len(specs), block=case["block"], storage=STORAGE[case["storage"]])
        return dict(case=case, batch=b, members=[b.admit(s) for s in specs])
    d = native.Domain(specs[0])
    if case["kind"] == "sweep":
        d.set_fields(0, *_initial(case, seed))
    return dict(case=case, domain=d, body=specs[0].body is not None)


def run(state):
    c = state["case"]
    kept = RESULT[c["storage"]]
    if c["kind"] == "batch":
        state["batch"].step(c["steps"])
        out = {"forces": torch.from_numpy(np.concatenate([m.forces() for m in state["members"]])).to(kept)}
        seen = state["members"][0]
    else:
        seen, out = state["domain"], {}
        seen.step(c["steps"])
        if state["body"]:
            out["forces"] = torch.from_numpy(seen.forces()).to(kept)
    for level in range(c["snapshot"]):
        rho, ux, uy = seen.fields(level)
        out[f"rho{level}"] = torch.from_numpy(rho).to(kept)
        out[f"u{level}"] = torch.stack([torch.from_numpy(ux).to(kept), torch.from_numpy(uy).to(kept)])
    return out


def work(case):
    """The populations of every cell read once and written once in a pass, and the results; the arithmetic of
    its cell updates."""
    s, updates, n_bytes = BYTES[case["storage"]], 0, 0
    specs = _specs(case, 0)
    for spec in specs:
        states = _plan(spec, _boxes(spec))
        updates += _updates(spec, states) * case["steps"]
        n_bytes += 18 * s * sum(int((b == 1).sum()) for b in states) * spec.block**2
        if spec.body is not None:
            n_bytes += 24 * case["steps"] << (spec.levels - 1)
    n_bytes += sum(24 * specs[0].nx0 * specs[0].ny0 << (2 * l) for l in range(case["snapshot"]))
    return {"bytes": n_bytes, "flops": updates * FLOPS[case["coll"]]}


# ---------------------------------------------------------------------------
# the refinement, planned again from the specification
# ---------------------------------------------------------------------------
def _outline(b):
    """points of the body's outline at its first pose"""
    t = 2 * np.pi * np.arange(256) / 256
    if b.kind in (0, 1):
        p = np.stack([b.a * np.cos(t), (b.a if b.kind == 0 else b.b) * np.sin(t)], 1)
    elif b.kind == 2:
        p = np.array([(b.a, b.b), (-b.a, b.b), (-b.a, -b.b), (b.a, -b.b)])
    else:
        u = 0.5 * (1 + np.cos(t))
        h = 10 * b.b * (0.2969 * np.sqrt(u) - 0.1260 * u - 0.3516 * u**2 + 0.2843 * u**3 - 0.1036 * u**4)
        p = np.stack([b.a * np.cos(t), np.sign(np.sin(t)) * h], 1)
    p = p - np.asarray(b.pivot)
    al = b.alpha_mean
    x0 = np.asarray(b.x0) + (0.5 * b.heave_amp * np.array([math.cos(b.beta), math.sin(b.beta)]) if b.motion == 2 else 0)
    r = np.array([[math.cos(al), -math.sin(al)], [math.sin(al), math.cos(al)]])
    return p @ r.T + np.asarray(b.pivot) + x0


def _boxes(spec):
    boxes = list(spec.boxes)
    if spec.body is not None:
        p = _outline(spec.body)
        (x0, y0), (x1, y1) = p.min(0), p.max(0)
        for l in range(1, spec.levels):
            g = spec.margin[l]
            if g > 0:
                boxes.append((l, x0 - g, y0 - g, x1 + g + spec.wake[l], y1 + g))
    return boxes


def _plan(spec, boxes):
    """Block states per level (0 absent, 1 leaf, 2 refined) for these boxes, 2:1 balanced; None when a refined block
    touches a non-periodic side."""
    m, B = spec.levels, spec.block
    st = [np.zeros(((spec.ny0 << l) // B, (spec.nx0 << l) // B), np.int8) for l in range(m)]
    st[0][:] = 1
    px, py = spec.bc[0] == wl.BC_PERIODIC, spec.bc[2] == wl.BC_PERIODIC

    def split(l, j, i):
        st[l][j, i] = 2
        st[l + 1][2 * j:2 * j + 2, 2 * i:2 * i + 2] = 1

    for l in range(m - 1):
        side = B * 2.0 ** (m - 1 - l)
        for lv, x0, y0, x1, y1 in boxes:
            if lv <= l:
                continue
            for j in range(max(0, math.floor(y0 / side)), min(st[l].shape[0], math.ceil(y1 / side))):
                for i in range(max(0, math.floor(x0 / side)), min(st[l].shape[1], math.ceil(x1 / side))):
                    if st[l][j, i] == 1:
                        split(l, j, i)
    again = m > 2
    while again:
        again = False
        for l in range(m - 2):
            fine = np.pad(st[l + 1] == 2, 1)
            if px:
                fine[:, 0], fine[:, -1] = fine[:, -2], fine[:, 1]
            if py:
                fine[0], fine[-1] = fine[-2], fine[1]
            for j, i in np.argwhere(st[l] == 1):
                if fine[2 * j:2 * j + 4, 2 * i:2 * i + 4].any():
                    split(l, j, i)
                    again = True
    for l in range(1, m):
        s = st[l] != 0
        if (not px and (s[:, 0].any() or s[:, -1].any())) or (not py and (s[0].any() or s[-1].any())):
            return None
    return st


def _updates(spec, states):
    return sum(int((s == 1).sum()) * spec.block**2 << l for l, s in enumerate(states))


# ---------------------------------------------------------------------------
# the same results in 64 bits: dense arrays per level, plain torch
# ---------------------------------------------------------------------------
CX = [0, 1, 0, -1, 0, 1, -1, -1, 1]
CY = [0, 0, 1, 0, -1, 1, 1, -1, -1]
OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]
FLIP_Y = [0, 1, 4, 3, 2, 8, 7, 6, 5]
W9 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4


def exact(case, seed):
    # moving bodies: their refinement is planned again every step and their dense finest level has over ten
    # million cells; the batch and the paper's cylinder study have dense finest levels of over a hundred million:
    # each takes well over 20 seconds
    if case["kind"] in ("wing", "plate", "naca", "table1", "batch"):
        return None
    spec = _specs(case, seed)[0]
    cells = sum((spec.nx0 * spec.ny0 << (2 * l)) << l for l in range(spec.levels))
    if case["steps"] * (cells / 2.0e9 + 0.004 * (2**spec.levels - 1)) > 20:  # seconds, about
        return None
    ref = _Dense(spec)
    if case["kind"] == "sweep":
        ref.start(_initial(case, seed))
    else:
        ref.start(None)
    for _ in range(case["steps"]):
        ref.step(0)
    out = {}
    if spec.body is not None:
        out["forces"] = torch.stack(ref.forces[:case["steps"] << (spec.levels - 1)])
    for level in range(case["snapshot"]):
        rho, ux, uy = ref.fields(level)
        out[f"rho{level}"], out[f"u{level}"] = rho, torch.stack([ux, uy])
    return out


class _Dense:
    def __init__(self, spec):
        self.s = spec
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        t = lambda v: torch.tensor(v, dtype=torch.float64, device=self.dev)  # noqa: E731
        self.cx, self.cy, self.w = (t(v).view(9, 1, 1) for v in (CX, CY, W9))
        self.tau = [0.5 + (spec.tau_finest - 0.5) / 2 ** (spec.levels - 1 - l) for l in range(spec.levels)]
        self.periodic = spec.bc[0] == wl.BC_PERIODIC
        states, B, m = _plan(spec, _boxes(spec)), spec.block, spec.levels
        up = lambda a: torch.from_numpy(np.kron(a, np.ones((B, B), np.uint8)) != 0).to(self.dev)  # noqa: E731
        self.leaf = [up((s == 1).astype(np.uint8)) for s in states]
        refined = [up((s == 2).astype(np.uint8)) for s in states]
        self.live, self.from_fine = [], []
        for l in range(m):
            grown = torch.nn.functional.max_pool2d(self.leaf[l][None].float(), 5, 1, 2)[0] > 0
            outside = up((states[l] == 0).astype(np.uint8))
            self.live.append(self.leaf[l] | (grown & outside))  # interior and the two halo layers
            self.from_fine.append(torch.stack([self.leaf[l] & self._shift(refined[l], q) for q in range(9)])
                                  if l + 1 < m else None)
        # a population whose source is neither interior nor halo stays where it is (the halo's outer layer)
        self.pulls = [torch.stack([self._shift(self.live[l], q) for q in range(9)]) for l in range(m)]
        self.forces = []
        if spec.body is not None:
            self._markers()
        if spec.collision == 1:
            e = -4 + 3 * (self.cx**2 + self.cy**2)
            c2 = self.cx**2 + self.cy**2
            rows = [torch.ones_like(c2), e, 4 - 10.5 * c2 + 4.5 * c2**2, self.cx, (-5 + 3 * c2) * self.cx, self.cy,
                    (-5 + 3 * c2) * self.cy, self.cx**2 - self.cy**2, self.cx * self.cy]
            self.M = torch.stack([r.view(9) for r in rows])
            self.Minv = torch.linalg.inv(self.M)
        if spec.solid[0]:
            self._solid()

    @staticmethod
    def _shift(a, q):
        return torch.roll(a, (CY[q], CX[q]), (-2, -1))

    def feq(self, rho, ux, uy):
        cu = self.cx * ux + self.cy * uy
        return self.w * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (ux * ux + uy * uy))

    def start(self, fields):
        s = self.s
        self.pre, self.f = [], []
        for l in range(s.levels):
            shape = (s.ny0 << l, s.nx0 << l)
            if fields is None:
                fields_l = [torch.full(shape, v, dtype=torch.float64, device=self.dev)
                            for v in (s.rho0, s.u_in[0], s.u_in[1])]
            else:
                fields_l = [torch.from_numpy(v).to(self.dev) for v in fields]
            self.pre.append(self.feq(*fields_l))
        for l in range(s.levels):
            force = self._ibm(self.pre[l]) if s.body is not None and l == s.levels - 1 else None
            self.f.append(self._collide(l, self.pre[l], force))

    def step(self, l):
        s, last = self.s, self.s.levels - 1
        if l < last:
            up = self.f[l].repeat_interleave(2, 1).repeat_interleave(2, 2)
            halo = self.live[l + 1] & ~self.leaf[l + 1]
            self.f[l + 1] = torch.where(halo, up, self.f[l + 1])
            self.step(l + 1)
            self.step(l + 1)
        f = self.f[l]
        new = self._stream(f) if l == 0 else torch.stack([self._shift(f[q], q) for q in range(9)])
        if s.levels > 1:
            new = torch.where(self.pulls[l], new, f) if l > 0 else new
            if l < last:
                new = torch.where(self.from_fine[l], torch.nn.functional.avg_pool2d(self.f[l + 1][None], 2)[0], new)
        if s.solid[0]:
            new = self._bounce(f, new)
        self.pre[l] = new
        force = self._ibm(new) if s.body is not None and l == last else None
        post = self._collide(l, new, force)
        if s.solid[0]:  # solid cells are never updated
            self.f[l] = torch.where(self.fluid, post, f)
        else:
            self.f[l] = torch.where(self.leaf[l], post, new) if s.levels > 1 else post

    def _stream(self, f):
        s = self.s
        if self.periodic:
            return torch.stack([self._shift(f[q], q) for q in range(9)])
        ny, nx = f.shape[1:]
        g = torch.nn.functional.pad(f[None], (1, 1, 1, 1), mode="replicate")[0]
        if s.bc[2] == wl.BC_SYMMETRY:
            g[:, 0] = g[FLIP_Y, 1]
            g[:, -1] = g[FLIP_Y, -2]
        new = torch.stack([g[q, 1 - CY[q]:1 - CY[q] + ny, 1 - CX[q]:1 - CX[q] + nx] for q in range(9)])
        if s.bc[0] == wl.BC_WALL:
            for q in range(1, 9):
                gain = [6 * W9[q] * s.rho0 * (CX[q] * s.uwall[2 * k] + CY[q] * s.uwall[2 * k + 1]) for k in range(4)]
                if CX[q]:
                    i, k = (0, 0) if CX[q] > 0 else (nx - 1, 1)
                    new[q, :, i] = f[OPP[q], :, i] + gain[k]
                if CY[q]:
                    j, k = (0, 2) if CY[q] > 0 else (ny - 1, 3)
                    new[q, j] = f[OPP[q], j] + gain[k]
        if s.bc[0] == wl.BC_INLET:
            new[:, :, 0] = self.feq(s.rho0, s.u_in[0], s.u_in[1])[:, :, 0]
        return new

    def _solid(self):
        s = self.s
        _, cx, cy, r = s.solid
        y = torch.arange(s.ny0, dtype=torch.float64, device=self.dev).view(-1, 1) + 0.5
        x = torch.arange(s.nx0, dtype=torch.float64, device=self.dev).view(1, -1) + 0.5
        inside = lambda px, py: (px - cx) ** 2 + (py - cy) ** 2 < r * r  # noqa: E731
        self.fluid = ~inside(x, y)
        self.links = []
        for q in range(1, 9):
            hit = self.fluid & inside(x - CX[q], y - CY[q])
            j, i = torch.nonzero(hit, as_tuple=True)
            px, py = i + 0.5 - cx, j + 0.5 - cy
            a, b = CX[q] ** 2 + CY[q] ** 2, -(px * CX[q] + py * CY[q])
            t = (-b - torch.sqrt(b * b - a * (px * px + py * py - r * r))) / a
            near = (t < 0.5) & ~inside(i + 0.5 + CX[q], j + 0.5 + CY[q])
            self.links.append((q, j, i, t, near))

    def _bounce(self, f, new):
        out = new.clone()
        for q, j, i, t, near in self.links:
            a, b, g = f[OPP[q], j, i], f[q, j, i], new[OPP[q], j, i]
            out[q, j, i] = torch.where(near, 2 * t * a + (1 - 2 * t) * g, a / (2 * t) + (1 - 1 / (2 * t)) * b)
        return out

    def _collide(self, l, f, force):
        s, om = self.s, 1 / self.tau[l]
        rho = f.sum(0)
        ux, uy = (f * self.cx).sum(0), (f * self.cy).sum(0)
        fx = fy = None
        if force is not None:
            fx, fy = force
            ux, uy = ux + 0.5 * fx, uy + 0.5 * fy
        ux, uy = ux / rho, uy / rho
        eq = self.feq(rho, ux, uy)
        guo = 0.0
        if force is not None:
            cu = self.cx * ux + self.cy * uy
            guo = self.w * ((3 * (self.cx - ux) + 9 * cu * self.cx) * fx + (3 * (self.cy - uy) + 9 * cu * self.cy) * fy)
        if s.collision == 1:
            se, sp, sq = s.mrt_rates
            rates = torch.tensor([0, se, sp, 0, sq, 0, sq, om, om], dtype=torch.float64, device=self.dev)
            relax = self.Minv @ torch.diag(rates) @ self.M
            out = f - torch.einsum("ij,jyx->iyx", relax, f - eq)
            if force is not None:
                half = torch.eye(9, dtype=torch.float64, device=self.dev) - 0.5 * relax
                out = out + torch.einsum("ij,jyx->iyx", half, guo)
            return out
        if s.collision == 2:
            ne = f - eq
            pxx, pyy, pxy = ((ne * c).sum(0) for c in (self.cx**2, self.cy**2, self.cx * self.cy))
            stress = torch.sqrt(2 * (pxx * pxx + pyy * pyy + 2 * pxy * pxy))
            om = 2 / (self.tau[l] + torch.sqrt(self.tau[l] ** 2 + 18 * s.les_cs**2 * stress / rho))
        return f + om * (eq - f) + (1 - 0.5 * om) * guo

    def _markers(self):
        s, b = self.s, self.s.body  # a static circle: markers at equal angles
        t = 2 * np.pi * np.arange(b.n_markers) / b.n_markers
        x, y = b.x0[0] + b.a * np.cos(t), b.x0[1] + b.a * np.sin(t)

        def phi(r):
            r = np.abs(r)
            one = 0.125 * (3 - 2 * r + np.sqrt(np.maximum(0, 1 + 4 * r - 4 * r * r)))
            two = 0.125 * (5 - 2 * r - np.sqrt(np.maximum(0, -7 + 12 * r - 4 * r * r)))
            return np.where(r <= 1, one, np.where(r <= 2, two, 0.0))

        nx = s.nx0 << (s.levels - 1)
        i0, j0 = np.floor(x - 0.5).astype(int) - 1, np.floor(y - 0.5).astype(int) - 1
        k = np.arange(4)
        gx, gy = i0[:, None] + k, j0[:, None] + k
        wt = phi(gy + 0.5 - y[:, None])[:, :, None] * phi(gx + 0.5 - x[:, None])[:, None, :]
        cell = gy[:, :, None] * nx + gx[:, None, :]
        self.cells, at = np.unique(cell.ravel(), return_inverse=True)
        spread = np.zeros((b.n_markers, len(self.cells)))
        np.add.at(spread, (np.repeat(np.arange(b.n_markers), 16), at.ravel()), wt.ravel())
        dev = lambda v: torch.from_numpy(v).to(self.dev)  # noqa: E731
        self.cells, self.spread = dev(self.cells), dev(spread)
        self.arm = dev(np.stack([b.a * np.cos(t), b.a * np.sin(t)], 1))
        self.ds = 2 * np.pi * b.a / b.n_markers

    def _ibm(self, pre):
        p = pre.reshape(9, -1)[:, self.cells]
        rho = p.sum(0)
        u = torch.stack([(p * self.cx.view(9, 1)).sum(0), (p * self.cy.view(9, 1)).sum(0)], 1) / rho[:, None]
        rho_m = (self.spread @ rho)[:, None]
        total, field = torch.zeros_like(self.arm), torch.zeros_like(u)
        for _ in range(self.s.body.K):
            d = -2 * rho_m * (self.spread @ u)
            total = total + d
            g = self.spread.T @ d * self.ds
            field = field + g
            u = u + g / (2 * rho[:, None])
        out = torch.zeros((2,) + pre.shape[1:], dtype=torch.float64, device=self.dev)
        out.view(2, -1)[:, self.cells] = field.T
        moment = (self.arm[:, 0] * total[:, 1] - self.arm[:, 1] * total[:, 0]).sum()
        self.forces.append(-self.ds * torch.stack([total[:, 0].sum(), total[:, 1].sum(), moment]))
        return out

    def fields(self, l):
        f, keep = self.pre[l], self.leaf[l]
        rho = f.sum(0)
        ux, uy = (f * self.cx).sum(0) / rho, (f * self.cy).sum(0) / rho
        return [torch.where(keep, v, torch.zeros_like(v)) for v in (rho, ux, uy)]
