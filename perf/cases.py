"""The work this library is timed on: whole time steps of single cases and of batches in each
precision, the pressure solve alone, the vortex diagnostic, the step's vector-Jacobian product and
the allocation-free residual, each through the binding's public calls.

A step case is what a program does with a case between two looks at it: put a flow state into the
case (``Case.write_flat``, pinned host memory), advance it (``Case.step`` or ``Batch.step``), take
the state back (``Case.read_flat``).  The flow states are seeded: the workload's base flow with
smooth large-scale modes and the +-1 % cell noise the channel workloads start from.  ``geometry``
is the seed of the workload generators in ``cases.py`` (vents, boxes, batch sizes): it belongs to
the case, the flow state to the seed of ``prepare``.

``exact`` restates the method in plain 64-bit torch (``Reference``), with the pressure solved by
conjugate gradients far below the solver's tolerance.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2603_21869_gb300 import binding, cases

FIELDS = cases.FIELDS                       # u v w p T k omega
PRECISION = {"f64": cases.FP64, "f32": cases.FP32, "bf16": cases.BF16_MIXED}
EXACT_CELL_STEPS = 12e6                     # 64-bit torch steps beyond this take too long


def listed():
    return [
        # the plain 2D channel (128 x 32, FP64): 4096 cells, every launch is latency
        dict(name="channel2d_128x32_f64", kind="step", family="channel2d", nx=128, ny=32, nz=1, levels=5,
             precision="f64", steps=20, pre=3, post=3, inner=0, krylov=0, smoother=0, geometry=0),
        # a small ragged room as the served stream admits it, stepped alone: under 2^20 cells
        dict(name="room_112x80x48_bf16", kind="step", family="room", nx=112, ny=80, nz=48, levels=4,
             precision="bf16", steps=10, pre=2, post=2, inner=2, krylov=1, smoother=0, geometry=3),
        # the 3D heated channel in FP32 with the autotuner's usual choice: about 2^20 cells
        dict(name="channel_256x64x64_f32", kind="step", family="channel", nx=256, ny=64, nz=64, levels=6,
             precision="f32", steps=10, pre=3, post=3, inner=1, krylov=1, smoother=1, geometry=0),
        # the same channel on the FP64 path with the plain V(3,3) cycle (the accuracy yardstick)
        dict(name="channel_256x64x64_f64", kind="step", family="channel", nx=256, ny=64, nz=64, levels=6,
             precision="f64", steps=4, pre=3, post=3, inner=0, krylov=0, smoother=0, geometry=0),
        # a long FP32 channel, 128 x 128 cells across (the method's published timing geometry)
        dict(name="channel_512x128x128_f32", kind="step", family="channel", nx=512, ny=128, nz=128, levels=6,
             precision="f32", steps=4, pre=3, post=3, inner=1, krylov=1, smoother=1, geometry=0),
        # the indoor room, 16.8 M cells, BF16 corrections: the default benchmark workload
        dict(name="room_512x256x128_bf16", kind="step", family="room", nx=512, ny=256, nz=128, levels=7,
             precision="bf16", steps=4, pre=2, post=2, inner=1, krylov=1, smoother=1, geometry=0),
        # uneven channels stepped together (FP32): a parameter study
        dict(name="batch_8_channels_f32", kind="batch", family="channels", n=8, precision="f32", steps=4, geometry=0),
        # served rooms and channels of uneven sizes stepped together (BF16 corrections)
        dict(name="batch_8_served_bf16", kind="batch", family="served", n=8, precision="bf16", steps=2, geometry=1),
        # the pressure solve alone: V-cycles with the flexible-CG step from zero on a served room
        dict(name="vcycle_room_256x128x128_bf16", kind="vcycle", family="room", nx=256, ny=128, nz=128, levels=5,
             precision="bf16", cycles=24, pre=2, post=2, inner=1, krylov=1, smoother=1, geometry=2),
        # the lambda_2 vortex field of a room's velocity, for a picture every few steps
        dict(name="lambda2_room_256x128x128_f32", kind="lambda2", family="room", nx=256, ny=128, nz=128, levels=5,
             precision="f32", geometry=2),
        # backward: cotangents of one whole step (a gradient for a small design problem, FP64)
        dict(name="step_vjp_96x48x32_f64", kind="vjp", family="channel", nx=96, ny=48, nz=32, levels=4,
             precision="f64", pre=3, post=3, geometry=0),
        # the allocation-free residual on caller-owned device buffers, odd sizes
        dict(name="residual_201x130x97_f64", kind="residual", nx=201, ny=130, nz=97),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, cells_lo, cells_hi):
    """An even-coarsening 3D grid: (nx, ny, nz, levels), its coarsest level at most 1024 cells."""
    while True:
        levels = rng.choice([4, 4, 5, 5, 6])
        unit = 2 ** (levels - 1)
        n = [unit * _log_int(rng, 2, 512 // unit if unit < 64 else 8) for _ in range(3)]
        n[0] = max(n)
        coarse = math.prod(x // unit for x in n)
        if cells_lo <= math.prod(n) <= cells_hi and coarse <= 1024 and max(n) <= 512 and min(n) >= 32:
            return n[0], n[1], n[2], levels


def draw(rng):
    kind = rng.choice(["channel2d", "channel", "channel", "room", "room", "batch", "vcycle", "lambda2", "vjp",
                       "residual"])
    g = rng.randrange(1, 500)
    if kind == "channel2d":
        levels = rng.choice([2, 3, 4, 5])
        unit = 2 ** (levels - 1)
        nx, ny = unit * rng.randrange(256 // unit // 4, 384 // unit), unit * max(2, _log_int(rng, 16, 96) // unit)
        while (nx // unit) * (ny // unit) > 1024:
            nx //= 2 * unit
            nx *= unit
        return dict(kind="step", family="channel2d", nx=nx, ny=ny, nz=1, levels=levels, precision=rng.choice(["f64", "f32"]),
                    steps=rng.choice([5, 10, 20]), pre=rng.choice([2, 3]), post=rng.choice([2, 3]), inner=0, krylov=0,
                    smoother=0, geometry=0)
    if kind in ("channel", "room"):
        prec = rng.choice(["f64", "f32", "f32", "bf16"] if kind == "channel" else ["f32", "bf16", "bf16"])
        top = _log_int(rng, 2e5, 1e6 if prec == "f64" else 9e6)
        nx, ny, nz, levels = _grid(rng, top // 2, top)
        krylov = 1 if kind == "room" else rng.choice([0, 1])
        return dict(kind="step", family=kind, nx=nx, ny=ny, nz=nz, levels=levels, precision=prec,
                    steps=rng.choice([2, 3, 4]), pre=rng.choice([2, 3]), post=2 if kind == "room" else 3,
                    inner=2 if kind == "room" else rng.choice([0, 1, 3]), krylov=krylov,
                    smoother=rng.choice([0, 1]), geometry=g)
    if kind == "batch":
        if rng.random() < 0.5:
            return dict(kind="batch", family="channels", n=rng.randrange(2, 9), precision="f32", steps=rng.choice([2, 3, 4]),
                        geometry=g)
        return dict(kind="batch", family="served", n=rng.randrange(2, 9), precision="bf16", steps=2, geometry=g)
    if kind == "residual":
        return dict(kind="residual", nx=_log_int(rng, 17, 400), ny=_log_int(rng, 17, 200), nz=_log_int(rng, 1, 200))
    if kind == "vjp":
        nx, ny, nz, levels = _grid(rng, 3e4, 2.2e5)
        return dict(kind="vjp", family="channel", nx=nx, ny=ny, nz=nz, levels=levels, precision="f64", pre=3, post=3,
                    geometry=g)
    nx, ny, nz, levels = _grid(rng, 2e5, 5e6)
    if kind == "lambda2":
        return dict(kind="lambda2", family="room", nx=nx, ny=ny, nz=nz, levels=levels, precision="f32", geometry=g)
    return dict(kind="vcycle", family="room", nx=nx, ny=ny, nz=nz, levels=levels, precision=rng.choice(["f32", "bf16"]),
                cycles=24, pre=2, post=2, inner=1, krylov=1, smoother=1, geometry=g)


# ------------------------------------------------------------------ the cases' descriptions
def _spec(c):
    prec = PRECISION[c["precision"]]
    kw = {"max_vcycles": 200}
    for here, there in (("pre", "pre_sweeps"), ("post", "post_sweeps"), ("inner", "inner_cycles"),
                        ("krylov", "krylov"), ("smoother", "smoother")):
        if here in c:
            kw[there] = c[here]
    if c["family"] == "channel2d":
        return cases.channel_2d(c["nx"], c["ny"], c["levels"], precision=prec, **kw)
    if c["family"] == "channel":
        return cases.heated_channel_3d(c["nx"], c["ny"], c["nz"], mg_levels=c["levels"], precision=prec, **kw)
    h = 0.02 if c["nx"] == 512 else 0.04
    return cases.room_3d(c["nx"], c["ny"], c["nz"], seed=c["geometry"], mg_levels=c["levels"], precision=prec, h=h, **kw)


def _specs(c):
    if c["family"] == "channels":
        return [s.replace(pre_sweeps=3, post_sweeps=3, inner_cycles=2, krylov=1, smoother=1, max_vcycles=200)
                for s in cases.batched_channels(c["n"], seed=c["geometry"], precision=PRECISION[c["precision"]])]
    specs = cases.served_rooms(c["n"], seed=c["geometry"], precision=PRECISION[c["precision"]])[1]
    return [s.replace(max_vcycles=200) for s in specs]


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _modes(gen, shape):
    """A smooth field in [-1, 1]: four separable modes of one to three waves a side."""
    out = torch.zeros(shape, dtype=torch.float64, device=_device())
    for _ in range(4):
        f = None
        for axis, n in enumerate(shape):
            wave, phase = 1.0 + 2.0 * torch.rand(1, generator=gen).item(), 6.3 * torch.rand(1, generator=gen).item()
            x = (torch.arange(n, dtype=torch.float64, device=out.device) + 0.5) / n
            s = torch.sin(2.0 * math.pi * wave * x + phase).reshape([-1 if a == axis else 1 for a in range(3)])
            f = s if f is None else f * s
        out += 0.25 * f
    return out


def _solid(spec):
    m = torch.zeros((spec.nz, spec.ny, spec.nx), dtype=torch.bool, device=_device())
    for b in spec.boxes:
        m[b.k0:b.k1, b.j0:b.j1, b.i0:b.i1] = True
    return m


def _flow(spec, seed):
    """A seeded flow state of the case: seven 64-bit fields (nz, ny, nx), p = 0."""
    gen = torch.Generator().manual_seed(1000003 * seed + 17)
    dgen = torch.Generator(device=_device()).manual_seed(1000003 * seed + 29)
    shape = (spec.nz, spec.ny, spec.nx)
    inlet = next(p for p in list(spec.faces) + [v.bc for v in spec.vents] if p.kind == cases.INLET)
    k0 = 1.5 * (inlet.intensity * inlet.u_normal) ** 2
    om0 = math.sqrt(k0) / (0.09 * inlet.length_scale)
    noise = lambda: 2.0 * torch.rand(shape, generator=dgen, dtype=torch.float64, device=_device()) - 1.0  # noqa: E731
    f = {}
    base = max(abs(x) for x in spec.init_vel) or 0.2
    bump = torch.ones(shape, dtype=torch.float64, device=_device())
    if spec.buoyancy:                       # a room: the motion dies away towards the walls
        for axis, n in enumerate(shape):
            x = (torch.arange(n, dtype=torch.float64, device=bump.device) + 0.5) / n
            bump = bump * (4.0 * x * (1.0 - x)).reshape([-1 if a == axis else 1 for a in range(3)])
    for n, name in enumerate(("u", "v", "w")):
        if spec.nz == 1 and name == "w":
            f[name] = torch.zeros(shape, dtype=torch.float64, device=_device())
            continue
        swing = 0.5 if spec.buoyancy else 0.04
        f[name] = spec.init_vel[n] + base * bump * (swing * _modes(gen, shape) + 0.01 * noise())
    f["p"] = torch.zeros(shape, dtype=torch.float64, device=_device())
    f["T"] = spec.init_T + 1.5 * _modes(gen, shape) + 0.05 * noise()
    f["k"] = k0 * (1.0 + 0.4 * _modes(gen, shape) + 0.01 * noise())
    f["omega"] = om0 * (1.0 + 0.3 * _modes(gen, shape) + 0.01 * noise())
    solid = _solid(spec)
    return {name: torch.where(solid, torch.zeros_like(x), x) for name, x in f.items()}


def _pinned(n, dtype):
    return torch.empty(n, dtype=dtype, pin_memory=torch.cuda.is_available()).numpy()


def _host(spec, tensors):
    """The tensors in one pinned host buffer, one after the other, in the case's storage type."""
    dtype = torch.float64 if spec.precision == cases.FP64 else torch.float32
    flat = torch.empty(len(tensors) * spec.cells, dtype=dtype, pin_memory=torch.cuda.is_available())
    for i, t in enumerate(tensors):
        flat[i * spec.cells:(i + 1) * spec.cells].copy_(t.reshape(-1).to(dtype))
    return flat.numpy()


def _stored(spec, f):
    """The fields as the case stores them."""
    if spec.precision == cases.FP64:
        return f
    return {name: x.float().double() for name, x in f.items()}


def _xyz(flat, spec):
    """A flat x-fastest array as the binding's (nx, ny, nz) view."""
    return flat.reshape(spec.nz, spec.ny, spec.nx).transpose(2, 1, 0)


def _rhs(spec, seed):
    """A right-hand side like -div(u*)/dt of a flow at rest disturbed at large and small scale."""
    gen = torch.Generator().manual_seed(1000003 * seed + 41)
    dgen = torch.Generator(device=_device()).manual_seed(1000003 * seed + 43)
    shape = (spec.nz, spec.ny, spec.nx)
    b = _modes(gen, shape) + 0.2 * (2.0 * torch.rand(shape, generator=dgen, dtype=torch.float64, device=_device()) - 1.0)
    b = torch.where(_solid(spec), torch.zeros_like(b), b)
    return b if spec.precision == cases.FP64 else b.float().double()


def _cotangents(spec, seed):
    gen = torch.Generator().manual_seed(1000003 * seed + 59)
    shape = (spec.nz, spec.ny, spec.nx)
    return [_modes(gen, shape) for _ in FIELDS]


VJP_DT = 2e-4
RESIDUAL_H = (0.01, 0.0125, 0.02)
RESIDUAL_DIRICHLET = (0, 1, 0, 0, 0, 0)


# ------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    kind = case["kind"]
    if kind == "residual":
        nx, ny, nz = case["nx"], case["ny"], case["nz"]
        p, b = _residual_inputs(case, seed)
        return {"kind": kind, "n": (nx, ny, nz), "p": p, "b": b, "r": torch.empty_like(p),
                "norms": torch.empty(2, dtype=torch.float64, device=p.device),
                "h": (ctypes.c_double * 3)(*RESIDUAL_H), "dir": (ctypes.c_int32 * 6)(*RESIDUAL_DIRICHLET)}
    specs = _specs(case) if kind == "batch" else [_spec(case)]
    s = {"kind": kind, "case": case, "specs": specs, "cs": [binding.Case(spec) for spec in specs]}
    if kind in ("step", "batch"):
        s["in"] = [_host(spec, list(_flow(spec, seed + 7919 * i).values())) for i, spec in enumerate(specs)]
        s["out"] = [np.empty_like(x) if not torch.cuda.is_available() else
                    _pinned(x.size, torch.float64 if x.dtype == np.float64 else torch.float32) for x in s["in"]]
        if kind == "batch":
            s["batch"] = binding.Batch(s["cs"])
        return s
    spec, c = specs[0], s["cs"][0]
    if kind == "vcycle":
        c.set_rhs(_xyz(_rhs(spec, seed).reshape(-1).cpu().numpy(), spec))
        s["in"] = _host(spec, [torch.zeros(spec.cells)])
        s["out"] = _pinned(spec.cells, torch.float32)
        return s
    c.write_flat(_host(spec, list(_flow(spec, seed).values())))
    if kind == "lambda2":
        s["out"] = _pinned(spec.cells, torch.float64)
    else:
        s["ybar"] = [_xyz(y.reshape(-1).cpu().numpy(), spec) for y in _cotangents(spec, seed)]
    return s


def _split(flat, spec):
    N = spec.cells
    return {name: flat[i * N:(i + 1) * N] for i, name in enumerate(FIELDS)}


def run(s):
    kind = s["kind"]
    if kind == "residual":
        st = binding.lib().fvm_poisson_residual_static(
            s["p"].data_ptr(), s["b"].data_ptr(), *s["n"], s["h"], s["dir"], s["r"].data_ptr(), s["norms"].data_ptr(),
            torch.cuda.current_stream().cuda_stream)
        if st != binding.OK:
            raise binding.FvmError(st, binding.last_error())
        return {"r": s["r"], "norms": s["norms"]}
    c, spec = s["cs"][0], s["specs"][0]
    if kind in ("step", "batch"):
        for c, x in zip(s["cs"], s["in"]):
            c.write_flat(x)
        (s["batch"] if kind == "batch" else c).step(s["case"]["steps"])
        for c, x in zip(s["cs"], s["out"]):
            c.read_flat(x)
        return [_split(x, spec) for x, spec in zip(s["out"], s["specs"])]
    if kind == "vcycle":
        c.write_flat(s["in"], fields=("p",))
        c.vcycle(s["case"]["cycles"])
        return {"p": c.read_flat(s["out"], fields=("p",))}
    if kind == "lambda2":
        c.lambda2(out=s["out"])
        return {"lambda2": s["out"]}
    xbar, _ = c.step_vjp(VJP_DT, *s["ybar"], rel_tol=1e-10)
    return {name: x.transpose(2, 1, 0).reshape(-1) for name, x in zip(("u", "v", "w", "T", "k", "omega"), xbar)}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind == "residual":
        n = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 24.0 * n + 16.0, "flops": 17.0 * n}
    specs = _specs(case) if kind == "batch" else [_spec(case)]
    cells = float(sum(spec.cells for spec in specs))
    size = 8 if case["precision"] == "f64" else 4
    if kind in ("step", "batch"):
        # per step: the six state fields and p (8 bytes a cell) read and written once, at least one
        # pass over the pressure system; the closure, fluxes and gradients are about 700 operations
        return {"bytes": case["steps"] * cells * 2.0 * (6 * size + 8) + 2.0 * cells * 7 * size,
                "flops": case["steps"] * cells * 700.0}
    if kind == "vcycle":   # p in and out, b, the correction and its right-hand side once a cycle
        return {"bytes": case["cycles"] * cells * (16.0 + 4.0 + 2.0 * (2 if case["precision"] == "bf16" else 4)),
                "flops": case["cycles"] * cells * 80.0}
    if kind == "lambda2":
        return {"bytes": cells * (3 * size + 1 + 8.0), "flops": cells * 300.0}
    return {"bytes": cells * 8.0 * (7 + 6 + 6), "flops": cells * 4000.0}


# ------------------------------------------------------------------ the method in plain 64-bit torch
class _Solve(torch.autograd.Function):
    """A p = b (A symmetric on the fluid cells), exactly: the backward pass is the same solve."""

    @staticmethod
    def forward(ctx, b, ref, start):
        ctx.ref = ref
        return ref.cg(b, start)

    @staticmethod
    def backward(ctx, g):
        return ctx.ref.cg(g, torch.zeros_like(g)), None, None


class Reference:
    """One case's discrete equations on (nz, ny, nx) arrays."""

    def __init__(self, spec):
        self.s, self.dev = spec, _device()
        self.shape = (spec.nz, spec.ny, spec.nx)
        self.h = (spec.Lx / spec.nx, spec.Ly / spec.ny, spec.Lz / spec.nz)
        self.active = [n > 1 for n in (spec.nx, spec.ny, spec.nz)]
        self.alpha = spec.nu / spec.Pr
        self.solid = _solid(spec)
        self.fluid = ~self.solid
        patches = list(spec.faces) + [v.bc for v in spec.vents]
        box = torch.zeros(self.shape, dtype=torch.int64, device=self.dev)
        for n, b in enumerate(spec.boxes):
            box[b.k0:b.k1, b.j0:b.j1, b.i0:b.i1] = n + 1
        # per axis and side: the face kind (-1 inside) and the ghosts' sign and constant per field
        self.kind, self.sign, self.const = {}, {}, {}
        for a in range(3):
            if not self.active[a]:
                continue
            d = 2 - a
            for side in (0, 1):
                kind = torch.full(self.shape, -1, dtype=torch.int64, device=self.dev)
                sign = {f: torch.zeros(self.shape, dtype=torch.float64, device=self.dev) for f in FIELDS}
                const = {f: torch.zeros(self.shape, dtype=torch.float64, device=self.dev) for f in FIELDS}
                nb = self.shift(box, a, side)
                edge = torch.zeros(self.shape, dtype=torch.bool, device=self.dev)
                edge.select(d, self.shape[d] - 1 if side else 0).fill_(True)
                for n, b in enumerate(spec.boxes):
                    self._ghost((nb == n + 1) & ~edge & self.fluid, kind, sign, const, cases.Patch(
                        kind=cases.WALL, thermal=b.thermal, T_value=b.T_value), a, side)
                face = 2 * a + side
                pid = torch.full([n for i, n in enumerate(self.shape) if i != d], face, dtype=torch.int64, device=self.dev)
                for n, v in enumerate(spec.vents):
                    if v.face == face:                     # (the second tangential axis is the slower one)
                        pid[v.b0:v.b1, v.a0:v.a1] = 6 + n
                pid = pid.unsqueeze(d).expand(self.shape)
                for i in pid.unique().tolist():
                    self._ghost(edge & (pid == i), kind, sign, const, patches[i], a, side)
                self.kind[a, side], self.sign[a, side], self.const[a, side] = kind, sign, const

    def _ghost(self, where, kind, sign, const, p, a, side):
        """Ghost = sign * cell + const across the faces `where` with the patch p."""
        s = self.s
        kind[where] = p.kind
        sg = {f: 1.0 for f in FIELDS}
        ct = {f: 0.0 for f in FIELDS}
        if p.kind == cases.WALL:
            sg["u"] = sg["v"] = sg["w"] = -1.0
            if p.thermal == cases.FIXED_T:
                sg["T"], ct["T"] = -1.0, 2.0 * p.T_value
            elif p.thermal == cases.HEAT_FLUX:
                ct["T"] = p.T_value * self.h[a] / (s.rho * s.cp * self.alpha)
        elif p.kind == cases.INLET:
            k0 = 1.5 * (p.intensity * p.u_normal) ** 2
            for f in ("u", "v", "w", "T", "k", "omega"):
                sg[f] = -1.0
            ct["uvw"[a]] = 2.0 * p.u_normal * (-1.0 if side else 1.0)
            ct["T"], ct["k"], ct["omega"] = 2.0 * p.T_in, 2.0 * k0, 2.0 * math.sqrt(k0) / (0.09 * p.length_scale)
        elif p.kind == cases.OUTLET:
            sg["p"] = -1.0
        for f in FIELDS:
            sign[f][where] = sg[f]
            const[f][where] = ct[f]

    def shift(self, x, a, side):
        """The neighbour's value on that side (the cell's own at a domain face)."""
        d = 2 - a
        n = self.shape[d]
        if side:
            return torch.cat([x.narrow(d, 1, n - 1), x.narrow(d, n - 1, 1)], d)
        return torch.cat([x.narrow(d, 0, 1), x.narrow(d, 0, n - 1)], d)

    def across(self, x, f, a, side):
        inside = self.kind[a, side] < 0
        return torch.where(inside, self.shift(x, a, side), self.sign[a, side][f] * x + self.const[a, side][f])

    def gradient(self, x, f):
        return [0.5 * (self.across(x, f, a, 1) - self.across(x, f, a, 0)) / self.h[a] if self.active[a]
                else torch.zeros_like(x) for a in range(3)]

    # the closure
    def ret(self, k, om):
        return k / (self.s.nu * om.clamp(min=1e-12))

    def alpha_star(self, k, om):
        r = self.ret(k, om) / 6.0
        return (0.024 + r) / (1.0 + r)

    def nut(self, k, om):
        return torch.where(self.fluid, self.alpha_star(k, om) * k / om.clamp(min=1e-12), torch.zeros_like(k))

    def stable_dt(self, f, dt0):
        nut = self.nut(f["k"], f["omega"])
        gam = torch.maximum(self.s.nu + nut, self.alpha + nut / self.s.Prt)
        lam = sum(f["uvw"[a]].abs() / self.h[a] + 2.0 * gam / self.h[a] ** 2 for a in range(3) if self.active[a])
        lam = torch.where(self.fluid, lam, torch.zeros_like(lam)).max().item()
        return min(dt0, self.s.cfl / lam) if lam > 0.0 else dt0

    def destruction(self, f, dt):
        k, om = f["k"], f["omega"]
        oms = om.clamp(min=1e-12)
        g = [self.gradient(f[n], n) for n in "uvw"]
        gk, gw = self.gradient(k, "k"), self.gradient(om, "omega")
        chik = sum(x * y for x, y in zip(gk, gw)) / oms ** 3
        fbs = torch.where(chik <= 0.0, torch.ones_like(k), (1.0 + 680.0 * chik ** 2) / (1.0 + 400.0 * chik ** 2))
        fbs = torch.where(chik > 1e8, torch.full_like(k, 680.0 / 400.0), fbs)
        x4 = (self.ret(k, om) / 8.0) ** 4
        bs = torch.where(x4 > 1e16, torch.full_like(k, 0.09), 0.09 * (4.0 / 15.0 + x4) / (1.0 + x4))
        S = [[0.5 * (g[i][j] + g[j][i]) for j in range(3)] for i in range(3)]
        O = [[0.5 * (g[i][j] - g[j][i]) for j in range(3)] for i in range(3)]
        t = sum(O[i][j] * O[j][m] * S[m][i] for i in range(3) for j in range(3) for m in range(3))
        chiw = (t / (0.09 * oms) ** 3).abs()
        fb = (1.0 + 70.0 * chiw) / (1.0 + 80.0 * chiw)
        out = dict(f)
        out["k"] = torch.where(self.fluid, k / (1.0 + dt * bs * fbs * om), k)
        out["omega"] = torch.where(self.fluid, om / (1.0 + dt * 0.072 * fb * om), om)
        return out

    def explicit(self, f, dt):
        s, names = self.s, ("u", "v", "w", "T", "k", "omega")
        mol = {"u": s.nu, "v": s.nu, "w": s.nu, "T": self.alpha, "k": s.nu, "omega": s.nu}
        sig = {"u": 1.0, "v": 1.0, "w": 1.0, "T": s.Prt, "k": s.sigma_k, "omega": s.sigma_w}
        k, om = f["k"], f["omega"]
        safe_k = torch.where(self.fluid, k, torch.ones_like(k))
        nut = self.nut(k, om)
        rhs = {n: torch.zeros_like(k) for n in names}
        wall = torch.zeros_like(k)
        for a in range(3):
            if not self.active[a]:
                continue
            h, normal = self.h[a], "uvw"[a]
            for side in (0, 1):
                kind = self.kind[a, side]
                up = 1.0 if side else -1.0
                ghost = {n: self.across(f[n], n, a, side) for n in names}
                uf = 0.5 * (f[normal] + ghost[normal])
                nf = torch.where(kind < 0, 0.5 * (nut + self.shift(nut, a, side)), nut)
                nf = torch.where(kind == cases.WALL, torch.zeros_like(nf), nf)
                own = (uf >= 0.0) if side else (uf < 0.0)     # the face takes this cell's value
                for n in names:
                    flux = -(torch.where(own, f[n], ghost[n]) * uf) + (mol[n] + nf / sig[n]) * up * (ghost[n] - f[n]) / h
                    if n == normal:
                        flux = flux - (2.0 / 3.0) * 0.5 * (k + ghost["k"])
                    rhs[n] = rhs[n] + up * flux / h
                wall = torch.where(kind == cases.WALL, wall.clamp(min=6.0 * s.nu / (0.072 * (0.5 * h) ** 2)), wall)
        g = [self.gradient(f[n], n) for n in "uvw"]
        S2 = 2.0 * sum((0.5 * (g[i][j] + g[j][i])) ** 2 for i in range(3) for j in range(3))
        r = self.ret(k, om) / 2.95
        alpha = 0.52 / self.alpha_star(k, om) * (1.0 / 9.0 + r) / (1.0 + r)
        rhs["k"] = rhs["k"] + nut * S2
        rhs["omega"] = rhs["omega"] + alpha * om / safe_k * nut * S2
        if s.buoyancy:
            for i, n in enumerate("uvw"):
                rhs[n] = rhs[n] - s.gravity[i] * s.beta_T * (f["T"] - s.T_ref)
        out = dict(f)
        for n in names:
            out[n] = torch.where(self.fluid, f[n] + dt * rhs[n], f[n])
        out["k"] = torch.where(self.fluid, out["k"].clamp(min=1e-14), k)
        out["omega"] = torch.where(self.fluid, out["omega"].clamp(min=1e-8), om)
        out["omega"] = torch.where(self.fluid & (wall > 0.0), wall, out["omega"])
        return out

    def rhs(self, f, dt):
        div = torch.zeros_like(f["u"])
        for a in range(3):
            if self.active[a]:
                n = "uvw"[a]
                div = div + 0.5 * (self.across(f[n], n, a, 1) - self.across(f[n], n, a, 0)) / self.h[a]
        return torch.where(self.fluid, -div / dt, torch.zeros_like(div))

    def A(self, p):
        out = torch.zeros_like(p)
        for a in range(3):
            if self.active[a]:
                out = out + (2.0 * p - self.across(p, "p", a, 0) - self.across(p, "p", a, 1)) / self.h[a] ** 2
        return torch.where(self.fluid, out, torch.zeros_like(out))

    def cg(self, b, start):
        """Conjugate gradients to a 1e-13 relative residual, or as far as rounding lets it."""
        with torch.no_grad():
            b = torch.where(self.fluid, b, torch.zeros_like(b))
            p = start.clone()
            r = b - self.A(p)
            d, rr, goal = r.clone(), (r * r).sum(), 1e-26 * (b * b).sum().item()
            for it in range(8000):
                q = self.A(d)
                step = rr / (d * q).sum().clamp(min=1e-300)
                p = p + step * d
                r = r - step * q
                new = (r * r).sum()
                d = r + (new / rr.clamp(min=1e-300)) * d
                rr = new
                if it % 50 == 49 and rr.item() <= goal:
                    break
            return p

    def project(self, f, p, dt):
        out, g = dict(f), self.gradient(p, "p")
        for a, n in enumerate("uvw"):
            out[n] = torch.where(self.fluid, f[n] - dt * g[a], f[n])
        out["p"] = p
        return out

    def step(self, f, dt):
        f = self.destruction(f, 0.5 * dt)
        f = self.explicit(f, dt)
        f = self.destruction(f, 0.5 * dt)
        return self.project(f, _Solve.apply(self.rhs(f, dt), self, f["p"].detach()), dt)


def _steps_exact(spec, seed, steps):
    ref, f = Reference(spec), _stored(spec, _flow(spec, seed))
    hmin = min(h for h, on in zip(ref.h, ref.active) if on)
    dt0 = spec.cfl * hmin / max(p.u_normal for p in list(spec.faces) + [v.bc for v in spec.vents]
                                if p.kind == cases.INLET)
    with torch.no_grad():
        for _ in range(steps):
            f = ref.step(f, ref.stable_dt(f, dt0))
    return {name: f[name].reshape(-1) for name in FIELDS}


def _middle_eigenvalue(m00, m11, m22, m01, m02, m12):
    """The middle eigenvalue of a symmetric 3 x 3 matrix, by torch's own solver in slices."""
    out = torch.empty_like(m00)
    for lo in range(0, m00.numel(), 1 << 20):
        a, b, c, d, e, f = (x.reshape(-1)[lo:lo + (1 << 20)] for x in (m00, m11, m22, m01, m02, m12))
        M = torch.stack([a, d, e, d, b, f, e, f, c], -1).reshape(-1, 3, 3).cpu()
        out.view(-1)[lo:lo + (1 << 20)] = torch.from_numpy(np.linalg.eigvalsh(M.numpy())[:, 1]).to(out.device)
    return out


def _residual_inputs(case, seed):
    shape = (case["nz"], case["ny"], case["nx"])
    gen = torch.Generator().manual_seed(1000003 * seed + 71)
    dgen = torch.Generator(device=_device()).manual_seed(1000003 * seed + 73)
    p = 5.0 + _modes(gen, shape)
    b = 50.0 * _modes(gen, shape) + torch.randn(shape, generator=dgen, dtype=torch.float64, device=p.device)
    return p, b


def exact(case, seed):
    kind = case["kind"]
    if kind == "residual":
        p, b = _residual_inputs(case, seed)
        r = b.clone()
        for a, d in ((0, 2), (1, 1), (2, 0)):
            n = p.shape[d]
            if n == 1:
                continue
            first, last = p.narrow(d, 0, 1), p.narrow(d, n - 1, 1)
            lo = torch.cat([-first if RESIDUAL_DIRICHLET[2 * a] else first, p.narrow(d, 0, n - 1)], d)
            hi = torch.cat([p.narrow(d, 1, n - 1), -last if RESIDUAL_DIRICHLET[2 * a + 1] else last], d)
            r -= ((p - lo) + (p - hi)) / RESIDUAL_H[a] ** 2
        return {"r": r, "norms": torch.stack([(r * r).sum(), (b * b).sum()])}
    specs = _specs(case) if kind == "batch" else [_spec(case)]
    spec, cells = specs[0], sum(s.cells for s in specs)
    if kind in ("step", "batch"):
        if cells * case["steps"] > EXACT_CELL_STEPS:
            return None
        return [_steps_exact(s, seed + 7919 * i, case["steps"]) for i, s in enumerate(specs)]
    if kind == "vcycle":
        b = _rhs(spec, seed)
        return {"p": Reference(spec).cg(b, torch.zeros_like(b)).reshape(-1)}
    f = _stored(spec, _flow(spec, seed))
    ref = Reference(spec)
    if kind == "lambda2":
        g = [ref.gradient(f[n], n) for n in "uvw"]
        S = [[0.5 * (g[i][j] + g[j][i]) for j in range(3)] for i in range(3)]
        O = [[0.5 * (g[i][j] - g[j][i]) for j in range(3)] for i in range(3)]
        M = [[sum(S[i][m] * S[m][j] + O[i][m] * O[m][j] for m in range(3)) for j in range(3)] for i in range(3)]
        lam = _middle_eigenvalue(M[0][0], M[1][1], M[2][2], M[0][1], M[0][2], M[1][2])
        return {"lambda2": torch.where(ref.fluid, lam, torch.zeros_like(lam)).reshape(-1)}
    x = {name: t.clone().requires_grad_(name != "p") for name, t in f.items()}
    y = ref.step(x, VJP_DT)
    total = sum((y[name] * ybar).sum() for name, ybar in zip(FIELDS, _cotangents(spec, seed)))
    names = ("u", "v", "w", "T", "k", "omega")
    return {name: g.reshape(-1) for name, g in zip(names, torch.autograd.grad(total, [x[n] for n in names]))}
