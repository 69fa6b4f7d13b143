"""The work that users of this framework have it do, as cases that can be timed.

A case is a dict of plain values; ``prepare`` makes what a program has in hand before the
call, ``run`` is one pass through the public entry points (the Context class, the module
functions and the C ABI of ``paper_2403_11156_gb300.sph``), ``work`` the bytes and operations a
pass cannot do without and ``exact`` the same result in 64 bits, written in plain torch.

Kinds of cases:

* ``step``: a rollout.  A saved state (positions, velocities, the solves' warm-start memory,
  rigid poses) is written into a context, a number of steps is taken with the scene's own
  tolerances, and the new state is read back into device buffers.  This is what a program
  does that continues from checkpoints, compares settings from one state or collects
  training data; the solves, which stop at their tolerances, then do the same work in every
  pass.  A warm-started rollout is one step long: its gates (compressing or not) are
  decisions, and from the second step on the last bit of a sum decides some of them.
* ``order``: the grid order of a caller's points without allocation.
* ``mlp_forward``, ``mlp_grad``, ``mlp_train``: the warm-start network evaluated, its gradient,
  and training epochs.
* ``post``: the post-processing of one frame, the volume-fraction field, its iso-surface and
  the height map.
"""
from __future__ import annotations

import ctypes
import math

import numpy as np
import torch

from paper_2403_11156_gb300 import scenes, sph, warmstart

G = 9.81
DISORDER = 0.03   # displacement of the start state's particles, in lattice spacings
SHEAR = 0.6       # m/s, the smooth part of the start state's velocities
NOISE = 0.01      # m/s, their random part


# ------------------------------------------------------------------------------ the cases
def _step(name, scene, steps, **kw):
    c = dict(name=name, kind="step", scene=scene, steps=steps)
    c.update(kw)
    return c


def listed():
    return [
        # the small dam break of the tests and the benchmark: a scene far too small to fill
        # the GPU, where a step is bound by latency and launches; solves from zero
        _step("dam_8k", "small", 4, nx=20, ny=20, nz=20, box=0.8, warm="zero"),
        # a ragged scene of ordinary size in a longer tank, CFL time step
        _step("dam_100k", "random", 1, n=100_003, aspect=2.3, fill=0.37, radius=0.005),
        # the headline workload: 1.2M particles, walls and three floating boxes, CFL time
        # step, 0.1 % tolerances of both solves, previous-step warm start
        _step("rigid_1200k", "rigid", 1, nx=125, ny=98, nz=98, bodies=3, strong=False),
        # many independent scenes of 20k-200k particles stepped in one context
        _step("batch_8", "batch", 1, scenes=8, lo=20_000, hi=200_000, radius=0.01),
        # the high-viscosity column: a conjugate-gradient solve in every step
        _step("column_250k", "column", 1, nx=50, ny=50, nz=100),
        # the equation-of-state solver, which takes many short steps without iterating
        _step("wcsph_500k", "random", 3, n=500_009, aspect=1.4, fill=0.45, radius=0.005, solver="wcsph"),
        # the smallest call: the grid order of a few thousand points of a caller
        dict(name="order_3k", kind="order", n=3001, cell=0.04, extent=0.8),
        # the same call at the largest size it takes
        dict(name="order_262k", kind="order", n=262_143, cell=0.04, extent=2.0),
        # the warm-start network over a scene's particles, as the learned start or an
        # evaluation of its fit runs it
        dict(name="mlp_forward_1200k", kind="mlp_forward", n=1_200_500),
        # gradient of the network's loss over a data set (a full-batch optimiser's call)
        dict(name="mlp_grad_200k", kind="mlp_grad", n=200_000),
        # training epochs in mini-batches
        dict(name="mlp_train_50k", kind="mlp_train", n=50_021, epochs=2, batch=4096),
        # one frame of output of the large scene: field on a grid of spacing r, surface, view
        dict(name="post_1200k", kind="post", nx=125, ny=98, nz=98, grid=1.0),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["order", "mlp_forward", "mlp_grad", "mlp_train", "post"])
    if kind == "order":
        n = int(_log(rng, 500, sph.NOALLOC_MAX_POINTS))
        return dict(kind=kind, n=n, cell=0.04, extent=round(rng.uniform(0.6, 2.4), 3))
    if kind == "mlp_forward":
        return dict(kind=kind, n=int(_log(rng, 100, 1_200_000)))
    if kind == "mlp_grad":
        return dict(kind=kind, n=int(_log(rng, 1000, 200_000)))
    if kind == "mlp_train":
        return dict(kind=kind, n=int(_log(rng, 2000, 50_000)), epochs=rng.randint(1, 2),
                    batch=rng.choice([256, 1000, 1024, 4096]))
    nx, ny, nz = (int(_log(rng, 16, 98)) for _ in range(3))
    if kind == "post":
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, grid=rng.choice([1.0, 1.5, 2.0]))
    scene = rng.choice(["small", "random", "random", "random", "rigid", "batch", "column"])
    steps = 1   # of the warm-started ones
    if scene == "small":
        n = [rng.randint(12, 40) for _ in range(3)]
        return dict(kind=kind, scene=scene, steps=rng.randint(1, 4), warm="zero", nx=n[0], ny=n[1], nz=n[2],
                    box=round((max(n) + 3) * 0.02 * rng.uniform(1.0, 1.5), 2),
                    solver=rng.choice(["dfsph", "dfsph", "wcsph", "pcisph"]),
                    viscosity=rng.choice(["none", "explicit", "xsph"]))
    if scene == "rigid":
        return dict(kind=kind, scene=scene, steps=steps, nx=nx, ny=ny, nz=nz,
                    bodies=rng.randint(1, 3), strong=rng.random() < 0.3)
    if scene == "batch":
        return dict(kind=kind, scene=scene, steps=steps, scenes=rng.randint(2, 6), lo=5000,
                    hi=int(_log(rng, 10_000, 150_000)), radius=0.01)
    if scene == "column":
        return dict(kind=kind, scene=scene, steps=steps, nx=rng.randint(10, 50),
                    ny=rng.randint(10, 50), nz=rng.randint(16, 100))
    solver = rng.choice(["dfsph"] * 4 + ["wcsph", "pcisph"])
    warm = rng.choice(["previous", "zero"]) if solver == "dfsph" else "zero"
    return dict(kind=kind, scene=scene, steps=steps if warm == "previous" else rng.randint(1, 3),
                n=int(_log(rng, 3000, 700_000)), aspect=round(rng.uniform(1.0, 3.0), 2),
                fill=round(rng.uniform(0.2, 0.6), 2), radius=0.005, solver=solver, warm=warm)


# ------------------------------------------------------------------------- scenes of a case
VISCOSITY = dict(none=scenes.VISC_NONE, explicit=scenes.VISC_EXPLICIT, xsph=scenes.VISC_XSPH)


def _options(case, height, radius):
    kw = {}
    if case.get("viscosity"):
        kw["viscosity_mode"] = VISCOSITY[case["viscosity"]]
        kw["xsph_c"] = 0.05
    if case.get("warm") == "zero":
        kw["warm_start"] = scenes.WARM_ZERO
    if case.get("solver") == "wcsph":
        kw.update(scenes.wcsph_parameters(height, radius))
    elif case.get("solver") == "pcisph":
        kw.update(pressure_solver=scenes.SOLVER_PCISPH, warm_start=scenes.WARM_ZERO, divergence_solve=0,
                  min_iter_density=3)
    return kw


def _descs(case, seed):
    """The scene descriptions of a step case, their lattices jittered by the seed."""
    k = case["scene"]
    if k == "small":
        n = (case["nx"], case["ny"], case["nz"])
        return [scenes.dam_break_small(seed=seed, n=n, box=case["box"], **_options(case, 0.02 * n[2], 0.01))]
    if k == "random":
        height = (case["n"] * (2 * case["radius"]) ** 3 / case["fill"] / case["aspect"]) ** (1 / 3)
        return [scenes.dam_break_random(seed, case["n"], radius=case["radius"], aspect=case["aspect"],
                                        fill=case["fill"], **_options(case, height, case["radius"]))]
    if k == "rigid":
        return [scenes.dam_break_rigid(seed=seed, n=(case["nx"], case["ny"], case["nz"]), n_boxes=case["bodies"],
                                       rigid_coupling=scenes.COUPLING_STRONG if case["strong"] else 0)]
    if k == "batch":
        sizes = scenes.batch_scene_sizes(case["scenes"], case["lo"], case["hi"], 5)
        return [scenes.dam_break_random(seed * 100 + i, n, radius=case["radius"], aspect=1.0, fill=0.4,
                                        dt_max=4e-4, cfl=0.0) for i, n in enumerate(sizes)]
    return [scenes.viscous_column(seed=seed, n=(case["nx"], case["ny"], case["nz"]))]


def _start_state(d, seed):
    """Positions, velocities and warm-start memory of a flow that has been running: the
    lattice disordered, a smooth shearing flow with some noise, the hydrostatic stiffness."""
    rng = np.random.default_rng(seed)
    x0 = d["fluid_x"].astype(np.float64)
    lo, hi = x0.min(axis=0), x0.max(axis=0)
    size = np.maximum(hi - lo, 1e-6)
    u = (x0 - lo) / size
    v = np.stack([SHEAR * u[:, 2] * np.cos(2.0 * u[:, 1]), 0.3 * SHEAR * np.sin(3.0 * u[:, 0]),
                  -0.5 * SHEAR * u[:, 2] * u[:, 0]], axis=1)
    v += rng.normal(scale=NOISE, size=v.shape)
    s = 2.0 * d["radius"]
    x = x0 + rng.uniform(-DISORDER * s, DISORDER * s, size=x0.shape)
    depth = hi[2] - x0[:, 2]
    kappa = G * depth * rng.uniform(0.0, 1.0, size=len(x0))
    dt = d["dt_max"]
    f = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()  # noqa: E731
    return dict(x=f(x), v=f(v), kp=f(kappa * dt * dt), kvp=f(0.1 * kappa * dt))


class _StepState:
    def __init__(self, case, seed):
        self.steps = case["steps"]
        descs = _descs(case, seed)
        self.context = sph.Context(descs)
        self.start = [_start_state(d, seed * 1000 + i) for i, d in enumerate(descs)]
        self.bodies = [self.context.sph_read_bodies(i) if d["bodies"] else None for i, d in enumerate(descs)]
        self.out = [{"x": torch.empty_like(s["x"]), "v": torch.empty_like(s["v"]),
                     "rho": torch.empty_like(s["kp"])} for s in self.start]


def _run_step(s):
    g = s.context
    for i, q in enumerate(s.start):
        st = sph.load().sph_write_state(g.ctx, i, q["x"].data_ptr(), q["v"].data_ptr(), q["kp"].data_ptr(),
                                        q["kvp"].data_ptr(), 1)
        if st != sph.SPH_OK:
            raise sph.SphError(st, "sph_write_state")
        if s.bodies[i] is not None:
            g.sph_write_bodies(i, s.bodies[i])
    g.sph_steps(s.steps)
    for i, o in enumerate(s.out):
        g.sph_read_state_device(i, sync=False, **o)
    # poses in single precision, as a renderer takes them
    poses = [torch.from_numpy(g.sph_read_bodies(i)[:, :13].astype(np.float32))
             for i in range(len(s.out)) if s.bodies[i] is not None]
    return {"scenes": s.out, "poses": poses}


# ------------------------------------------------------------------------- the other kinds
def _mlp_data(n, seed):
    """Standardised features and labels of the kind the solver's states give: heavy-tailed
    labels that depend on the features."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    f = torch.randn((n, 4), generator=g, device="cuda")
    y = torch.sin(f[:, 0]) + 0.5 * f[:, 1] * torch.sigmoid(f[:, 2]) + 0.1 * torch.randn(n, generator=g, device="cuda") ** 3
    return f, y


def _mlp_params(seed):
    return torch.from_numpy(warmstart.init_params(seed)).cuda()


def _checked(status, name):
    if status != sph.SPH_OK:
        raise sph.SphError(status, name)


def prepare(case, seed):
    k = case["kind"]
    if k == "step":
        return case, _StepState(case, seed)
    s = {}
    if k == "order":
        g = torch.Generator(device="cuda").manual_seed(seed)
        s["x"] = torch.rand((case["n"], 3), generator=g, device="cuda") * case["extent"]
        s["order"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
        s["keys"] = torch.empty(case["n"], dtype=torch.int32, device="cuda")
        return case, s
    if k == "post":
        d = scenes.dam_break_rigid(seed=seed, n=(case["nx"], case["ny"], case["nz"]), n_boxes=0)
        s["desc"], s["context"] = d, sph.Context(d)
        q = _start_state(d, seed)
        s["x"] = q["x"]
        s["context"].sph_write_state(0, x=q["x"].cpu().numpy())
        r = d["radius"] * case["grid"]
        s["spacing"] = r
        s["dims"] = [int((d["domain_max"][a] - d["domain_min"][a]) / r) + 1 for a in range(3)]
        s["image"] = [int(2 * d["domain_max"][a] / d["radius"]) for a in range(2)]
        # the caller's triangle buffer: room for a surface rougher than the block's own
        faces = sum(a * b for a, b in ((case["nx"], case["ny"]), (case["ny"], case["nz"]), (case["nx"], case["nz"])))
        s["triangles"] = torch.zeros((int(128 * faces / case["grid"] ** 2) + 4096, 3, 3), device="cuda")
        return case, s
    s["params"] = _mlp_params(seed)
    s["features"], s["labels"] = _mlp_data(case["n"], seed)
    s["error"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    if k == "mlp_forward":
        s["y"] = torch.empty(case["n"], device="cuda")
    elif k == "mlp_grad":
        s["grad"] = torch.empty(sph.MLP_WEIGHTS, device="cuda")
        s["loss"] = torch.empty(1, dtype=torch.float64, device="cuda")
    else:
        s["trained"] = torch.empty_like(s["params"])
        s["adam"] = torch.empty(2 * sph.MLP_WEIGHTS, device="cuda")
        s["history"] = torch.empty(case["epochs"], device="cuda")
    return case, s


def run(state):
    case, s = state
    k = case["kind"]
    if k == "step":
        return _run_step(s)
    if k == "order":
        _checked(sph.sph_grid_order_noalloc(s["x"], case["n"], [0.0] * 3, [case["extent"]] * 3, case["cell"],
                                            s["order"], s["keys"]), "sph_grid_order_noalloc")
        return {"order": s["order"], "keys": s["keys"]}
    if k == "mlp_forward":
        _checked(sph.sph_mlp_forward(s["params"], s["features"], case["n"], s["y"], s["error"]), "sph_mlp_forward")
        return s["y"]
    if k == "mlp_grad":
        _checked(sph.sph_mlp_grad(s["params"], s["features"], s["labels"], case["n"], s["grad"], s["loss"],
                                  s["error"]), "sph_mlp_grad")
        # the loss in single precision, as a training log keeps it
        return {"grad": s["grad"], "loss": s["loss"].float()}
    if k == "mlp_train":
        s["trained"].copy_(s["params"])
        s["adam"].zero_()
        _checked(sph.sph_mlp_train(s["features"], s["labels"], case["n"], s["trained"], s["adam"], case["epochs"],
                                   case["batch"], 1e-3, 4, s["history"], s["error"]), "sph_mlp_train")
        return {"params": s["trained"], "adam": s["adam"], "history": s["history"]}
    g, d = s["context"], s["desc"]
    lo, hi = d["domain_min"], d["domain_max"]
    field = g.sph_surface_field(lo, s["spacing"], s["dims"])
    count = ctypes.c_int64()
    _checked(sph.load().sph_surface_mesh(field.data_ptr(), (ctypes.c_int32 * 3)(*s["dims"]), (ctypes.c_float * 3)(*lo),
                                         s["spacing"], 0.5, s["triangles"].data_ptr(), len(s["triangles"]),
                                         ctypes.byref(count), torch.cuda.current_stream().cuda_stream),
             "sph_surface_mesh")
    image = g.sph_render_heightmap(lo[:2], hi[:2], s["image"][0], s["image"][1], d["radius"])
    return {"field": field, "triangles": s["triangles"], "count": count.value, "image": image}


# ------------------------------------------------------------------------- what it cannot do without
def _counts(case):
    """(fluid, boundary) particles of a step case, from its sizes."""
    k = case["scene"]
    if k == "batch":
        sizes = scenes.batch_scene_sizes(case["scenes"], case["lo"], case["hi"], 5)
        return sum(sizes), sum(int(12 * (n / 0.4) ** (2 / 3)) for n in sizes)
    if k == "random":
        return case["n"], int(6 * (case["n"] / case["fill"]) ** (2 / 3))
    n = case["nx"] * case["ny"] * case["nz"]
    return n, {"small": int(6 * (case.get("box", 0.8) / 0.02) ** 2), "rigid": 100_002, "column": 40_401}[k]


def work(case):
    k = case["kind"]
    if k == "step":
        nf, nb = _counts(case)
        # the state written in (32 B a particle) and read out (28 B); per step the particle
        # and boundary state once; operations: 30 neighbours a particle, a density sum and
        # the fewest iterations of both solves at 22-40 operations a pair
        it = 1 if case.get("solver") == "wcsph" else 4
        return {"bytes": 60.0 * nf + case["steps"] * (64.0 * nf + 16.0 * nb),
                "flops": case["steps"] * nf * 30.0 * (40 + 30 + 24 * 2 * it)}
    n = case.get("n", 0)
    if k == "order":
        return {"bytes": 20.0 * n + 4.0 * (case["extent"] / case["cell"] + 2) ** 3, "flops": 10.0 * n}
    per_row = 2.0 * (4 * 64 + 64 * 64 + 64)
    if k == "mlp_forward":
        return {"bytes": 20.0 * n, "flops": per_row * n}
    if k == "mlp_grad":
        return {"bytes": 20.0 * n, "flops": 3.0 * per_row * n}
    if k == "mlp_train":
        return {"bytes": 20.0 * n * case["epochs"], "flops": 3.0 * per_row * n * case["epochs"]}
    nf = case["nx"] * case["ny"] * case["nz"]
    nodes = (200 / case["grid"] + 1) ** 2 * (400 / case["grid"] + 1) / 1.0
    surface = 2.0 * (case["nx"] * case["ny"] + case["ny"] * case["nz"] + case["nx"] * case["nz"]) * 16
    return {"bytes": 16.0 * nf + 8.0 * nodes + 36.0 * surface + 4.0 * 800 * 400,
            "flops": nf * (8 / case["grid"]) ** 3 * 0.52 * 15.0}


# ------------------------------------------------------------------------- the same in 64 bits
def _row_pairs(xa, xb, h):
    """All (a, b) with |xa - xb| < h, sorted by a: index tensors."""
    lo = torch.minimum(xa.min(0).values, xb.min(0).values) - 2.0 * h
    n = ((torch.maximum(xa.max(0).values, xb.max(0).values) - lo) / h).floor().long() + 3
    cell = lambda x: ((x - lo) / h).floor().long()  # noqa: E731
    cb = cell(xb)
    kb, order = torch.sort(cb[:, 0] + n[0] * (cb[:, 1] + n[1] * cb[:, 2]))
    ca = cell(xa)
    ii, jj = [], []
    rows = torch.arange(len(xa), device=xa.device)
    for dz in (-1, 0, 1):
        for dy in (-1, 0, 1):
            k = ca[:, 0] + n[0] * (ca[:, 1] + dy + n[1] * (ca[:, 2] + dz))
            first, last = torch.searchsorted(kb, k - 1), torch.searchsorted(kb, k + 1, right=True)
            count = last - first
            i = torch.repeat_interleave(rows, count)
            at = torch.arange(len(i), device=xa.device) - torch.repeat_interleave(count.cumsum(0) - count, count)
            j = order[first[i] + at]
            near = ((xa[i] - xb[j]) ** 2).sum(1) < h * h
            ii.append(i[near])
            jj.append(j[near])
    return torch.cat(ii), torch.cat(jj)


def _w(r, h):
    q = r / h
    w = torch.where(q <= 0.5, 6.0 * (q ** 3 - q ** 2) + 1.0, 2.0 * (1.0 - q).clamp(min=0.0) ** 3)
    return 8.0 / (math.pi * h ** 3) * w


def _grad(dx, h):
    r = dx.norm(dim=1)
    q = r / h
    g = torch.where(q <= 0.5, q * (3.0 * q - 2.0), -((1.0 - q).clamp(min=0.0) ** 2))
    return (48.0 / (math.pi * h ** 4) * g / r.clamp(min=1e-300))[:, None] * dx


class _Exact:
    """One scene of walls and fluid in 64 bits: the step of the framework's documentation."""

    def __init__(self, d, q):
        t = lambda a: torch.from_numpy(np.asarray(a)).cuda().double()  # noqa: E731
        r32 = lambda k: float(np.float32(d[k]))  # noqa: E731
        self.d = {k: r32(k) for k in ("radius", "rest_density", "viscosity", "dt_max", "cfl", "eta_density",
                                      "eta_divergence", "cg_tol", "eos_stiffness", "xsph_c")}
        self.h = 4.0 * self.d["radius"]
        self.m = self.d["rest_density"] * (2.0 * self.d["radius"]) ** 3
        self.g = t(np.asarray(d["gravity"], np.float32))
        self.desc = d
        self.x, self.v, self.kp, self.kvp = (q[k].double() for k in ("x", "v", "kp", "kvp"))
        self.xb = t(d["boundary_x"])
        self.n = len(self.x)
        i, j = _row_pairs(self.xb, self.xb, self.h)
        self.psi = self.d["rest_density"] / self.total(_w((self.xb[i] - self.xb[j]).norm(dim=1), self.h), i, len(self.xb))
        self.dt_next = self.cfl()

    def cfl(self):
        dt, vm = self.d["dt_max"], float(self.v.norm(dim=1).max())
        return min(dt, self.d["cfl"] * 2.0 * self.d["radius"] / vm) if self.d["cfl"] > 0 and vm > 0 else dt

    @staticmethod
    def total(values, index, n):
        out = torch.zeros((n,) + values.shape[1:], dtype=torch.float64, device=values.device)
        return out.index_add_(0, index, values)

    def drho(self, v):
        f = self.m * ((v[self.i] - v[self.j]) * self.gw).sum(1)
        return self.total(f, self.i, self.n) + self.total((v[self.bi] * self.gb).sum(1), self.bi, self.n)

    def push(self, v, k, dt):
        a = self.total(self.m * (k[self.i] + k[self.j])[:, None] * self.gw, self.i, self.n)
        return v - dt * (a + self.total(k[self.bi][:, None] * self.gb, self.bi, self.n))

    def viscous(self, v):
        u = v[self.i] - v[self.j]
        dx = self.x[self.i] - self.x[self.j]
        f = (u * dx).sum(1) / (((dx ** 2).sum(1) + 0.01 * self.h ** 2) * self.rho[self.j])
        mu = self.d["viscosity"] * self.d["rest_density"]
        return 10.0 * mu * self.m / self.rho[:, None] * self.total(f[:, None] * self.gw, self.i, self.n)

    def implicit(self, b, dt):
        apply = lambda p: p - dt * self.viscous(p)  # noqa: E731
        x, r = b.clone(), b - apply(b)
        p, rr, bb = r.clone(), (r ** 2).sum(), (b ** 2).sum()
        it = 0
        while it < self.desc["cg_max_iter"] and float(rr) > self.d["cg_tol"] ** 2 * float(bb):
            ap = apply(p)
            a = rr / (p * ap).sum()
            x, r = x + a * p, r - a * ap
            old, rr = rr, (r ** 2).sum()
            p, it = r + rr / old * p, it + 1
        return x

    def step(self):
        d, rho0, dt = self.desc, self.d["rest_density"], self.dt_next
        self.i, self.j = _row_pairs(self.x, self.x, self.h)
        off = self.i != self.j
        self.i, self.j = self.i[off], self.j[off]
        self.bi, bj = _row_pairs(self.x, self.xb, self.h)
        dx, db = self.x[self.i] - self.x[self.j], self.x[self.bi] - self.xb[bj]
        self.gw, self.gb = _grad(dx, self.h), self.psi[bj][:, None] * _grad(db, self.h)
        self.rho = (self.m * 8.0 / (math.pi * self.h ** 3) + self.total(self.m * _w(dx.norm(dim=1), self.h), self.i, self.n)
                    + self.total(self.psi[bj] * _w(db.norm(dim=1), self.h), self.bi, self.n))
        s1 = self.total(self.m * self.gw, self.i, self.n) + self.total(self.gb, self.bi, self.n)
        den = (s1 ** 2).sum(1) + self.total((self.m * self.gw).pow(2).sum(1), self.i, self.n)
        small = 1e-6 * (self.m * 48.0 / (math.pi * self.h ** 4)) ** 2
        alpha = torch.where(den > small, self.rho / den.clamp(min=1e-300), torch.zeros_like(den))
        solver, warm = d["pressure_solver"], d["warm_start"] != 0 and d["pressure_solver"] == 0
        v = self.v
        kvsum = torch.zeros_like(self.rho)
        if d["divergence_solve"] and solver == 0:
            if warm:
                kvsum = torch.where(self.drho(v) > 0, 0.5 * self.kvp / dt, kvsum)
                v = self.push(v, kvsum / self.rho, dt)
            it, err = 0, math.inf
            while it < d["max_iter_divergence"] and (it < d["min_iter_divergence"] or err > self.d["eta_divergence"]):
                e = self.drho(v).clamp(min=0.0)
                k = alpha * e / dt
                kvsum, v = kvsum + k, self.push(v, k / self.rho, dt)
                it, err = it + 1, float(e.mean()) / rho0 * dt
        acceleration = self.g.expand_as(v)
        if d["viscosity_mode"] == scenes.VISC_EXPLICIT:
            acceleration = acceleration + self.viscous(v)
        star = v + dt * acceleration
        if d["viscosity_mode"] == scenes.VISC_XSPH:
            w = self.m / self.rho[self.j] * _w(dx.norm(dim=1), self.h)
            star = star + self.d["xsph_c"] * self.total(w[:, None] * (v[self.j] - v[self.i]), self.i, self.n)
        v = self.implicit(star, dt) if d["viscosity_mode"] == scenes.VISC_IMPLICIT else star
        ksum = torch.zeros_like(self.rho)
        if solver == 1:
            gamma = float(np.float32(d["eos_exponent"]))
            ksum = (self.d["eos_stiffness"] * ((self.rho / rho0) ** gamma - 1.0)).clamp(min=0.0) / self.rho
            v = self.push(v, ksum / self.rho, dt)
        elif warm:
            ksum = torch.where(self.rho + dt * self.drho(v) > rho0, 0.5 * self.kp / dt ** 2, ksum)
            v = self.push(v, ksum / self.rho, dt)
        it, err = 0, math.inf
        while solver != 1 and it < d["max_iter_density"] and (it < d["min_iter_density"] or err > self.d["eta_density"]):
            dev = self.rho + dt * self.drho(v) - rho0
            e = dev.clamp(min=0.0)
            if solver == 2:
                old = ksum
                ksum = (ksum * self.rho + self.prototype() / dt ** 2 * dev).clamp(min=0.0) / self.rho
                k = ksum - old
            else:
                k = alpha * e / dt ** 2
                ksum = ksum + k
            v = self.push(v, k / self.rho, dt)
            it, err = it + 1, float(e.mean()) / rho0
        self.v, self.x = v, self.x + dt * v
        self.kp, self.kvp = ksum * dt * dt, kvsum * dt
        self.dt_next = self.cfl()

    def prototype(self):
        """The predictive-corrective stiffness times dt^2, of a full lattice neighbourhood."""
        s = 2.0 * self.d["radius"]
        a = torch.arange(-3, 4, dtype=torch.float64, device="cuda") * s
        p = torch.cartesian_prod(a, a, a)
        p = p[(p.norm(dim=1) > 0) & (p.norm(dim=1) <= self.h)]
        return 1.0 / (2.0 * (s ** 3) ** 2 * float((_grad(p, self.h) ** 2).sum()))


def _exact_mlp(params, f):
    w = params.double()
    cut = lambda o, *shape: w[o:o + math.prod(shape)].reshape(shape)  # noqa: E731
    p = [cut(0, 64, 4), cut(256, 64), cut(320, 64, 64), cut(4416, 64), cut(4480, 64), cut(4544, 1)]
    p = [t.clone().requires_grad_(True) for t in p]
    a = torch.nn.functional.gelu(f.double() @ p[0].T + p[1])
    return torch.nn.functional.gelu(a @ p[2].T + p[3]) @ p[4] + p[5], p


def exact(case, seed):
    k = case["kind"]
    if k == "step":
        if case["scene"] == "rigid":
            return None  # moving bodies: their boundary particles' update is no plain sum
        out = []
        for i, d in enumerate(_descs(case, seed)):
            e = _Exact(d, _start_state(d, seed * 1000 + i))
            for _ in range(case["steps"]):
                e.step()
            out.append({"x": e.x, "v": e.v, "rho": e.rho})
            del e
        return {"scenes": out, "poses": []}
    if k == "mlp_forward":
        with torch.no_grad():
            f, _ = _mlp_data(case["n"], seed)
            return torch.cat([_exact_mlp(_mlp_params(seed), q)[0] for q in f.split(1 << 18)])
    if k == "mlp_grad":
        f, y = _mlp_data(case["n"], seed)
        out, p = _exact_mlp(_mlp_params(seed), f)
        e = out - y.double()
        (e ** 2).mean().backward()
        return {"grad": torch.cat([t.grad.reshape(-1) for t in p]), "loss": (e.detach() ** 2).sum().reshape(1)}
    if k == "post":
        d = scenes.dam_break_rigid(seed=seed, n=(case["nx"], case["ny"], case["nz"]), n_boxes=0)
        return {"field": _exact_field(d, _start_state(d, seed)["x"].double(), d["radius"] * case["grid"]),
                "triangles": None, "count": None, "image": None}
    return None  # whole numbers, or mini-batches that depend on the library's own order


def _exact_field(d, x, spacing):
    dims = [int((d["domain_max"][a] - d["domain_min"][a]) / spacing) + 1 for a in range(3)]
    sp = float(np.float32(spacing))
    volume, h = (2.0 * float(np.float32(d["radius"]))) ** 3, 4.0 * float(np.float32(d["radius"]))
    reach = int(math.ceil(h / sp))
    out = torch.zeros(dims[0] * dims[1] * dims[2], dtype=torch.float64, device="cuda")
    base = (x / sp).round().long()
    span = range(-reach, reach + 1)
    for dz in span:
        for dy in span:
            for dx in span:
                n = base + torch.tensor([dx, dy, dz], device="cuda")
                ok = ((n >= 0) & (n < torch.tensor(dims, device="cuda"))).all(1)
                r = (n * sp - x).norm(dim=1)
                ok &= r < h
                n = n[ok]
                out.index_add_(0, n[:, 0] + dims[0] * (n[:, 1] + dims[1] * n[:, 2]), volume * _w(r[ok], h))
    return out.reshape(dims[2], dims[1], dims[0])

