"""What the substep library is used for, as cases that can be timed and checked.

A pass is one frame of a host program: the particle state is set (a rollout
that starts again from a given state), the tools get their pose and velocity,
the scene advances by a number of substeps, and the new state is read.  The
exceptions are the differentiable trajectory (forward and backward through
``autograd.trajectory``) and the frames whose state lives in pinned host memory.

States are those met in the middle of a simulation: a soft block close to the
floor, in motion, with deformation gradients away from the identity.
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_2502_18437_gb300 import mpm, workloads

BOUND = 3          # wall thickness in nodes
BOTTOM = 3.3       # cells below the block: it touches the floor's stencils
YIELD = 50.0       # von Mises yield of the plastic blocks (Pa)
SPEED = {"fall": 2.0, "rest": 0.05}


def _case(name, n, count, *, substeps, dt, model="fixed_corotated", plastic=False, E=1e4, nu=0.3, rho=1000.0,
          ppc=8.0, flat=1.0, fill="uniform", varied=False, tools="none", solver="mls", cycles=0, motion="fall",
          io="device", scenes=1, low=0, layout=0, checkpoint=0):
    c = dict(name=name, n=n, count=count, substeps=substeps, dt=dt, model=model, plastic=plastic, E=E, nu=nu, rho=rho,
             ppc=ppc, flat=flat, fill=fill, varied=varied, tools=tools, solver=solver, cycles=cycles, motion=motion,
             io=io, scenes=scenes, low=low, layout=layout, checkpoint=checkpoint)
    if name is None:
        del c["name"]
    return c


def listed():
    return [
        # the smallest scene in use: the elastic cube of the oracle comparison, where launches and latency count
        _case("cube_4k", 32, 4096, substeps=20, dt=1e-4, rho=1.0, fill="jitter"),
        # the falling cube of the paper's speed comparison (56^3 grid, ten substeps a rendered step), smallest count
        _case("paper_cube_16k", 56, 16384, substeps=10, dt=2e-3, model="neo_hookean", E=3e3, ppc=1.46),
        # tissue blocks with plastic flow hitting the floor: the scale sweep from small to the largest
        _case("block_64k", 64, 65536, substeps=25, dt=5e-5, plastic=True),
        _case("block_1m", 256, 1048576, substeps=25, dt=5e-5, plastic=True),
        _case("block_4m", 256, 4194304, substeps=10, dt=5e-5, plastic=True),
        # a cutting and suturing scene: a slab of uneven material with a moving blade and a thread
        _case("slab_256k", 128, 262144, substeps=25, dt=1e-4, model="neo_hookean", nu=0.4, ppc=5.0, flat=0.2,
              fill="jitter", varied=True, tools="blade_thread", motion="rest"),
        # an indenter pressing into a block: solid contact with push-out, an odd count on a grid that is no power of two
        _case("indenter_100k", 96, 100003, substeps=25, dt=1e-4, ppc=7.0, flat=0.6, tools="sphere", motion="rest"),
        # the paper's two other solvers on its timing scene
        _case("standard_131k", 56, 131072, substeps=10, dt=2e-3, model="neo_hookean", E=3e3, ppc=11.66,
              solver="standard"),
        _case("pb_131k", 56, 131072, substeps=2, dt=2e-2, model="fixed_corotated", E=3e3, ppc=11.66, solver="pb",
              cycles=10, motion="rest"),
        # many training environments of uneven size, each with its blade, in one context
        _case("batched_256", 64, 32768, substeps=100, dt=1e-4, flat=0.5, tools="blade", motion="rest", scenes=256,
              low=2048, layout=4),
        # gradients of a trajectory with respect to the material and the initial velocity
        _case("gradient_32k", 64, 32768, substeps=40, dt=1e-4, fill="lattice", varied=True, checkpoint=20,
              motion="rest"),
        # a host-resident simulation: the whole state comes from pinned host memory and goes back every frame
        _case("host_1m", 256, 1048576, substeps=25, dt=5e-5, plastic=True, io="host"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["block", "block", "tools", "solver", "batched", "gradient", "host"])
    model = rng.choice(["fixed_corotated", "neo_hookean"])
    nu = round(rng.uniform(0.2, 0.42), 3)
    E = round(_log(rng, 3e3, 2e4), 1)
    rho = 1000.0
    ppc = round(rng.uniform(4.0, 14.0), 2)
    flat = round(rng.uniform(0.3, 1.0), 2)
    top = {"block": 2.5e6, "tools": 6e5, "solver": 3e5, "batched": 20000, "gradient": 60000, "host": 1.2e6}[kind]
    count = int(_log(rng, 2500, top)) | 1
    side = (count / ppc / flat) ** (1.0 / 3.0)
    least = max(32, int(side / 0.7) + 1)
    n = min(256, 4 * math.ceil(least * rng.uniform(1.0, 1.5) / 4))
    speed = math.sqrt(E * (1 - nu) / ((1 + nu) * (1 - 2 * nu)) / rho)
    dt = float("%.2g" % (min(0.15 / (n * speed), 0.04 / (n * SPEED["fall"]))))
    substeps = rng.randint(8, 30)
    motion = rng.choice(["fall", "rest"])
    fill = rng.choice(["uniform", "jitter"])
    more = {}
    if kind in ("block", "host"):
        more["plastic"] = rng.random() < 0.5
        more["varied"] = rng.random() < 0.3
        more["io"] = "host" if kind == "host" else "device"
    elif kind == "tools":
        more["tools"] = rng.choice(["blade", "blade_thread", "sphere"])
        more["varied"] = rng.random() < 0.5
    elif kind == "solver":
        more["solver"] = rng.choice(["standard", "pb"])
        more["cycles"] = rng.randint(4, 12) if more["solver"] == "pb" else 0
        if more["solver"] == "pb":
            substeps, dt, motion = rng.randint(1, 4), float("%.2g" % (0.4 / n)), "rest"
    elif kind == "batched":
        more.update(scenes=rng.randint(24, 160), low=2048, layout=rng.randint(0, 1 << 20), tools=rng.choice(["none", "blade"]))
        n, count, substeps = 64, max(count, 4097), rng.randint(20, 80)
    elif kind == "gradient":
        more.update(varied=True, checkpoint=rng.choice([8, 16, 20]))
        motion = "rest"
    return _case(None, n, count, substeps=substeps, dt=dt, model=model, E=E, nu=nu, rho=rho, ppc=ppc, flat=flat,
                 fill=fill, motion=motion, **more)


# ------------------------------------------------------------------ inputs

def _layout(case):
    """Particle counts and grid sizes of the scenes: by the case alone."""
    if case["scenes"] == 1:
        return [case["count"]], [case["n"]]
    r = random.Random(case["layout"])
    counts, grids = [], []
    for _ in range(case["scenes"]):
        k = int(round(_log(r, case["low"], case["count"])))
        counts.append(k)
        grids.append(case["n"] if k > case["count"] // 2 else r.choice([case["n"] // 2, case["n"]]))
    return counts, grids


def _scene(case, count, n, g, hostrng):
    """Positions, velocities, affine velocities, deformation gradients, material and tools of one scene."""
    dev, dx = "cuda", 1.0 / n
    rand = lambda *s: torch.rand(*s, generator=g, device=dev, dtype=torch.float32)
    randn = lambda *s: torch.randn(*s, generator=g, device=dev, dtype=torch.float32)
    a = (count / case["ppc"] / case["flat"]) ** (1.0 / 3.0)
    cells = torch.tensor([a, a * case["flat"], a], device=dev)
    if case["fill"] == "uniform":
        u = rand(count, 3)
    else:
        # one particle in each of the cells of a regular division of the block
        m = [max(1, round(float(c) * case["ppc"] ** (1.0 / 3.0))) for c in cells]
        m[1] = max(m[1], -(-count // (m[0] * m[2])))
        at = torch.arange(count, device=dev)
        ijk = torch.stack([at // (m[1] * m[2]), (at // m[2]) % m[1], at % m[2]], -1).float()
        ijk[:, 0] = torch.clamp(ijk[:, 0], max=m[0] - 1)
        u = (ijk + (0.5 if case["fill"] == "lattice" else rand(count, 3))) / torch.tensor(m, device=dev).float()
    size = cells * dx
    low = 0.5 - 0.5 * size + 0.13 * dx
    low[1] = 0.5 - 0.5 * size[1] if case["checkpoint"] else BOTTOM * dx
    x = low + u * size
    # smooth fields over the block: two waves each, and a little noise
    ph = 2 * math.pi * rand(4)
    s1 = torch.sin(5.0 * u[:, 0] + 3.0 * u[:, 1] + ph[0]) + torch.cos(4.0 * u[:, 2] + ph[1])
    s2 = torch.cos(6.0 * u[:, 1] - 2.0 * u[:, 2] + ph[2]) + torch.sin(3.0 * u[:, 0] + ph[3])
    A, B, P, Q = (randn(3, 3) for _ in range(4))
    d, w = randn(3), randn(3)
    eye = torch.eye(3, device=dev)
    F = eye + 0.01 * (s1[:, None, None] * A + s2[:, None, None] * B) + 0.002 * randn(count, 3, 3)
    C = s1[:, None, None] * P + s2[:, None, None] * Q
    v = 0.05 * (s1[:, None] * d + s2[:, None] * w) + 0.01 * randn(count, 3)
    v[:, 1] -= SPEED[case["motion"]]
    E = case["E"] * (0.5 + 1.5 * rand(count)) if case["varied"] else None
    nu = torch.full((count,), case["nu"], device=dev) if case["varied"] else None
    if case["checkpoint"]:
        nu = case["nu"] * (0.8 + 0.2 * rand(count))
        C, F = None, None
        v[:, 1] += SPEED[case["motion"]]
    V0 = float(np.float32(dx ** 3 / case["ppc"]))
    rigids = _tools(case, n, [float(t) for t in low], [float(t) for t in size], hostrng)
    return SimpleNamespace(x=x.contiguous(), v=v, C=C, F=F, E=E, nu=nu, V0=V0, n=n, rigids=rigids)


def _tools(case, n, low, size, r):
    dx, top = 1.0 / n, low[1] + size[1]
    mid = [low[i] + 0.5 * size[i] for i in range(3)]
    if case["tools"] == "none":
        return []
    if case["tools"] == "sphere":
        rad = 0.22 * size[0]
        at = (mid[0] + r.uniform(-0.1, 0.1) * size[0], top + 0.6 * rad, mid[2] + r.uniform(-0.1, 0.1) * size[2])
        return [workloads.sphere(at, rad, vel=(0.02, -0.2, 0.0), mu_k=0.3, margin=0.5 * dx)]
    yaw, depth = r.uniform(0.1, 1.4), 0.05
    half = yaw / 2
    qy, qb = (math.cos(half), 0.0, math.sin(half), 0.0), workloads.BLADE_EDGE_Z_DOWN
    quat = (qy[0] * qb[0] - qy[2] * qb[2], qy[0] * qb[1] + qy[2] * qb[3], qy[0] * qb[2] + qy[2] * qb[0],
            qy[0] * qb[3] - qy[2] * qb[1])
    at = (mid[0] + r.uniform(-0.1, 0.1) * size[0], top - 1.5 * dx + depth, mid[2] + r.uniform(-0.1, 0.1) * size[2])
    got = [workloads.quad_slicer(at, quat, half_edge=0.3 * size[0], half_depth=depth, thickness=0.002,
                                 vel=(0.0, -r.uniform(0.05, 0.2), 0.0), mu_k=0.3, c_d=1.0, margin=dx)]
    if case["tools"] == "blade_thread":
        length = 0.8 * size[0]
        pts = np.stack([np.linspace(-length / 2, length / 2, 33), 0.002 * np.sin(np.linspace(0, 9, 33)),
                        np.zeros(33)], -1)
        got.append(workloads.segments((mid[0], mid[1] + 0.29 * dx, mid[2] + r.uniform(0.1, 0.4) * dx), (1, 0, 0, 0), pts,
                                      radius=0.003, vel=(0.05, 0.0, 0.0), mu_k=0.3, c_d=1.0, margin=dx))
    return got


def _inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    r = random.Random(int(seed) ^ 0x5EED)
    counts, grids = _layout(case)
    return [_scene(case, k, n, g, r) for k, n in zip(counts, grids)]


FIELDS = ("x", "v", "C", "F")
SHAPES = {"x": (3,), "v": (3,), "C": (3, 3), "F": (3, 3)}


def prepare(case, seed):
    scenes = _inputs(case, seed)
    s = SimpleNamespace(case=case, scenes=scenes, stream=torch.cuda.Stream())
    torch.cuda.synchronize()
    if case["checkpoint"]:
        sc = scenes[0]
        s.target = sc.x.mean(0) + torch.tensor([0.01, -0.02, 0.015], device="cuda")
        torch.cuda.synchronize()
        return s
    counts = [len(sc.x) for sc in scenes]
    s.first = np.concatenate([[0], np.cumsum(counts)]).tolist()
    s.sim = mpm.Simulation(case["n"], s.first[-1], n_scenes=len(scenes),
                           scene_grid_n=[sc.n for sc in scenes] if len(scenes) > 1 else None, model=case["model"],
                           plasticity=case["plastic"], yield_stress=YIELD if case["plastic"] else 0.0,
                           solver=case["solver"], pb_iterations=case["cycles"] or 10, bound=BOUND,
                           stream=s.stream.cuda_stream)
    for i, sc in enumerate(scenes):
        s.sim.add_particles(i, sc.x, sc.v, sc.E, sc.nu, E0=0.0 if case["varied"] else case["E"],
                            nu0=0.0 if case["varied"] else case["nu"], rho=case["rho"], V0=sc.V0)
        for k, t in enumerate(sc.rigids):
            s.sim.set_rigid(i, k, t)
    if case["io"] == "host":
        s.given = {f: getattr(scenes[0], f).cpu().pin_memory() for f in FIELDS}
        s.got = {f: torch.empty_like(s.given[f]).pin_memory() for f in FIELDS}
    torch.cuda.synchronize()
    return s


def run(s):
    with torch.cuda.stream(s.stream):
        if s.case["checkpoint"]:
            return _run_gradient(s)
        if s.case["io"] == "host":
            return _run_host(s)
        return _run_frame(s)


def _run_frame(s):
    sim, case = s.sim, s.case
    for i, sc in enumerate(s.scenes):
        sim.write_state(i, x=sc.x, v=sc.v, C=sc.C, F=sc.F)
        for k, t in enumerate(sc.rigids):
            sim.set_rigid(i, k, t)
    sim.substep(case["dt"], case["substeps"])
    tools = case["tools"] != "none"
    if len(s.scenes) == 1:
        out = sim.read_state(0, FIELDS + (("impulse",) if tools else ()), device=True)
        impulse = out.pop("impulse").unsqueeze(0) if tools else None
    else:
        # the scenes' states side by side in one tensor a field
        out = {f: torch.empty((s.first[-1],) + SHAPES[f], device="cuda") for f in FIELDS}
        impulse = torch.empty((len(s.scenes), mpm.MAX_RIGIDS, 6), dtype=torch.float64, device="cuda") if tools else None
        for i in range(len(s.scenes)):
            ptrs = [out[f][s.first[i]:].data_ptr() for f in FIELDS] + ([impulse[i].data_ptr()] if tools else [])
            mask = sum(mpm.FIELD[f] for f in FIELDS) + (mpm.FIELD["impulse"] if tools else 0)
            status = mpm.mpm_read_state(sim.h, i, mask, ptrs, mpm.MEM_DEVICE)
            if status != mpm.MPM_OK:
                raise mpm.MPMError(status, "mpm_read_state")
    if tools:
        out["impulse"] = impulse.float()  # summed in single precision; what a force display takes
    return out


def _run_host(s):
    h, mask = s.sim.h, sum(mpm.FIELD[f] for f in FIELDS)
    mpm.mpm_write_state(h, 0, mask, [s.given[f].data_ptr() for f in FIELDS], mpm.MEM_HOST)
    s.sim.substep(s.case["dt"], s.case["substeps"])
    status = mpm.mpm_read_state(h, 0, mask, [s.got[f].data_ptr() for f in FIELDS], mpm.MEM_HOST)
    if status != mpm.MPM_OK:
        raise mpm.MPMError(status, "mpm_read_state")
    return dict(s.got)


def _loss(x, v, target):
    return ((x.mean(0) - target) ** 2).sum() + (v * v).sum() / x.shape[0]


def _run_gradient(s):
    from paper_2502_18437_gb300.autograd import trajectory

    sc, case = s.scenes[0], s.case
    E, nu, v0 = (t.detach().requires_grad_() for t in (sc.E, sc.nu, sc.v))
    x, v = trajectory(E, nu, v0, sc.x, n=case["n"], substeps=case["substeps"], dt=case["dt"], rho=case["rho"], V0=sc.V0,
                      model=case["model"], checkpoint_every=case["checkpoint"])
    gE, gnu, gv = torch.autograd.grad(_loss(x, v, s.target), (E, nu, v0))
    return {"x": x.detach(), "v": v.detach(), "dE": gE, "dnu": gnu, "dv0": gv}


def work(case):
    """Each substep reads the particle state (x, v, C, F: 96 B) and writes it once (a PB-MPM cycle v and C, 48 B, and
    reads all of it); setting and reading the state moves it once more each.  Operations a particle-substep: 27 nodes
    at 14 each in the scatter and 16 in the gather, 300 for the constitutive update.  The way back of a gradient reads
    the state and its adjoint, writes the adjoint and takes about three times the operations."""
    N, K = sum(_layout(case)[0]), case["substeps"]
    per = 27 * 30 + 300
    if case["checkpoint"]:
        return {"bytes": N * (K * (192 + 96 + 192) + 24 + 44), "flops": 4.0 * N * K * per}
    loops = K * max(1, case["cycles"])
    moved = K * 192 if not case["cycles"] else loops * (96 + 48) + K * 144
    return {"bytes": N * (moved + 192), "flops": float(N) * loops * per}


# ------------------------------------------- the same in 64 bits, in torch

def _mm(A, B):
    return (A.unsqueeze(-1) * B.unsqueeze(-3)).sum(-2)


def _cof(F):
    a = [[F[:, i, j] for j in range(3)] for i in range(3)]
    m = lambda p, q, r, s: a[p][r] * a[q][s] - a[p][s] * a[q][r]
    return torch.stack([m(1, 2, 1, 2), -m(1, 2, 0, 2), m(1, 2, 0, 1), -m(0, 2, 1, 2), m(0, 2, 0, 2), -m(0, 2, 0, 1),
                        m(0, 1, 1, 2), -m(0, 1, 0, 2), m(0, 1, 0, 1)], -1).reshape(-1, 3, 3)


def _det(F):
    return (F[:, 0] * _cof(F)[:, 0]).sum(-1)


def _polar(F):
    """Rotation of F = R S by the Newton iteration R <- (R + R^-T) / 2."""
    R = F
    for _ in range(8):
        K = _cof(R)
        R = 0.5 * (R + K / (R[:, 0] * K[:, 0]).sum(-1)[:, None, None])
    return R


def _eigen(A):
    """Eigenvalues and vectors of symmetric 3x3 matrices: cyclic Jacobi."""
    a = {(i, j): A[:, i, j].clone() for i in range(3) for j in range(i, 3)}
    U = [[torch.full_like(a[0, 0], float(i == j)) for j in range(3)] for i in range(3)]
    for _ in range(6):
        for p, q in ((0, 1), (0, 2), (1, 2)):
            k = 3 - p - q
            apq = a[p, q]
            th = (a[q, q] - a[p, p]) / torch.where(apq == 0, torch.ones_like(apq), 2 * apq)
            t = torch.where(th >= 0, 1.0, -1.0) / (th.abs() + torch.sqrt(th * th + 1))
            t = torch.where(apq == 0, torch.zeros_like(t), t)
            c = 1 / torch.sqrt(t * t + 1)
            s = t * c
            a[p, p], a[q, q] = a[p, p] - t * apq, a[q, q] + t * apq
            a[p, q] = torch.zeros_like(apq)
            kp, kq = tuple(sorted((k, p))), tuple(sorted((k, q)))
            a[kp], a[kq] = c * a[kp] - s * a[kq], s * a[kp] + c * a[kq]
            for i in range(3):
                U[i][p], U[i][q] = c * U[i][p] - s * U[i][q], s * U[i][p] + c * U[i][q]
    return torch.stack([a[i, i] for i in range(3)], -1), torch.stack([torch.stack(r, -1) for r in U], -2)


def _return_map(F, mu):
    l, U = _eigen(_mm(F, F.transpose(1, 2)))
    e = 0.5 * torch.log(l)
    dev = e - e.mean(-1, keepdim=True)
    size = dev.norm(dim=-1)
    gamma = torch.clamp(size - float(np.float32(YIELD)) / (2 * mu), min=0.0)
    new = -(gamma / torch.where(size > 0, size, torch.ones_like(size)))[:, None] * dev
    return _mm(_mm(U * torch.exp(new)[:, None, :], U.transpose(1, 2)), F)


def _stress(model, F, mu, lam):
    eye = torch.eye(3, dtype=F.dtype, device=F.device)
    J = _det(F)
    mu = mu[:, None, None]
    if model == "neo_hookean":
        return mu * (_mm(F, F.transpose(1, 2)) - eye) + (lam * torch.log(J))[:, None, None] * eye
    return 2 * mu * _mm(F - _polar(F), F.transpose(1, 2)) + (lam * (J - 1) * J)[:, None, None] * eye


class _Sim64:
    """The scenes of a case in 64 bits: one list of particles, one list of nodes."""

    def __init__(self, case, scenes):
        f64 = lambda t: t.double()
        dev = "cuda"
        self.case, self.keep_graph = case, bool(case["checkpoint"])
        sid = torch.cat([torch.full((len(s.x),), i, device=dev) for i, s in enumerate(scenes)])
        ns = torch.tensor([s.n for s in scenes], device=dev)
        self.starts = torch.cumsum(ns ** 3, 0) - ns ** 3
        self.nodes = int((ns ** 3).sum())
        self.ns, self.n, self.start = ns, ns[sid].double(), self.starts[sid]
        self.ni = ns[sid]
        self.V0 = torch.tensor([s.V0 for s in scenes], dtype=torch.float64, device=dev)[sid]
        self.m = self.V0 * float(np.float32(case["rho"]))
        self.x, self.v = (torch.cat([f64(getattr(s, f)) for s in scenes]) for f in ("x", "v"))
        N = len(self.x)
        eye = torch.eye(3, dtype=torch.float64, device=dev).repeat(N, 1, 1)
        self.C = torch.cat([f64(s.C) for s in scenes]) if scenes[0].C is not None else torch.zeros_like(eye)
        self.F = torch.cat([f64(s.F) for s in scenes]) if scenes[0].F is not None else eye
        full = lambda v: torch.full((N,), float(np.float32(v)), dtype=torch.float64, device=dev)
        self.E = torch.cat([f64(s.E) for s in scenes]) if case["varied"] else full(case["E"])
        self.nu = torch.cat([f64(s.nu) for s in scenes]) if case["varied"] else full(case["nu"])
        self.rigids = [_Rigids([s.rigids[k] for s in scenes], dev) for k in range(len(scenes[0].rigids))]
        self.impulse = torch.zeros((len(scenes), mpm.MAX_RIGIDS, 6), dtype=torch.float64, device=dev)
        self.sid, self.t = sid, 0.0

    def weights(self):
        xs = self.x * self.n[:, None]
        base = torch.floor(xs.detach() - 0.5)
        f = xs - base
        w = [0.5 * (1.5 - f) ** 2, 0.75 - (f - 1) ** 2, 0.5 * (f - 0.5) ** 2]
        dw = [f - 1.5, -2 * (f - 1), f - 0.5]
        b = base.long()
        return (b[:, 0] * self.ni + b[:, 1]) * self.ni + b[:, 2] + self.start, f, w, dw

    def stencil(self):
        for i in range(3):
            for j in range(3):
                for k in range(3):
                    yield (i, j, k), (i * self.ni + j) * self.ni + k

    def scatter(self, A, w, dw, f, node, force):
        G = torch.zeros((self.nodes, 4), dtype=torch.float64, device="cuda")
        mv = self.m[:, None] * self.v
        for (i, j, k), off in self.stencil():
            W = (w[i][:, 0] * w[j][:, 1] * w[k][:, 2])[:, None]
            if force is None:
                d = (torch.tensor([i, j, k], device="cuda") - f) / self.n[:, None]
                mom = W * (mv + (A * d[:, None, :]).sum(-1))
            else:
                g = torch.stack([dw[i][:, 0] * w[j][:, 1] * w[k][:, 2], w[i][:, 0] * dw[j][:, 1] * w[k][:, 2],
                                 w[i][:, 0] * w[j][:, 1] * dw[k][:, 2]], -1) * self.n[:, None]
                mom = W * mv - (force * g[:, None, :]).sum(-1)
            val = torch.cat([W * self.m[:, None], mom], -1)
            G = G.index_add(0, node + off, val) if self.keep_graph else G.index_add_(0, node + off, val)
        return G

    def grid(self, G, gravity, dt):
        act = torch.nonzero(G[:, 0].detach() > 0)[:, 0]
        g = G[act]
        m = g[:, :1]
        v = g[:, 1:] / m
        v = torch.stack([v[:, 0], v[:, 1] + dt * gravity, v[:, 2]], -1)
        sc = torch.bucketize(act, self.starts, right=True) - 1
        n, loc = self.ns[sc], act - self.starts[sc]
        idx = torch.stack([loc // (n * n), (loc // n) % n, loc % n], -1)
        for r, rig in enumerate(self.rigids):
            x = idx.double() / n[:, None]
            vn, d, arm = rig.contact(x, sc, v, self.t)
            dp = -m * d
            v = vn
            self.impulse[:, r].index_add_(0, sc, torch.cat([dp, torch.cross(arm, dp, dim=-1)], -1))
        lo, hi = idx < BOUND, idx > (n - 1 - BOUND)[:, None]
        v = torch.where(lo, torch.clamp(v, min=0.0), v)
        v = torch.where(hi, torch.clamp(v, max=0.0), v)
        v = torch.where(lo[:, 1:2], torch.zeros_like(v), v)
        return torch.zeros((self.nodes, 3), dtype=torch.float64, device="cuda").index_put((act,), v)

    def gather(self, V, w, dw, f, node, standard):
        v = torch.zeros_like(self.v)
        B = torch.zeros_like(self.C)
        for (i, j, k), off in self.stencil():
            vi = V[node + off]
            W = (w[i][:, 0] * w[j][:, 1] * w[k][:, 2])[:, None]
            v = v + W * vi
            if standard:
                g = torch.stack([dw[i][:, 0] * w[j][:, 1] * w[k][:, 2], w[i][:, 0] * dw[j][:, 1] * w[k][:, 2],
                                 w[i][:, 0] * w[j][:, 1] * dw[k][:, 2]], -1)
            else:
                g = 4 * W * (torch.tensor([i, j, k], device="cuda") - f)
            B = B + vi[:, :, None] * (g * self.n[:, None])[:, None, :]
        return v, B

    def material(self):
        return self.E / (2 * (1 + self.nu)), self.E * self.nu / ((1 + self.nu) * (1 - 2 * self.nu))

    def integrate(self, dt, mu):
        self.x = self.x + dt * self.v
        self.F = self.F + dt * _mm(self.C, self.F)
        if self.case["plastic"]:
            self.F = _return_map(self.F, mu)
        self.t += dt
        for rig in self.rigids:
            self.x = rig.push_out(self.x, self.sid, self.t)

    def substep(self, dt, gravity):
        case = self.case
        mu, lam = self.material()
        node, f, w, dw = self.weights()
        if case["solver"] == "pb":
            cycles = case["cycles"] or 10
            for c in range(cycles):
                A = self.m[:, None, None] * self.constraint(dt)
                V = self.grid(self.scatter(A, w, dw, f, node, None), gravity if c == 0 else 0.0, dt)
                self.v, self.C = self.gather(V, w, dw, f, node, False)
            self.integrate(dt, mu)
            return
        tau = _stress(case["model"], self.F, mu, lam)
        standard = case["solver"] == "standard"
        if standard:
            G = self.scatter(None, w, dw, f, node, dt * self.V0[:, None, None] * tau)
        else:
            A = self.m[:, None, None] * self.C - (dt * self.V0 * 4 * self.n ** 2)[:, None, None] * tau
            G = self.scatter(A, w, dw, f, node, None)
        V = self.grid(G, gravity, dt)
        self.v, self.C = self.gather(V, w, dw, f, node, standard)
        self.integrate(dt, mu)

    def constraint(self, dt):
        """PB-MPM with beta = 1: C <- (R F^-1 - I) / dt with R the rotation of (I + dt C) F."""
        R = _polar(self.F + dt * _mm(self.C, self.F))
        K = _cof(self.F)
        inv = K.transpose(1, 2) / (self.F[:, 0] * K[:, 0]).sum(-1)[:, None, None]
        return (_mm(R, inv) - torch.eye(3, dtype=R.dtype, device=R.device)) / dt


class _Rigids:
    """The same tool slot of every scene (they move without turning)."""

    def __init__(self, descs, dev):
        # single precision, as they are given to the library
        t = lambda key: torch.tensor(np.array([np.asarray(d[key], np.float32) for d in descs], np.float64), device=dev)
        self.type = descs[0]["type"]
        self.c, self.vel, self.mu, self.cd, self.margin = (t(k) for k in ("center", "vel", "mu_k", "c_d", "margin"))
        q = t("quat")
        w, x, y, z = (q / q.norm(dim=-1, keepdim=True)).unbind(-1)
        self.R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                              1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                              1 - 2 * (x * x + y * y)], -1).reshape(-1, 3, 3)
        if self.type == "quad_slicer":
            self.half, self.thick, self.spine = t("half"), t("thickness"), t("spine_radius")
        else:
            self.radius = t("radius")
        if self.type == "segments":
            self.pts = t("pts")[0]

    def region(self, p, sc):
        """Code (0 none, 1 surface, 2 line, 3 sticky), normal and tangent at points p of the body frame."""
        nrm, tan = torch.zeros_like(p), torch.zeros_like(p)
        code = torch.zeros(len(p), dtype=torch.long, device=p.device)
        margin = self.margin[sc]
        unit = lambda d: d / torch.where(d.norm(dim=-1, keepdim=True) > 0, d.norm(dim=-1, keepdim=True), torch.ones_like(d[:, :1]))
        if self.type == "sphere":
            hit = p.norm(dim=-1) - self.radius[sc] < margin
            return torch.where(hit, 1, 0), unit(p), tan
        if self.type == "quad_slicer":
            h = self.half[sc]
            es = torch.clamp(p[:, 0].abs() - h[:, 0], min=0)
            spine = torch.sqrt(es ** 2 + (p[:, 1] + h[:, 1]) ** 2 + p[:, 2] ** 2) < self.spine[sc] + margin
            q = torch.stack([torch.maximum(torch.minimum(p[:, 0], h[:, 0]), -h[:, 0]),
                             torch.maximum(torch.minimum(p[:, 1], h[:, 1]), -h[:, 1]), torch.zeros_like(es)], -1)
            d = p - q
            face = d.norm(dim=-1) < 0.5 * self.thick[sc] + margin
            flat = (p[:, 0].abs() <= h[:, 0]) & (p[:, 1].abs() <= h[:, 1])
            side = torch.stack([torch.zeros_like(es), torch.zeros_like(es), torch.where(p[:, 2] >= 0, 1.0, -1.0).double()], -1)
            code = torch.where(spine, 3, torch.where(face, 1, 0))
            return code, torch.where(flat[:, None], side, unit(d)), tan
        a, e = self.pts[:-1], self.pts[1:] - self.pts[:-1]
        u = torch.clamp(((p[:, None] - a) * e).sum(-1) / (e * e).sum(-1), 0, 1)
        d = p[:, None] - (a + u[..., None] * e)
        best, at = d.norm(dim=-1).min(1)
        code = torch.where(best < self.radius[sc] + margin, 2, 0)
        return code, unit(d[torch.arange(len(p), device=p.device), at]), unit(e)[at]

    def contact(self, x, sc, v, t):
        """New node velocities, their change, and the arm about the tool's centre."""
        arm = x - (self.c + t * self.vel)[sc]
        R = self.R[sc]
        code, nl, tl = self.region((R * arm[:, :, None]).sum(1), sc)
        n, tan = (R * nl[:, None, :]).sum(-1), (R * tl[:, None, :]).sum(-1)
        vr = self.vel[sc]
        e = v - vr
        vn = (e * n).sum(-1, keepdim=True)
        has = (n * n).sum(-1, keepdim=True) > 0
        vt = torch.where((code == 2)[:, None], (e * tan).sum(-1, keepdim=True) * tan, e - vn * n)
        lt = vt.norm(dim=-1, keepdim=True)
        scale = self.cd[sc][:, None] * torch.clamp(1 - self.mu[sc][:, None] * vn.abs() / torch.where(lt > 0, lt, torch.ones_like(lt)), min=0)
        new = vr + torch.where((code == 3)[:, None], torch.zeros_like(vt), scale * vt)
        on = (code[:, None] == 3) | ((code[:, None] > 0) & ~(has & (vn >= 0)))
        out = torch.where(on, new, v)
        return out, out - v, arm

    def push_out(self, x, sid, t):
        if self.type != "sphere":
            return x
        c = (self.c + t * self.vel)[sid]
        d = x - c
        l = d.norm(dim=-1, keepdim=True)
        r = self.radius[sid][:, None]
        return torch.where(l < r, c + r / l * d, x)


def exact(case, seed):
    scenes = _inputs(case, seed)
    s = _Sim64(case, scenes)
    dt, g = float(np.float32(case["dt"])), float(np.float32(-9.8))
    if not case["checkpoint"]:
        with torch.no_grad():
            for _ in range(case["substeps"]):
                s.substep(dt, g)
        out = {f: getattr(s, f) for f in FIELDS}
        if case["tools"] != "none":
            out["impulse"] = s.impulse
        return {f: t.cpu() for f, t in out.items()} if case["io"] == "host" else out
    E, nu, v0 = (t.detach().requires_grad_() for t in (s.E, s.nu, s.v))
    s.E, s.nu, s.v = E, nu, v0
    for _ in range(case["substeps"]):
        s.substep(dt, g)
    target = (scenes[0].x.mean(0) + torch.tensor([0.01, -0.02, 0.015], device="cuda")).double()
    gE, gnu, gv = torch.autograd.grad(_loss(s.x, s.v, target), (E, nu, v0))
    return {"x": s.x.detach(), "v": s.v.detach(), "dE": gE, "dnu": gnu, "dv0": gv}
