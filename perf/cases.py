"""Workloads of the PSM-LBM library, as a user's program runs them, for timing.

Each case is one kind of call sequence through the public Python API:

  step      a batch of time steps on caller-owned PDF buffers, then the
            force/torque series of every body (a production run's inner loop)
  adjoint   one gradient of the force/torque series on a kept handle: a
            recorded forward run and its backward pass
  autograd  the same through the torch.autograd.Function, a design iteration
  snapshot  density and velocity, the full state out, and a saved state in
            (output frames and checkpoint / restart), in device memory
  mesh      a closed triangle mesh voxelised into a body's geometry field

listed() holds fixed sizes, draw() more of the same ranges.  exact() computes
the same outputs in 64 bits with plain torch and numpy.
"""

from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2502_20049_gb300 import psm
from paper_2502_20049_gb300 import workloads as W
from paper_2502_20049_gb300.autograd import PSMTorque

DTYPE = {"fp64": torch.float64, "fp32": torch.float32, "fp16": torch.float16, "bf16": torch.bfloat16}
BYTES = {"fp64": 8, "fp32": 4, "fp16": 2, "bf16": 2}
FLUID_FLOPS = {("bgk", 19): 250, ("trt", 19): 250, ("bgk", 27): 360, ("trt", 27): 360, ("cumulant", 19): 480}

# lattice velocities in the library's direction order (D3Q19: the first 19)
C27 = ((0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
       (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
       (0, -1, 1), (1, 1, 1), (-1, -1, -1), (1, 1, -1), (-1, -1, 1), (1, -1, 1), (-1, 1, -1), (-1, 1, 1), (1, -1, -1))
W19 = (1 / 3, 1 / 18, 1 / 36)
W27 = (8 / 27, 2 / 27, 1 / 54, 1 / 216)
TRT_LAMBDA = 3.0 / 16.0


def weights(Q):
    return [(W19 if Q == 19 else W27)[sum(abs(k) for k in c)] for c in C27[:Q]]


def step_case(name, nx, ny, nz, Q=19, storage="fp32", streaming="aa", fluid="bgk", tau=0.55, solid=1, weighting=1,
              bc_z=1, u_in=0.04, body="rotors", free=False, steps=2):
    c = dict(kind="step", nx=nx, ny=ny, nz=nz, Q=Q, storage=storage, streaming=streaming, fluid=fluid, tau=tau,
             solid=solid, weighting=weighting, bc_z=bc_z, u_in=u_in, body=body, free=free, steps=steps)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest validation run (a sphere in an inflow, 64 bits): latency and launches count
        step_case("sphere_32_fp64", 32, 32, 32, storage="fp64", tau=0.8, u_in=0.01, body="sphere", steps=20),
        # a free body moving under the fluid's load in a small box, two-way coupled
        step_case("coupled_64x64x96_fp32", 64, 64, 96, fluid="trt", tau=0.8, solid=2, bc_z=0, u_in=0.0,
                  body="sphere", free=True, steps=20),
        # a reduced rotor run on a grid whose rows are no power of two
        step_case("rotors_96x96x120_q27_fp32", 96, 96, 120, Q=27, steps=20),
        # odd extents on every axis, 16-bit storage
        step_case("ellipsoid_203x117x151_fp16", 203, 117, 151, storage="fp16", streaming="twogrid", fluid="trt",
                  u_in=0.05, body="ellipsoid", steps=10),
        # the rotating-ellipsoid benchmark
        step_case("ellipsoid_256_fp32", 256, 256, 256, streaming="twogrid", fluid="trt", u_in=0.05,
                  body="ellipsoid", steps=8),
        # the cumulant operator, which the paper's performance runs use, in 16-bit storage
        step_case("cumulant_256_fp16", 256, 256, 256, storage="fp16", fluid="cumulant", u_in=0.05,
                  body="ellipsoid", steps=8),
        # the D3Q27 counter-rotating rotor benchmark
        step_case("rotors_512x512x640_q27_fp16", 512, 512, 640, Q=27, storage="fp16", steps=4),
        # the largest single-GPU run, 1.0e9 cells
        step_case("rotors_1024x1024x960_fp16", 1024, 1024, 960, storage="fp16", steps=4),
        # the adjoint benchmark's grid and body: forward and backward on a kept handle
        dict(name="adjoint_128_fp32", kind="adjoint", n=128, storage="fp32", fluid="trt", tau=0.55, steps=64, K=16),
        # one design iteration through torch.autograd: perturbation in a shell around the body
        dict(name="autograd_64_fp32", kind="autograd", n=64, storage="fp32", fluid="trt", tau=0.55, steps=32, K=8),
        # output frame, checkpoint and restart of a mid-size run
        dict(name="snapshot_256x256x192_fp32", kind="snapshot", nx=256, ny=256, nz=192, Q=19, storage="fp32",
             bc_z=1, u_in=0.05),
        # a body's surface mesh voxelised once per run
        dict(name="mesh_131k_s2", kind="mesh", extent=60.5, nu=512, nv=128, s=2),
    ]


def _extent(rng, lo, hi):
    """A grid extent: a multiple of 32 as often as any number."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(32, v // 32 * 32) if rng.random() < 0.5 else v


def draw(rng):
    kind = rng.choice(["step"] * 6 + ["adjoint", "autograd", "snapshot", "mesh"])
    if kind == "step":
        Q = rng.choice([19, 19, 27])
        storage = rng.choice(["fp32"] * 4 + ["fp16"] * 4 + ["bf16", "fp64"])
        top = 200 if storage == "fp64" else 480
        nx, ny, nz = (_extent(rng, 32, top) for _ in range(3))
        fluid = rng.choice(["bgk", "trt", "cumulant"] if Q == 19 else ["bgk", "trt"])
        free = rng.random() < 0.15
        body = "sphere" if free else rng.choice(["sphere", "ellipsoid", "rotors"])
        steps = 2 * max(1, min(10, (1 << 25) // (nx * ny * nz)))
        return step_case(None, nx, ny, nz, Q=Q, storage=storage, streaming=rng.choice(["aa", "twogrid"]), fluid=fluid,
                         tau=round(rng.uniform(0.7 if free else 0.6, 0.9), 3),
                         solid=rng.choice([1, 2] if free else [1, 2, 3]),
                         weighting=rng.choice([0, 1]), bc_z=0 if free else rng.choice([0, 1, 1]),
                         u_in=0.0 if free else round(rng.uniform(0.01, 0.05), 4), body=body, free=free, steps=steps)
    if kind in ("adjoint", "autograd"):
        K = rng.choice([4, 8, 16])
        return dict(kind=kind, n=_extent(rng, 40, 144 if kind == "adjoint" else 80),
                    storage=rng.choice(["fp32", "fp32", "fp16"]),
                    fluid=rng.choice(["bgk", "trt"]), tau=round(rng.uniform(0.6, 0.9), 3), steps=4 * K, K=K)
    if kind == "snapshot":
        nx, ny, nz = (_extent(rng, 40, 300) for _ in range(3))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, Q=rng.choice([19, 27]),
                    storage=rng.choice(["fp64", "fp32", "fp16", "bf16"]), bc_z=rng.choice([0, 1]),
                    u_in=round(rng.uniform(0.01, 0.05), 4))
    return dict(kind="mesh", extent=rng.randrange(12, 80) + 0.5, nu=rng.randrange(40, 600), nv=rng.randrange(20, 140),
                s=rng.choice([1, 2, 3]))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def initial(case, seed, dtype):
    """Shifted equilibrium PDFs [Q, nz, ny, nx] of a smooth flow: the inflow
    plus seeded waves of a few per cent of the speed of sound."""
    r = np.random.RandomState(seed % (1 << 32))
    Q, n = case["Q"], (case["nz"], case["ny"], case["nx"])
    dev = device()
    waves = []
    for k in range(4):  # rho, ux, uy, uz
        line = []
        for d in range(3):
            x = torch.arange(n[d], dtype=torch.float32, device=dev)
            line.append(torch.sin(x * (2 * math.pi * r.randint(1, 4) / n[d]) + r.uniform(0, 2 * math.pi)))
        waves.append((0.003 if k == 0 else 0.01 * r.uniform(0.5, 1.0), line))
    f = torch.empty((Q,) + n, dtype=dtype, device=dev)
    w = weights(Q)
    planes = max(1, (1 << 25) // (n[1] * n[2]))
    for z0 in range(0, n[0], planes):
        z1 = min(n[0], z0 + planes)
        v = [a * line[0][z0:z1, None, None] * line[1][None, :, None] * line[2][None, None, :] for a, line in waves]
        v[3] = v[3] + case["u_in"]
        base = -1.5 * (v[1] * v[1] + v[2] * v[2] + v[3] * v[3])
        for i, c in enumerate(C27[:Q]):
            e = base
            if i:
                cu = sum(v[k + 1] if c[k] > 0 else -v[k + 1] for k in range(3) if c[k])
                e = base + cu * (3.0 + 4.5 * cu)
            f[i, z0:z1] = w[i] * (v[0] + (1.0 + v[0]) * e)
    return f


def rotor_params(k, blades, phase, hand):
    return (20.0 * k, 40.0 * k, 120.0 * k, 24.0 * k, 4.0 * k, 60.0, 30.0, phase, float(blades), float(hand))


def bodies_of(case):
    """(shape kind, parameters, supersampling depth, centre, angular velocity) of every body."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    m = min(nx, ny, nz)
    if case["body"] == "sphere":
        return [(W.SPHERE, (0.1875 * m,), 3, (nx / 2, ny / 2, nz / 2), (0.0, 0.0, 0.004 if case["free"] else 0.0))]
    if case["body"] == "ellipsoid":
        a = (0.15625 * m, 0.078125 * m, 0.03125 * m)
        return [(W.ELLIPSOID, a, 2, (nx / 2, ny / 2, nz / 2), (0.0, 0.0, 0.008 / a[0]))]
    k = min(nx, ny, nz * 0.8) / 512.0
    om = 3e-4 / k
    z = (0.375, 0.625) if case["Q"] == 19 else (0.375, 0.5625)
    return [(W.ROTOR, rotor_params(k, 6, 0.0, 1), 2, (nx / 2, ny / 2, nz * z[0]), (0.0, 0.0, om)),
            (W.ROTOR, rotor_params(k, 5, math.pi / 5, -1), 2, (nx / 2, ny / 2, nz * z[1]), (0.0, 0.0, -om))]


def ball(case):
    """Mass and inertia of the free sphere: twenty times the fluid's density (explicit coupling stays
    stable over any number of steps)."""
    r = 0.1875 * min(case["nx"], case["ny"], case["nz"])
    mass = 20.0 * 4.0 / 3.0 * math.pi * r ** 3
    return mass, np.eye(3) * 0.4 * mass * r * r


_FIELDS = {}  # voxelised fields by shape: a program voxelises a body once and keeps the field


def field(kind, params, s):
    key = (kind, tuple(params), s)
    if key not in _FIELDS:
        _FIELDS[key] = psm.voxelize(kind, params, s)
    return _FIELDS[key]


def solver(case, bufs):
    cfg = psm.SolverConfig(case["nx"], case["ny"], case["nz"], Q=case["Q"], streaming=case.get("streaming", "aa"),
                           storage=case["storage"], fluid=case.get("fluid", "bgk"), tau=case.get("tau", 0.6),
                           trt_lambda=TRT_LAMBDA, solid=case.get("solid", 1), weighting=case.get("weighting", 1),
                           bc_z=case["bc_z"], u_in=(0.0, 0.0, case["u_in"]))
    return psm.Solver(cfg, buffers=bufs, keep=True)


def stored(case, f):
    """The populations a buffer holds, per direction: those that enter from a z ghost plane are not stored."""
    n = case["nz"]
    g = case["bc_z"] == 1
    return [f[i][(1 if g and c[2] > 0 else 0):(n - 1 if g and c[2] < 0 else n)] for i, c in enumerate(C27[:case["Q"]])]


def adjoint_case(case, u_in):
    """The adjoint benchmark's workload, its ellipsoid scaled with the grid."""
    k, n = case["n"] / 256.0, case["n"]
    return W.Case("adjoint", n, n, n, Q=19, storage=case["storage"], streaming="aa", fluid=case["fluid"],
                  tau=case["tau"], u_in=(0.0, 0.0, u_in), steps=case["steps"],
                  bodies=[W.BodyCase(W.ELLIPSOID, (80.0 * k, 40.0 * k, 16.0 * k), 2, (n / 2, n / 2, n / 2),
                                     omega=(0.0, 0.0, 2e-4))])


def adjoint_inputs(case, seed):
    """Inflow speed and the weights of the functional J = sum w . (force, torque)."""
    r = np.random.RandomState(seed % (1 << 32))
    return 0.05 * r.uniform(0.8, 1.0), r.standard_normal((case["steps"], 1, 6)) / case["steps"]


def shell(case, seed):
    """Perturbation of the solid fraction in a shell around the body's surface, zero elsewhere (not
    positive where the solid fraction is near 1, which it must not exceed)."""
    n, k = case["n"], case["n"] / 256.0
    g = torch.Generator().manual_seed(seed % (1 << 32))
    x = torch.arange(n, dtype=torch.float64) + 0.5 - n / 2
    lev = ((x[None, None, :] / (80 * k)) ** 2 + (x[None, :, None] / (40 * k)) ** 2 + (x[:, None, None] / (16 * k)) ** 2)
    d = 0.002 * torch.rand((n, n, n), generator=g, dtype=torch.float32)
    d = torch.where(lev < 1.3, -d, d)
    return torch.where((lev > 0.5) & (lev < 2.0), d, torch.zeros_like(d)).to(device())


def mesh(case, seed):
    """A bumpy closed torus, scaled onto the same box for every seed."""
    r = np.random.RandomState(seed % (1 << 32))
    u = (2 * np.pi * np.arange(case["nu"]) / case["nu"])[:, None]
    v = (2 * np.pi * np.arange(case["nv"]) / case["nv"])[None, :]
    tube = 0.35 * (1.0 + 0.1 * np.sin(5 * u + r.uniform(0, 6)) * np.cos(3 * v + r.uniform(0, 6)))
    p = np.stack([(1 + tube * np.cos(v)) * np.cos(u), (1 + tube * np.cos(v)) * np.sin(u),
                  tube * np.sin(v) + 0.2 * np.sin(2 * u + r.uniform(0, 6))], -1).reshape(-1, 3)
    p = (2 * (p - p.min(0)) / (p.max(0) - p.min(0)) - 1) * (case["extent"] * np.array([1.0, 1.0, 0.6]))
    i, j = np.meshgrid(np.arange(case["nu"]), np.arange(case["nv"]), indexing="ij")
    i1, j1 = (i + 1) % case["nu"], (j + 1) % case["nv"]
    a, b, c, d = (q[0] * case["nv"] + q[1] for q in ((i, j), (i1, j), (i1, j1), (i, j1)))
    t = np.stack([np.stack([a, b, c], -1), np.stack([a, c, d], -1)], 2).reshape(-1, 3)
    return p.astype(np.float32), t.astype(np.int32)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":
        f = initial(case, seed, DTYPE[case["storage"]])
        bufs = [f] if case["streaming"] == "aa" else [f, f.clone()]
        sol = solver(case, bufs)
        bodies = bodies_of(case)
        for b, (sh, params, s, centre, omega) in enumerate(bodies):
            sol.set_geometry(b, field(sh, params, s), np.eye(3), centre, omega, (0.0, 0.0, 0.0))
        if case["free"]:
            mass, inertia = ball(case)
            sol.set_body_dynamics(0, mass, inertia)
        return dict(case=case, sol=sol, out=stored(case, f), bodies=len(bodies))
    if kind == "adjoint":
        u_in, w = adjoint_inputs(case, seed)
        sol = psm.Solver.from_case(adjoint_case(case, u_in), geoms=_FIELDS)
        n = case["n"]
        return dict(case=case, sol=sol, u_in=u_in, w=w,
                    grad=torch.empty((n, n, n), dtype=torch.float64, device=device()))
    if kind == "autograd":
        u_in, _ = adjoint_inputs(case, seed)
        return dict(case=case, model=adjoint_case(case, u_in), delta=shell(case, seed).requires_grad_(),
                    omega=torch.tensor([0.0, 0.0, 2e-4], dtype=torch.float64, requires_grad=True),
                    u_in=torch.tensor([0.0, 0.0, u_in], dtype=torch.float64, requires_grad=True))
    if kind == "snapshot":
        f = initial(case, seed, DTYPE[case["storage"]])
        n = (case["nz"], case["ny"], case["nx"])
        new = dict(dtype=torch.float64, device=device())
        return dict(case=case, sol=solver(case, [f]), out=stored(case, f), saved=saved_state(case, seed),
                    rho=torch.empty(n, **new), u=torch.empty(n + (3,), **new),
                    f=torch.empty((case["Q"],) + n, **new))
    v, t = mesh(case, seed)
    return dict(case=case, v=v, t=t)


def saved_state(case, seed):
    """Another run's full state, unshifted, in 64 bits."""
    f = initial(case, seed + 1, torch.float64)
    for i, w in enumerate(weights(case["Q"])):
        f[i] += w
    return f


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        sol, n = state["sol"], case["steps"]
        t0 = sol.step_count
        sol.step(n)
        out = dict(f=state["out"], ft=[sol.force_torque(b, t0, n) for b in range(state["bodies"])])
        if case["free"]:
            out["body"] = sol.body_state(0)
        return out
    if kind == "adjoint":
        sol = state["sol"]
        sol.init_equilibrium(1.0, (0.0, 0.0, state["u_in"]))
        t0 = sol.step_count
        sol.record(case["K"], init_from_inflow=True)
        sol.step(case["steps"])
        ft = sol.force_torque(0, t0, case["steps"])
        ge, gw, gu = sol.backward(state["w"], grad_eps=state["grad"])
        return dict(ft=ft, grad_eps=ge, grad_omega=gw, grad_uin=gu)
    if kind == "autograd":
        J = PSMTorque.apply(state["delta"], state["omega"], state["u_in"], state["model"], case["steps"], case["K"])
        ge, gw, gu = torch.autograd.grad(J, (state["delta"], state["omega"], state["u_in"]))
        return dict(J=J.detach(), grad_eps=ge, grad_omega=gw, grad_uin=gu)
    if kind == "snapshot":
        sol = state["sol"]
        sol.macroscopic(state["rho"], state["u"])
        sol.get_state(state["f"])
        sol.set_state(state["saved"])
        return dict(rho=state["rho"], u=state["u"], state=state["f"], f=state["out"])
    g = psm.voxelize_mesh(state["v"], state["t"], case["s"])
    return dict(words=g.words().view(np.int64), dims=list(g.dims), lo=g.lo)


def work(case):
    """Bytes and operations of one pass: every PDF read and written once per
    step; backward reads the state and the adjoint field and writes the adjoint
    field and the gradient; exports and imports move their arrays once."""
    kind = case["kind"]
    if kind == "step":
        cells = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 2 * case["Q"] * BYTES[case["storage"]] * cells * case["steps"],
                "flops": FLUID_FLOPS[case["fluid"], case["Q"]] * cells * case["steps"]}
    if kind in ("adjoint", "autograd"):
        cells, b = case["n"] ** 3, BYTES[case["storage"]]
        return {"bytes": cells * (case["steps"] * (2 * 19 * b + 19 * b + 2 * 19 * 4 + 8) + 8),
                "flops": cells * case["steps"] * (250 + 500)}
    if kind == "snapshot":
        cells, Q, b = case["nx"] * case["ny"] * case["nz"], case["Q"], BYTES[case["storage"]]
        return {"bytes": cells * ((Q * b + 32) + (Q * b + 8 * Q) + (8 * Q + Q * b)), "flops": cells * 7 * Q}
    tri, e, n = 2 * case["nu"] * case["nv"], 2 * (case["extent"] + 1.5), 1 << case["s"]
    sub = e * e * (2 * (0.6 * case["extent"] + 1.5)) * n ** 3
    return {"bytes": tri * 12 + tri // 2 * 12 + sub / 8, "flops": 50 * tri}


# ---------------------------------------------------------------------------
# The same results in 64 bits, in plain torch and numpy
# ---------------------------------------------------------------------------
def pose(omega, n):
    wn = math.sqrt(sum(o * o for o in omega))
    if wn == 0.0:
        return np.eye(3)
    k, th = np.array(omega) / wn, wn * n
    K = np.array([[0, -k[2], k[1]], [k[2], 0, -k[0]], [-k[1], k[0], 0]])
    return math.cos(th) * np.eye(3) + math.sin(th) * K + (1 - math.cos(th)) * np.outer(k, k)


def half_extent(kind, p):
    if kind == W.SPHERE:
        return (p[0],) * 3
    if kind == W.ELLIPSOID:
        return p
    return (p[0] + p[2], p[0] + p[2], max(0.5 * p[1], 0.5 * math.hypot(p[3], p[4])))


class RefBody:
    """Sub-cell field of a body (as running sums) and its motion."""

    def __init__(self, kind, p, s, centre, omega):
        self.n, self.R, self.omega, self.v = 1 << s, np.array(centre, dtype=float), np.array(omega), np.zeros(3)
        self.Q0, self.spin = np.eye(3), tuple(omega)
        m = [int(math.floor(e)) + 2 for e in half_extent(kind, p)]
        self.lo = [-float(k) for k in m]
        dev = device()
        x, y, z = (-float(m[k]) + (torch.arange(2 * m[k] * self.n, dtype=torch.float64, device=dev) + 0.5) / self.n
                   for k in range(3))
        x, y = x[None, :], y[:, None]
        total = []
        for zz in z:  # layer by layer, running sums over y and x
            inside = self.inside(kind, p, x, y, zz)
            total.append(inside.to(torch.int32).cumsum(0, dtype=torch.int32).cumsum(1, dtype=torch.int32))
        self.S = torch.nn.functional.pad(torch.stack(total).cumsum(0, dtype=torch.int32), (1, 0, 1, 0, 1, 0))
        self.reach = math.sqrt(sum(k * k for k in m)) + 2.5

    @staticmethod
    def inside(kind, p, x, y, z):
        if kind == W.SPHERE:
            return x * x + y * y + z * z <= p[0] * p[0]
        if kind == W.ELLIPSOID:
            a, b, c = x / p[0], y / p[1], z / p[2]
            return a * a + b * b + c * c <= 1.0
        r_hub, hub_len, span, chord, thick, pitch, twist, phase, blades, hand = p
        r = torch.sqrt(x * x + y * y)
        hub = (r <= r_hub) & (z.abs() <= 0.5 * hub_len)
        beta = (pitch - twist * (r - r_hub) / span) * (math.pi / 180.0) * hand
        phi = torch.atan2(y.expand(r.shape), x.expand(r.shape))
        blade = torch.zeros_like(hub)
        for k in range(int(blades)):
            d = phi - (phase + 2.0 * math.pi * k / blades)
            t = r * (d - 2.0 * math.pi * torch.floor((d + math.pi) / (2.0 * math.pi)))
            xi, eta = t * beta.cos() + z * beta.sin(), -t * beta.sin() + z * beta.cos()
            blade |= (xi / (0.5 * chord)) ** 2 + (eta / (0.5 * thick)) ** 2 <= 1.0
        return hub | (blade & (r >= r_hub) & (r <= r_hub + span))

    def eps(self, dims, Qm):
        """(box of cells, solid fraction in it) at orientation Qm and position R."""
        box = [(max(0, int(math.floor(self.R[k] - self.reach))), min(dims[k], int(math.ceil(self.R[k] + self.reach))))
               for k in range(3)]
        d = [torch.arange(a, max(a, b), dtype=torch.float64, device=self.S.device) + 0.5 - self.R[k]
             for k, (a, b) in enumerate(box)]
        d = (d[0][None, None, :], d[1][None, :, None], d[2][:, None, None])
        lo, hi = [], []
        for k in range(3):
            X = (Qm[0, k] * d[0] + Qm[1, k] * d[1]) + Qm[2, k] * d[2]
            a = torch.floor(((X - 0.5) - self.lo[k]) * self.n + 0.5).long()
            top = self.S.shape[2 - k] - 1
            lo.append(a.clamp(0, top))
            hi.append((a + self.n).clamp(0, top))
        count = 0
        for sz, z in ((1, hi[2]), (-1, lo[2])):
            for sy, y in ((1, hi[1]), (-1, lo[1])):
                for sx, x in ((1, hi[0]), (-1, lo[0])):
                    count = count + sz * sy * sx * self.S[z, y, x].long()
        return box, count.double() / self.n ** 3


class Ref:
    """The time step on a list of Q unshifted populations [nz, ny, nx]."""

    def __init__(self, case, bodies):
        self.c, self.Q, self.dims = case, case["Q"], (case["nx"], case["ny"], case["nz"])
        self.w, self.C = weights(self.Q), C27[:self.Q]
        self.bodies = bodies
        self.opp = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, self.Q)]
        wp = 1.0 / case["tau"]
        self.wp, self.wm = wp, 1.0 / (TRT_LAMBDA / (case["tau"] - 0.5) + 0.5) if case["fluid"] == "trt" else wp

    def feq(self, i, rho, u, uu):
        cu = sum((u[k] * self.C[i][k] for k in range(3) if self.C[i][k]), 0.0 * rho)
        return self.w[i] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu)

    def moments(self, f):
        rho = sum(f)
        u = [sum(f[i] * self.C[i][k] for i in range(self.Q) if self.C[i][k]) / rho for k in range(3)]
        return rho, u, u[0] * u[0] + u[1] * u[1] + u[2] * u[2]

    def fluid(self, f):
        """Omega^F as a function of the direction."""
        rho, u, uu = self.moments(f)
        if self.c["fluid"] == "cumulant":
            new = self.cumulant(f, rho, u)
            return [a - b for a, b in zip(new, f)]
        out = [None] * self.Q
        out[0] = -self.wp * (f[0] - self.feq(0, rho, u, uu))
        for i in range(1, self.Q, 2):
            ni, nj = f[i] - self.feq(i, rho, u, uu), f[i + 1] - self.feq(i + 1, rho, u, uu)
            even, odd = 0.5 * self.wp * (ni + nj), 0.5 * self.wm * (ni - nj)
            out[i], out[i + 1] = -even - odd, -even + odd
        return out

    def cumulant(self, f, rho, u):
        """Central moments of the 19 exponents with at most two non-zero; second order relaxed with
        1 / tau (its trace with 1), third- and fourth-order cumulants to equilibrium."""
        exps = [(a, b, c) for a in range(3) for b in range(3) for c in range(3) if a * b * c == 0]
        d = [[c[k] - u[k] for k in range(3)] for c in self.C]
        k = {}
        for e in ((2, 0, 0), (0, 2, 0), (0, 0, 2), (1, 1, 0), (1, 0, 1), (0, 1, 1)):
            k[e] = sum(f[i] * math.prod([d[i][a] ** e[a] for a in range(3) if e[a]]) for i in range(self.Q))
        t = 1.0 - 1.0 / self.c["tau"]
        tr = (k[2, 0, 0] + k[0, 2, 0] + k[0, 0, 2]) / 3
        p = {e: 0.0 * rho for e in exps}
        p[0, 0, 0] = rho
        for e in ((2, 0, 0), (0, 2, 0), (0, 0, 2)):
            p[e] = rho / 3 + t * (k[e] - tr)
        for e in ((1, 1, 0), (1, 0, 1), (0, 1, 1)):
            p[e] = t * k[e]
        for e, a, b in (((2, 2, 0), 0, 1), ((2, 0, 2), 0, 2), ((0, 2, 2), 1, 2)):
            one = tuple(1 if q in (a, b) else 0 for q in range(3))
            two = [tuple(2 if q == r else 0 for q in range(3)) for r in (a, b)]
            p[e] = (p[two[0]] * p[two[1]] + 2 * p[one] ** 2) / rho
        M = np.array([[math.prod(float(c[a]) ** e[a] for a in range(3)) for c in self.C] for e in exps])
        inv = np.linalg.inv(M)
        raw = []
        for e in exps:  # raw moments from the central ones (binomial shift)
            m = 0.0
            for a in range(e[0] + 1):
                for b in range(e[1] + 1):
                    for c in range(e[2] + 1):
                        g = math.comb(e[0], a) * math.comb(e[1], b) * math.comb(e[2], c)
                        m = m + g * p[a, b, c] * u[0] ** (e[0] - a) * u[1] ** (e[1] - b) * u[2] ** (e[2] - c)
            raw.append(m)
        return [sum(float(round(inv[i, j] * 8) / 8) * raw[j] for j in range(self.Q) if abs(inv[i, j]) > 1e-9)
                for i in range(self.Q)]

    def weighting(self, eps):
        if self.c["weighting"] == 0:
            return eps
        t = self.c["tau"] - 0.5
        return eps * t / ((1 - eps) + t)

    def psm(self, f, B, us):
        """Post-collision populations and sum_i Omega^S_i c_i of cells with weight B."""
        of = self.fluid(f)
        rho, u, uu = self.moments(f)
        ss = us[0] * us[0] + us[1] * us[1] + us[2] * us[2]
        new, mom = [None] * self.Q, [0.0, 0.0, 0.0]
        for i in range(self.Q):
            j = self.opp[i]
            if self.c["solid"] == 1:
                os_ = (f[j] - self.feq(j, rho, u, uu)) - (f[i] - self.feq(i, rho, us, ss))
            elif self.c["solid"] == 2:
                os_ = -(f[i] - self.feq(i, rho, us, ss)) / self.c["tau"]
            else:
                os_ = (f[j] - self.feq(j, rho, us, ss)) - (f[i] - self.feq(i, rho, us, ss))
            new[i] = f[i] + (1 - B) * of[i] + B * os_
            for k in range(3):
                if self.C[i][k]:
                    mom[k] = mom[k] + self.C[i][k] * os_
        return new, mom

    def ghosts(self, f, u_in):
        if self.c["bc_z"] != 1:
            return f
        uu = u_in[0] * u_in[0] + u_in[1] * u_in[1] + u_in[2] * u_in[2]
        one = uu * 0 + 1
        out = []
        for i, fi in enumerate(f):
            cz = self.C[i][2]
            if cz:
                g = self.feq(i, one, u_in, uu).expand(1, *fi.shape[1:])
                fi = torch.cat([g, fi[1:]]) if cz > 0 else torch.cat([fi[:-1], g])
            out.append(fi)
        return out

    def stream(self, f):
        return [torch.roll(fi, (c[2], c[1], c[0]), (0, 1, 2)) if any(c) else fi for fi, c in zip(f, self.C)]

    def solid_fraction(self, poses):
        nx, ny, nz = self.dims
        dev = device()
        eps = torch.zeros((nz, ny, nx), dtype=torch.float64, device=dev)
        best, owner = torch.zeros_like(eps), torch.full(eps.shape, -1, dtype=torch.int8, device=dev)
        for b, (body, Qm) in enumerate(zip(self.bodies, poses)):
            box, e = body.eps(self.dims, Qm)
            s = tuple(slice(*box[k]) for k in (2, 1, 0))
            eps[s] += e
            owner[s] = torch.where(e > best[s], torch.full_like(owner[s], b), owner[s])
            best[s] = torch.maximum(best[s], e)
        return eps.clamp(max=1.0), owner

    def step(self, f, poses, u_in):
        """One step in the cells' own list f (replaced); returns (f, [bodies, 6] force and torque)."""
        f = self.ghosts(f, u_in)
        eps, owner = self.solid_fraction(poses)
        idx = eps.reshape(-1).nonzero()[:, 0]
        nx, ny, _ = self.dims
        own = owner.reshape(-1)[idx]
        x = [(idx % nx).double() + 0.5, (idx // nx % ny).double() + 0.5, (idx // (nx * ny)).double() + 0.5]
        r, us = self.lever(x, own)
        B = self.weighting(eps.reshape(-1)[idx])
        new, mom = self.psm([fi.reshape(-1)[idx] for fi in f], B, us)
        of = self.fluid(f)
        for i in range(self.Q):
            f[i] = f[i] + of[i]
            of[i] = None
            f[i].reshape(-1)[idx] = new[i]
        return self.stream(f), self.loads(B, mom, r, own)

    def lever(self, x, own):
        r, us = [torch.zeros_like(x[0]) for _ in range(3)], [torch.zeros_like(x[0]) for _ in range(3)]
        for b, body in enumerate(self.bodies):
            m = own == b
            q = [torch.where(m, x[k] - body.R[k], 0.0) for k in range(3)]
            om = body.omega
            for k in range(3):
                r[k] = r[k] + q[k]
                i, j = (k + 1) % 3, (k + 2) % 3
                us[k] = us[k] + torch.where(m, om[i] * q[j] - om[j] * q[i] + body.v[k], 0.0)
        return r, us

    def loads(self, B, mom, r, own):
        G = [B * m for m in mom]
        T = [r[1] * G[2] - r[2] * G[1], r[2] * G[0] - r[0] * G[2], r[0] * G[1] - r[1] * G[0]]
        return torch.stack([torch.stack([-torch.where(own == b, v, 0.0).sum() for v in G + T])
                            for b in range(len(self.bodies))])


def exact_step(case, seed):
    cells = case["nx"] * case["ny"] * case["nz"]
    if cells > 2.0e8:
        return None
    bodies = [RefBody(*b) for b in bodies_of(case)]
    ref = Ref(case, bodies)
    g = initial(case, seed, DTYPE[case["storage"]])
    f = [g[i].double() + w for i, w in enumerate(ref.w)]
    del g
    u_in = [torch.tensor(v, dtype=torch.float64, device=device()) for v in (0.0, 0.0, case["u_in"])]
    ft = []
    if case["free"]:
        mass, inertia = ball(case)
        Qm, L = np.eye(3), inertia @ bodies[0].omega
    for n in range(case["steps"]):
        poses = [Qm] if case["free"] else [pose(b.spin, n) for b in bodies]
        f, t = ref.step(f, poses, u_in)
        ft.append(t.cpu().numpy())
        if case["free"]:
            b = bodies[0]
            b.v = b.v + ft[-1][0, :3] / mass
            b.R = b.R + b.v
            L = L + ft[-1][0, 3:]
            Qm = pose(Qm @ np.linalg.solve(inertia, Qm.T @ L), 1.0) @ Qm
            b.omega = Qm @ np.linalg.solve(inertia, Qm.T @ L)
    for i, w in enumerate(ref.w):
        f[i] = f[i] - w
    out = dict(f=stored(case, f), ft=[np.array([t[b] for t in ft]) for b in range(len(bodies))])
    if case["free"]:
        out["body"] = dict(R=bodies[0].R, v=bodies[0].v, Q=Qm, omega=bodies[0].omega, L=L)
    return out


def exact_gradient(case, seed, delta, w):
    """Loads of the forward run and the gradient of sum w . loads in the solid fraction, omega and
    u_in (the geometry sequence held fixed), by torch.autograd with one step kept at a time."""
    u0, _ = adjoint_inputs(case, seed)
    n, N, dev = case["n"], case["steps"], device()
    k = n / 256.0
    full = dict(nx=n, ny=n, nz=n, Q=19, bc_z=1, fluid=case["fluid"], tau=case["tau"], solid=1, weighting=1)
    ref = Ref(full, [RefBody(W.ELLIPSOID, (80.0 * k, 40.0 * k, 16.0 * k), 2, (n / 2,) * 3, (0.0, 0.0, 2e-4))])
    body = ref.bodies[0]
    delta = delta.double().reshape(-1).requires_grad_()
    omega = torch.tensor([0.0, 0.0, 2e-4], dtype=torch.float64, device=dev, requires_grad=True)
    u_in = torch.tensor([0.0, 0.0, u0], dtype=torch.float64, device=dev, requires_grad=True)
    i = torch.arange(n ** 3, device=dev)
    x = [(i % n).double() + 0.5, (i // n % n).double() + 0.5, (i // (n * n)).double() + 0.5]

    def one(step, delta, omega, u_in, *f):
        f = ref.ghosts([fi.reshape(n, n, n) for fi in f], u_in)
        eps, owner = ref.solid_fraction([pose(body.spin, step)])
        own = owner.reshape(-1)
        body.omega = omega
        r, us = ref.lever(x, own)
        B = ref.weighting(eps.reshape(-1) + delta)
        new, mom = ref.psm([fi.reshape(-1) for fi in f], B, us)
        f = ref.stream([fi.reshape(n, n, n) for fi in new])
        return (ref.loads(B, mom, r, own)[0], *f)

    uu = (u_in * u_in).sum()
    f = [ref.feq(q, uu * 0 + 1, u_in, uu).expand(n, n, n) for q in range(19)]
    ft = []
    for step in range(N):
        t, *f = torch.utils.checkpoint.checkpoint(one, step, delta, omega, u_in, *f, use_reentrant=False)
        ft.append(t)
    ft = torch.stack(ft)
    J = (ft * torch.tensor(w[:, 0], dtype=torch.float64, device=dev)).sum()
    ge, gw, gu = torch.autograd.grad(J, (delta, omega, u_in))
    return J.detach(), ft.detach(), ge.reshape(n, n, n), gw, gu


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        return exact_step(case, seed)
    if kind == "adjoint":
        _, w = adjoint_inputs(case, seed)
        n = case["n"]
        _, ft, ge, gw, gu = exact_gradient(case, seed, torch.zeros(n ** 3, device=device()), w)
        return dict(ft=ft, grad_eps=ge, grad_omega=gw[None], grad_uin=gu)
    if kind == "autograd":
        w = np.zeros((case["steps"], 1, 6))
        w[:, 0, 5] = 1.0 / case["steps"]
        J, _, ge, gw, gu = exact_gradient(case, seed, shell(case, seed), w)
        return dict(J=J, grad_eps=ge, grad_omega=gw, grad_uin=gu)
    if kind == "snapshot":
        w, Q = weights(case["Q"]), case["Q"]
        full = dict(case, tau=1.0, fluid="bgk")
        ref = Ref(full, [])
        g = initial(case, seed, DTYPE[case["storage"]])
        u_in = [torch.tensor(v, dtype=torch.float64, device=device()) for v in (0.0, 0.0, case["u_in"])]
        f = ref.ghosts([g[i].double() + w[i] for i in range(Q)], u_in)
        rho, u, _ = ref.moments(f)
        saved = saved_state(case, seed)
        for i in range(Q):
            saved[i] -= w[i]
        return dict(rho=rho, u=torch.stack(u, -1), state=torch.stack(f), f=stored(case, saved))
    return None  # whole numbers
