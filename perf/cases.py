"""Performance cases: what a user of the library has it do, call by call.

A pass of an explicit case loads a canonical state that lies on the GPU (a
restart, or the field another code hands over), takes a few LSRK(5,4) steps
and reads the node moments and the whole state back to device buffers, all
through the Python binding of the C ABI, with the library's own choice of
kernel and tile.  The batched case does the same for many small cases at once
and the implicit case takes one backward-Euler step.

The API returns FP64 arrays whatever the solver's precision.  The FP32 and
16-bit solvers carry FP32 values, so a pass hands their results back as FP32
(for FP32 state the conversion is exact), those of the FP64 solver as FP64.

``exact`` restates the method in plain FP64 torch and numpy, without the
library: warp & blend nodal operators, face matching, upwind flux, diffuse
walls, BGK collision and the five LSRK stages.
"""
import math
import random

import numpy as np
import torch

from paper_2012_13487_gb300 import fedbm as fb

DEV = "cuda"
PREC = {"fp64": fb.FP64, "fp32": fb.FP32, "bf16": fb.BF16_DEV, "fp16": fb.FP16_DEV}
RED = {"default": fb.RED_DEFAULT, "fp64": fb.RED_FP64, "comp": fb.RED_COMP_FP32}
STATE_BYTES = {"fp64": 8, "fp32": 4, "bf16": 2, "fp16": 2}
RES_BYTES = {"fp64": 8, "fp32": 4, "bf16": 4, "fp16": 4}
CFL = 0.5
DRAWN_DOF = (2e4, 5e7)       # state values of a drawn case
DRAWN_DOF_STEPS = 4e8        # state values times steps of a drawn case


def _case(name, kind, nx, ny, p, vel, n, precision, steps, **more):
    c = dict(kind=kind, nx=nx, ny=ny, p=p, vel=vel, n=n, sqrt2=0, eq=2, kn=1.0, speed=0.1, mesh=0,
             precision=precision, reduction="default", steps=steps, batch=0, implicit_dt=0.0, mass=False)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: the coarsest grid of a Couette order-of-accuracy study, in FP64 as such
        # a study needs, with the conservation check after the march; launches and latency count
        _case("couette_8x8_p2_gh16_fp64", "couette", 8, 8, 2, "gh", 4, "fp64", 20, mass=True),
        # a finer grid of the same study, third-order equilibrium
        _case("couette_24x24_p3_gh16_fp64", "couette", 24, 24, 3, "gh", 4, "fp64", 10, eq=3),
        # the lid-driven cavity at Kn = 1 on 256 velocities, the benchmark's default workload
        _case("cavity_64x64_p4_nc16_fp32", "cavity", 64, 64, 4, "nc", 16, "fp32", 8),
        # the same cavity with the 16-bit state
        _case("cavity_64x64_p4_nc16_bf16", "cavity", 64, 64, 4, "nc", 16, "bf16", 8, speed=0.05),
        # Couette at high order on the largest grid, 16 velocities
        _case("couette_256x256_p5_gh16_fp32", "couette", 256, 256, 5, "gh", 4, "fp32", 4),
        _case("couette_256x256_p5_gh16_bf16", "couette", 256, 256, 5, "gh", 4, "bf16", 4, speed=0.05),
        # the highly rarefied cavity: 1,024 velocities, 16-bit state, FP64 moment sums (the largest case)
        _case("cavity_128x128_p3_nc32_bf16", "cavity", 128, 128, 3, "nc", 32, "bf16", 2, kn=8.0, speed=0.05,
              reduction="fp64"),
        # D2Q1089 at degree 5: one element's velocities do not fit one thread block
        _case("cavity_32x32_p5_nc33_fp32", "cavity", 32, 32, 5, "nc", 33, "fp32", 3, kn=8.0, sqrt2=1),
        # an unstructured mesh, an odd element count and a velocity count (36) without a kernel of its own
        _case("unstructured_45x37_p3_gh36_fp32", "cavity", 45, 37, 3, "gh", 6, "fp32", 10, kn=0.5, eq=3, mesh=7),
        # a parameter sweep: 24 cases of mixed degree, size, velocity set and Kn in one batch
        _case("batch_24_fp32", "couette", 0, 0, 0, "gh", 4, "fp32", 3, batch=24, mesh=201213487),
        # one backward-Euler step towards the steady state, far beyond the explicit step (Newton-GMRES)
        _case("implicit_couette_16x16_p3_fp64", "couette", 16, 16, 3, "gh", 4, "fp64", 1, implicit_dt=0.5),
        # a coupled code that owns the field: load, one step, read everything back; ragged grid, FP16 state
        _case("coupled_61x67_p2_nc16_fp16", "cavity", 61, 67, 2, "nc", 16, "fp16", 1, kn=2.0, speed=0.05),
    ]


def draw(rng):
    """A solver of one of the same kinds: degree 1..5, 16 to 1,089 velocities, every state type, structured and
    unstructured meshes of odd sizes, 2e4 to 5e7 state values, 1 to 10 steps."""
    vel, n = rng.choice([("gh", 4)] * 7 + [("nc", 16)] * 7 + [("gh", 6)] * 2 + [("gh", 5)] + [("nc", 32)] * 2
                        + [("nc", 33)])
    q = n * n
    p = rng.randint(1, 5)
    precision = rng.choice(["fp64", "fp32", "fp32", "fp32", "bf16", "bf16", "fp16"])
    if q > 256 and precision == "fp64":
        precision = "fp32"
    if q > 1024 and precision == "fp16":
        precision = "bf16"
    np_ = (p + 1) * (p + 2) // 2
    top = 2e6 if precision == "fp64" else DRAWN_DOF[1]
    low = max(DRAWN_DOF[0], 2.0 * 16 * np_ * q)
    dof = math.exp(rng.uniform(math.log(low), math.log(max(top, 2 * low))))
    cells = dof / (2.0 * np_ * q)
    aspect = math.exp(rng.uniform(math.log(0.5), math.log(2.0)))
    nx = max(4, int(round(math.sqrt(cells * aspect))))
    ny = max(4, int(cells / nx))
    used = 2.0 * nx * ny * np_ * q
    steps = max(1, min(rng.randint(1, 10), int(DRAWN_DOF_STEPS / used)))
    sixteen = precision in ("bf16", "fp16")
    return _case(None, rng.choice(["couette", "cavity"]), nx, ny, p, vel, n, precision, steps,
                 sqrt2=1 if n == 33 else 0, eq=rng.choice([2, 2, 3]),
                 kn=math.exp(rng.uniform(math.log(0.5), math.log(8.0))),
                 speed=0.05 if sixteen else rng.uniform(0.05, 0.2),
                 mesh=rng.choice([0, 0, 0, rng.randint(1, 1000)]),
                 reduction=rng.choice(["default", "default", "fp64", "comp"]) if precision != "fp64" else "default")


# ---- the problem of a case -----------------------------------------------------
def _subcases(case):
    """The single cases of a case: itself, or the batch's seeded mix."""
    if not case["batch"]:
        return [case]
    rng = random.Random(case["mesh"])
    out = []
    for c in range(case["batch"]):
        vel, n = rng.choice([("gh", 4), ("nc", 16)])
        side = rng.randint(16, 40)
        out.append(_case(None, "couette" if c % 2 else "cavity", side, side, rng.randint(2, 5), vel, n,
                         case["precision"], case["steps"], kn=math.exp(rng.uniform(math.log(0.5), math.log(8.0))),
                         speed=rng.uniform(0.05, 0.2)))
    return out


def _walls(c):
    u = c["speed"]
    return ((-u, 0.0), (0.0, 0.0), (u, 0.0), (0.0, 0.0)) if c["kind"] == "couette" else \
        ((0.0, 0.0), (0.0, 0.0), (u, 0.0), (0.0, 0.0))


def _mesh(c):
    """Vertices [nv, 2], triangles [K, 3] and the vertex identities across a periodic pair of sides."""
    nx, ny = c["nx"], c["ny"]
    ix, iy = np.meshgrid(np.arange(nx + 1), np.arange(ny + 1))
    vert = np.stack([ix / nx, iy / ny], axis=-1).reshape(-1, 2)
    cx, cy = np.meshgrid(np.arange(nx), np.arange(ny))
    a = (cy * (nx + 1) + cx).ravel()
    b, t, d = a + 1, a + nx + 2, a + nx + 1
    if c["mesh"]:
        # interior vertices jittered, cells split along a random diagonal, triangles in random order
        r = np.random.RandomState(c["mesh"])
        inner = ((ix > 0) & (ix < nx) & (iy > 0) & (iy < ny)).reshape(-1, 1)
        vert = vert + np.where(inner, r.uniform(-0.2, 0.2, vert.shape) / np.array([nx, ny]), 0.0)
        up = (r.uniform(size=a.size) < 0.5)[:, None, None]
        tri = np.where(up, np.stack([np.stack([a, b, t], 1), np.stack([a, t, d], 1)], 1),
                       np.stack([np.stack([a, b, d], 1), np.stack([b, t, d], 1)], 1)).reshape(-1, 3)
        tri = tri[r.permutation(len(tri))]
    else:
        tri = np.stack([np.stack([a, b, t], 1), np.stack([a, t, d], 1)], 1).reshape(-1, 3)
    ident = np.arange(len(vert))
    if c["kind"] == "couette":
        ident = ((ident // (nx + 1)) * (nx + 1)) + (ident % (nx + 1)) % nx
    return vert, tri, ident


def _velocities(c):
    n = c["n"]
    if c["vel"] == "gh":
        x, w = np.polynomial.hermite_e.hermegauss(n)
        w = w / math.sqrt(2.0 * math.pi)
    else:
        # equispaced on [-4, 4] (in sqrt(RT) or sqrt(2RT)), trapezoid weights of the Maxwellian with an even
        # quartic factor that makes the moments of order 0, 2, 4 exact
        x = np.linspace(-4.0, 4.0, n) * (math.sqrt(2.0) if c["sqrt2"] else 1.0)
        w = np.full(n, x[1] - x[0])
        w[[0, -1]] *= 0.5
        w = w * np.exp(-0.5 * x * x) / math.sqrt(2.0 * math.pi)
        m = np.array([[np.sum(w * x ** (2 * (i + j))) for j in range(3)] for i in range(3)])
        k = np.linalg.solve(m, np.array([1.0, 1.0, 3.0]))
        w = w * (k[0] + k[1] * x ** 2 + k[2] * x ** 4)
    return np.repeat(x, n), np.tile(x, n), np.outer(w, w).ravel()


def _ref_nodes(p):
    """Warp & blend nodes (alpha = 0) of the reference triangle, row by row in s."""
    leg = np.polynomial.legendre
    inner = leg.legroots(leg.legder([0] * p + [1])) if p > 1 else np.zeros(0)
    gll, eq = np.concatenate([[-1.0], np.sort(np.real(inner)), [1.0]]), np.linspace(-1.0, 1.0, p + 1)

    def warp(x):
        y = np.zeros_like(x)
        for j in range(p + 1):
            l = np.ones_like(x)
            for m in range(p + 1):
                if m != j:
                    l = l * (x - eq[m]) / (eq[j] - eq[m])
            y += (gll[j] - eq[j]) * l
        inside = np.abs(x) < 1 - 1e-10
        return np.where(inside, y / np.where(inside, 1 - x * x, 1.0), 0.0)

    l1 = np.array([i / p for i in range(p + 1) for _ in range(p + 1 - i)])
    l3 = np.array([j / p for i in range(p + 1) for j in range(p + 1 - i)])
    l2 = 1 - l1 - l3
    # displacements along the three edges, written in barycentric coordinates
    w1, w2, w3 = 4 * l2 * l3 * warp(l3 - l2), 4 * l1 * l3 * warp(l1 - l3), 4 * l1 * l2 * warp(l2 - l1)
    x = -l2 + l3 + w1 - 0.5 * w2 - 0.5 * w3
    y = (2 * l1 - l2 - l3) / math.sqrt(3.0) + math.sqrt(0.75) * (w2 - w3)
    b1, b3 = (math.sqrt(3.0) * y + 1) / 3, (3 * x - math.sqrt(3.0) * y + 2) / 6
    return 2 * b3 - 1, 2 * b1 - 1


def _basis(p, r, s):
    """Legendre products of total degree <= p and their r, s derivatives at the points."""
    leg = np.polynomial.legendre
    one = [np.eye(p + 1)[i] for i in range(p + 1)]
    der = [leg.legder(e) if p else np.zeros(1) for e in one]
    ij = [(i, j) for i in range(p + 1) for j in range(p + 1 - i)]
    v = [leg.legval(r, one[i]) * leg.legval(s, one[j]) for i, j in ij]
    vr = [leg.legval(r, der[i]) * leg.legval(s, one[j]) for i, j in ij]
    vs = [leg.legval(r, one[i]) * leg.legval(s, der[j]) for i, j in ij]
    return np.array(v).T, np.array(vr).T, np.array(vs).T


def _operators(p):
    r, s = _ref_nodes(p)
    v, vr, vs = _basis(p, r, s)
    inv = np.linalg.inv(v)
    g, gw = np.polynomial.legendre.leggauss(p + 3)
    a, b = (m.ravel() for m in np.meshgrid(g, g))
    wq = np.outer(gw, gw).ravel() * 0.5 * (1 - b)
    lq = _basis(p, 0.5 * (1 + a) * (1 - b) - 1, b)[0] @ inv
    mass = lq.T @ (wq[:, None] * lq)
    start = [i * (p + 1) - i * (i - 1) // 2 for i in range(p + 1)]
    # face nodes from vertex f to vertex f + 1
    face = np.array([[start[0] + j for j in range(p + 1)], [start[i] + p - i for i in range(p + 1)],
                     [start[i] for i in range(p, -1, -1)]])
    lift = np.zeros((len(r), 3, p + 1))
    for f, (rr, ss) in enumerate(((g, -np.ones_like(g)), (-g, g), (-np.ones_like(g), -g))):
        lf = _basis(p, rr, ss)[0] @ inv
        lift[:, f] = np.linalg.solve(mass, lf.T @ (gw[:, None] * lf[:, face[f]]))
    return dict(r=r, s=s, Dr=vr @ inv, Ds=vs @ inv, lift=lift.reshape(len(r), -1), face=face, colsum=mass.sum(0))


def _coordinates(vert, tri, r, s):
    x = vert[tri]
    return (-0.5 * (r + s))[None, :, None] * x[:, None, 0] + (0.5 * (1 + r))[None, :, None] * x[:, None, 1] \
        + (0.5 * (1 + s))[None, :, None] * x[:, None, 2]


def _equilibrium(rho, ux, uy, ex, ey, w, eq):
    eu = ux[..., None] * ex + uy[..., None] * ey
    uu = (ux * ux + uy * uy)[..., None]
    poly = 1 + eu + 0.5 * (eu * eu - uu)
    if eq == 3:
        poly = poly + eu * (eu * eu / 6 - 0.5 * uu)
    return w * rho[..., None] * poly


def _initial(c, seed):
    """A flow in progress: smooth density and velocity fields of random phase, and 1e-3 of noise off equilibrium."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    phase = random.Random(seed).random
    vert, tri, _ = _mesh(c)
    xy = torch.from_numpy(_coordinates(vert, tri, *_ref_nodes(c["p"]))).to(DEV)
    ex, ey, w = (torch.from_numpy(v).to(DEV) for v in _velocities(c))
    x, y = 2 * math.pi * xy[..., 0], math.pi * xy[..., 1]
    rho = 1 + 0.005 * torch.sin(x + 6 * phase()) * torch.cos(y)
    ux = 0.02 * torch.cos(x + 6 * phase()) * torch.sin(y)
    uy = 0.02 * torch.sin(x + 6 * phase()) * torch.sin(y)
    f = _equilibrium(rho, ux, uy, ex, ey, w, c["eq"])
    f.mul_(torch.empty_like(f).uniform_(1 - 1e-3, 1 + 1e-3, generator=g))
    return f if c["precision"] == "fp64" else f.float()


def _descriptors(c):
    bc = (fb.BC_WALL_DIFFUSE, fb.BC_PERIODIC, fb.BC_WALL_DIFFUSE, fb.BC_PERIODIC) if c["kind"] == "couette" \
        else (fb.BC_WALL_DIFFUSE,) * 4
    if c["mesh"]:
        vert, tri, _ = _mesh(c)
        m = fb.unstructured_mesh_desc(vert, tri, c["p"], bc=bc, wall_u=_walls(c))
    else:
        m = fb.mesh_desc(c["nx"], c["ny"], c["p"], bc=bc, wall_u=_walls(c))
    v = fb.velset_desc(fb.VELSET_GH if c["vel"] == "gh" else fb.VELSET_NC, c["n"], c["eq"], nc_sqrt2=c["sqrt2"])
    return m, v, fb.params(kn=c["kn"], precision=PREC[c["precision"]], reduction=RED[c["reduction"]], cfl=CFL)


def _sizes(c):
    np_ = (c["p"] + 1) * (c["p"] + 2) // 2
    return 2 * c["nx"] * c["ny"], np_, c["n"] ** 2


# ---- a pass --------------------------------------------------------------------
class State:
    """The solver (or batch) a user's program keeps, its input fields and its output buffers."""

    def __init__(self, case, seed):
        self.case, self.subs = case, _subcases(case)
        self.wide = case["precision"] == "fp64"
        self.inputs = [_initial(c, seed + 1000003 * i) for i, c in enumerate(self.subs)]
        stream = torch.cuda.current_stream().cuda_stream
        if case["batch"]:
            self.solver = fb.Batch([fb.case_desc(*_descriptors(c)) for c in self.subs], stream)
        else:
            self.solver = fb.Solver(*_descriptors(self.subs[0]), stream)
        sizes = [_sizes(c) for c in self.subs]
        self.out = torch.empty(sum(k * n * q for k, n, q in sizes), dtype=torch.float64, device=DEV)
        self.mom = torch.empty(3, sum(k * n for k, n, _ in sizes), dtype=torch.float64, device=DEV)
        self.out_at = self.out.split([k * n * q for k, n, q in sizes])
        self.mom_at = [m.split([k * n for k, n, _ in sizes]) for m in self.mom]
        self.implicit = fb.implicit_params(fb.IMPLICIT_BE, case["implicit_dt"], newton_rtol=1e-11,
                                           preconditioner=1) if case["implicit_dt"] else None


def prepare(case, seed):
    return State(case, seed)


def run(s):
    h = s.solver.h
    if s.case["batch"]:
        for c, f in enumerate(s.inputs):
            fb.fedbm_batch_set_state_f32(h, c, f, True)
        fb.fedbm_batch_rk_step(h, s.case["steps"])
        for c in range(len(s.inputs)):
            fb.fedbm_batch_get_moments(h, c, *(m[c] for m in s.mom_at), True)
            fb.fedbm_batch_get_state(h, c, s.out_at[c], True)
    else:
        (fb.fedbm_set_state if s.wide else fb.fedbm_set_state_f32)(h, s.inputs[0], True)
        if s.implicit is not None:
            fb.fedbm_implicit_step(h, s.implicit, s.case["steps"])
        else:
            fb.fedbm_rk_step(h, s.case["steps"])
        fb.fedbm_get_moments(h, *s.mom, True)
        fb.fedbm_get_state(h, s.out, True)
    got = {"state": s.out, "moments": s.mom}
    if not s.wide:
        got = {k: v.float() for k, v in got.items()}
    if s.case["mass"]:
        got["mass"] = s.solver.mass()
    return got


def work(case):
    """Bytes: the field in and out once in the caller's type, and for every LSRK stage, which needs its neighbours'
    previous stage, the state read and written and the residual written and (but for the first) read.  Operations:
    the two derivative contractions, the lift, and about 30 for flux, equilibrium, collision and update."""
    total = {"bytes": 0.0, "flops": 0.0}
    for c in _subcases(case):
        k, np_, q = _sizes(c)
        dof, sb, rb = float(k * np_ * q), STATE_BYTES[c["precision"]], RES_BYTES[c["precision"]]
        stages = 1 if case["implicit_dt"] else 5 * c["steps"]
        given = 8 if c["precision"] == "fp64" else 4
        total["bytes"] += dof * (given + 2 * sb + 8) + 24.0 * k * np_
        total["bytes"] += dof * (stages * (2 * sb + rb) + (0 if case["implicit_dt"] else 4 * c["steps"] * rb))
        total["flops"] += dof * stages * (2.0 * (2 * np_ + 3 * (c["p"] + 1)) + 30.0)
    return total


# ---- the same in FP64, without the library ----------------------------------------
LSRK_A = (0.0, -567301805773 / 1357537059087, -2404267990393 / 2016746695238, -3550918686646 / 2091501179385,
          -1275806237668 / 842570457699)
LSRK_B = (1432997174477 / 9575080441755, 5161836677717 / 13612068292357, 1720146321549 / 2090206949498,
          3134564353537 / 4481467310338, 2277821191437 / 14882151754819)


class _Exact:
    def __init__(self, c):
        self.c = c
        vert, tri, ident = _mesh(c)
        o = _operators(c["p"])
        x = vert[tri]
        e = np.roll(x, -1, axis=1) - x                                  # edge f: vertex f to f + 1
        length = np.hypot(e[..., 0], e[..., 1])
        xr, xs = 0.5 * (x[:, 1] - x[:, 0]), 0.5 * (x[:, 2] - x[:, 0])
        jac = xr[:, 0] * xs[:, 1] - xs[:, 0] * xr[:, 1]
        rx, ry, sx, sy = xs[:, 1] / jac, -xs[:, 0] / jac, -xr[:, 1] / jac, xr[:, 0] / jac
        normal = np.stack([e[..., 1], -e[..., 0]], -1) / length[..., None]
        a, b = ident[tri], ident[np.roll(tri, -1, axis=1)]
        nv = len(vert)
        key, want = (a * nv + b).ravel(), (b * nv + a).ravel()
        order = np.argsort(key)
        at = np.minimum(np.searchsorted(key[order], want), len(key) - 1)
        found = key[order][at] == want
        mate = order[at]
        k, np_ = len(tri), len(o["r"])
        other = (mate // 3)[:, None] * np_ + o["face"][mate % 3][:, ::-1]
        own = np.repeat(np.arange(k), 3)[:, None] * np_ + np.tile(o["face"], (k, 1))
        mid = 0.5 * (x + np.roll(x, -1, axis=1)).reshape(-1, 2)
        side = np.select([mid[:, 1] < 1e-9, mid[:, 0] > 1 - 1e-9, mid[:, 1] > 1 - 1e-9, mid[:, 0] < 1e-9],
                         [0, 1, 2, 3], -1)
        assert (side[~found] >= 0).all()
        ex, ey, w = _velocities(c)

        def dev(v):
            return torch.from_numpy(np.ascontiguousarray(v)).to(DEV)

        self.K, self.Np, self.Nfp, self.Q = k, np_, c["p"] + 1, len(w)
        self.Dr, self.Ds, self.lift = dev(o["Dr"]), dev(o["Ds"]), dev(o["lift"])
        self.face = dev(o["face"].ravel())
        self.metric = [dev(v)[:, None] for v in (rx, ry, sx, sy)]
        self.normal, self.fscale = dev(normal), dev(0.5 * length / jac[:, None])
        self.other = dev(np.where(found[:, None], other, own).reshape(k, 3 * self.Nfp))
        self.wall = dev(np.where(found, -1, side).reshape(k, 3))
        self.ex, self.ey, self.w = dev(ex), dev(ey), dev(w)
        self.feq_wall, self.den = [], []
        for u, n in zip(_walls(c), ((0, -1), (1, 0), (0, 1), (-1, 0))):
            fw = _equilibrium(torch.ones((), dtype=torch.float64, device=DEV),
                              *(torch.tensor(v, dtype=torch.float64, device=DEV) for v in u),
                              self.ex, self.ey, self.w, c["eq"])
            self.feq_wall.append(fw)
            self.den.append(((-(self.ex * n[0] + self.ey * n[1])).clamp(min=0) * fw).sum())
        self.tau = c["kn"] / math.sqrt(3.0)
        radius = (2 * jac) * 2 / length.sum(1)                         # 2 area / perimeter, area = 2 jac
        self.dt = CFL * radius.min() / (np.hypot(ex, ey).max() * (c["p"] + 1) ** 2)
        self.jac, self.colsum = dev(jac), dev(o["colsum"])

    def rhs(self, f, lo, hi):
        fe = f[lo:hi]
        rx, ry, sx, sy = (m[lo:hi] for m in self.metric)
        ar, as_ = rx * self.ex + ry * self.ey, sx * self.ex + sy * self.ey
        out = -(ar[:, None] * (self.Dr @ fe)) - as_[:, None] * (self.Ds @ fe)
        minus = fe[:, self.face].view(hi - lo, 3, self.Nfp, self.Q)
        plus = f.view(-1, self.Q)[self.other[lo:hi].reshape(-1)].view(minus.shape)
        en = self.normal[lo:hi, :, :1] * self.ex + self.normal[lo:hi, :, 1:] * self.ey
        for side in range(4):
            at = (self.wall[lo:hi] == side).nonzero(as_tuple=True)
            if at[0].numel():
                e = en[at][:, None]
                rho = (e.clamp(min=0) * minus[at]).sum(-1, keepdim=True) / self.den[side]
                plus[at] = torch.where(e < 0, rho * self.feq_wall[side], minus[at])
        c = 0.5 * (en - en.abs()) * self.fscale[lo:hi, :, None]
        flux = (c[:, :, None] * (minus - plus)).view(hi - lo, 3 * self.Nfp, self.Q)
        out += self.lift @ flux
        rho, jx, jy = self.moments(fe)
        out -= (fe - _equilibrium(rho, jx / rho, jy / rho, self.ex, self.ey, self.w, self.c["eq"])) / self.tau
        return out

    def moments(self, f):
        return f.sum(-1), f @ self.ex, f @ self.ey

    def march(self, f, steps):
        res = torch.zeros_like(f)
        chunk = max(1, int(3e7 // (self.Np * self.Q)))
        for _ in range(steps):
            for a, b in zip(LSRK_A, LSRK_B):
                for lo in range(0, self.K, chunk):
                    hi = min(self.K, lo + chunk)
                    res[lo:hi].mul_(a).add_(self.rhs(f, lo, hi), alpha=float(self.dt))
                f = f + b * res
        return f


def exact(case, seed):
    if case["implicit_dt"]:
        return None
    states, moments, mass = [], [], 0.0
    for i, c in enumerate(_subcases(case)):
        m = _Exact(c)
        f = m.march(_initial(c, seed + 1000003 * i).double(), c["steps"])
        rho, jx, jy = m.moments(f)
        states.append(f.view(-1))
        moments.append(torch.stack([rho, jx / rho, jy / rho]).view(3, -1))
        mass = float((m.jac[:, None] * m.colsum * rho).sum())
        del m, f
    got = {"state": torch.cat(states), "moments": torch.cat(moments, 1)}
    if case["mass"]:
        got["mass"] = mass
    return got
