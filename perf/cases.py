"""The workloads this library is timed on.

Every case is a use of the public entry points over whole arrays: an initial
state set on a solver that the program keeps, a run of time steps, and the
state and the moments read back (on the device).  Initial states are not in
equilibrium: a shock is a mixture of its two end Maxwellians, a cavity a
smooth field of anisotropic Maxwellians, both with seeded noise.

``exact`` is the same computation in plain FP64 torch, written from the
method's equations (upwind free streaming, moments, effective Maxwellian
parameters, relaxation), without the library's code.
"""
from __future__ import annotations

import math

import torch
from torch.utils.checkpoint import checkpoint

from paper_0903_4044_gb300 import adjoint as A
from paper_0903_4044_gb300 import bgk as B
from paper_0903_4044_gb300 import solver as S
from paper_0903_4044_gb300 import workloads as W

DEV = "cuda"
F64 = torch.float64
GAMMA = 5.0 / 3.0
PRECISIONS = {"f64": B.BGK_F64, "f32": B.BGK_F32, "bf16": B.BGK_BF16_DEV}
STATE_BYTES = {"f64": 16, "f32": 8, "bf16": 4}  # one (g, h) pair in storage


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def _shock(**over):
    return dict(dict(kind="shock", precision="f64", nx=200, nvx=64, vbox=8.0, length=40.0, mach=2.0, omega=0.5,
                     cfl=0.5, conservative=1, relax_exact=1, steps=200), **over)


def _cavity(**over):
    return dict(dict(kind="cavity", precision="f64", nx=64, ny=64, nvx=32, nvy=32, vbox=5.0, kn=0.1, lid=0.09,
                     wall="diffuse", omega=0.5, cfl=0.5, conservative=1, relax_exact=1, steps=100), **over)


def _shock3v(**over):
    return dict(dict(kind="shock3v", precision="f64", nx=512, nvx=16, nvy=16, nvz=16, vx0=-5.0, vx1=7.0, vt=6.0,
                     length=70.0, mach=1.5, omega=0.74, dt=0.05, conservative=1, relax_exact=1, steps=20), **over)


def listed():
    return [
        # the Mach 2 shock: 12 800 points, a step is a few microseconds and launches and latency count
        dict(name="shock_200x64_f64", **_shock()),
        # a faster shock in FP32 as in the batched workload, cells and velocities not multiples of anything
        dict(name="shock_777x88_f32", **_shock(precision="f32", nx=777, nvx=88, vbox=13.0, mach=3.0)),
        # one step on the caller's own buffers: the smallest call, tables and checks included
        dict(name="single_step_32x32_v16x16_f64", **_cavity(kind="single", nx=32, ny=32, nvx=16, nvy=16, steps=1)),
        # the lid-driven cavity at its ordinary size
        dict(name="cavity_64x64_v32x32_f64", **_cavity()),
        # the benchmark's grid
        dict(name="cavity_256x256_v48x48_f64",
             **_cavity(nx=256, ny=256, nvx=48, nvy=48, kn=0.05, lid=0.045, steps=20)),
        # a channel with mirror walls, an odd grid and a velocity grid of 20 x 28: nothing divides anything
        dict(name="channel_157x83_v20x28_f64",
             **_cavity(nx=157, ny=83, nvx=20, nvy=28, vbox=4.5, wall="specular", omega=0.74, cfl=0.9, steps=50)),
        # the benchmark's grid with the state in FP32
        dict(name="cavity_256x256_v48x48_f32",
             **_cavity(precision="f32", nx=256, ny=256, nvx=48, nvy=48, kn=0.05, lid=0.045, steps=50)),
        # the cavity of the drag table, the state as BF16 deviations
        dict(name="cavity_160x160_v40x40_bf16",
             **_cavity(precision="bf16", nx=160, ny=160, nvx=40, nvy=40, lid=0.05, steps=50)),
        # many small FP32 problems at once: a parameter study
        dict(name="batch_24cavities_8shocks_f32", kind="batch", precision="f32", instances=0, cavities=24, shocks=8,
             steps=20),
        # gradient of the lid shear: forward, recomputation and reverse pass
        dict(name="gradient_128x128_v32x32_f64", **_cavity(kind="gradient", nx=128, ny=128, steps=100)),
        # the shock on the full velocity grid at the paper's two grids
        dict(name="shock3v_512_v16x16x16_f64", **_shock3v()),
        dict(name="shock3v_2048_v30x30x30_f64",
             **_shock3v(nx=2048, nvx=30, nvy=30, nvz=30, vx0=-10.0, vx1=12.0, vt=11.0, mach=3.0, steps=10)),
    ]


# updates (points times steps) of the largest listed case
MOST = 256 * 256 * 48 * 48 * 20


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _steps(rng, points, most, cap=200):
    return max(1, min(cap, int(_log(rng, 1.0, max(1.5, most / points)))))


def draw(rng):
    kind = rng.choice(["shock", "shock", "cavity", "cavity", "cavity", "reduced", "reduced", "single", "batch",
                       "gradient", "shock3v", "shock3v"])
    if kind == "shock":
        f32 = rng.random() < 0.4
        mach = rng.uniform(1.2, 5.0)
        vbox = 4.0 + 3.0 * mach
        nvx = max(16, int(2.0 * vbox / rng.uniform(0.25, 0.55)))
        c = _shock(precision="f32" if f32 else "f64", nx=int(_log(rng, 40, 2000)), mach=mach, vbox=vbox,
                   nvx=min(nvx, 128) if f32 else nvx, cfl=rng.choice([0.5, 0.95, rng.uniform(0.2, 3.0)]),
                   omega=rng.choice([0.5, 0.74]), conservative=rng.choice([1, 1, 0]),
                   relax_exact=rng.choice([1, 1, 0]))
        c["steps"] = _steps(rng, c["nx"] * c["nvx"], MOST / 60)
        return c
    if kind in ("cavity", "single", "gradient"):
        top = {"cavity": 256, "single": 128, "gradient": 96}[kind]
        nx, ny = (int(_log(rng, 12, top)) for _ in range(2))
        nvx, nvy = (rng.choice([16, 20, 24, 28, 32, 40, 48, rng.randint(16, 48)]) for _ in range(2))
        c = _cavity(kind=kind, nx=nx, ny=ny, nvx=nvx, nvy=nvy, vbox=rng.choice([4.0, 4.5, 5.0]), kn=_log(rng, 0.01, 1.0),
                    lid=_log(rng, 0.02, 0.27), omega=rng.choice([0.5, 0.74]), cfl=rng.choice([0.5, 0.9, 1.0]))
        if kind != "gradient":
            c.update(wall=rng.choice(["diffuse", "diffuse", "specular"]), conservative=rng.choice([1, 1, 1, 0]),
                     relax_exact=rng.choice([1, 1, 1, 0]))
        else:
            # the objective's derivative takes the map to effective parameters as the identity, which needs a
            # velocity grid that resolves the Maxwellian
            c.update(ny=nx, nvx=max(24, nvx), nvy=max(24, nvx), vbox=5.0)
        points = c["nx"] * c["ny"] * c["nvx"] * c["nvy"]
        c["steps"] = 1 if kind == "single" else _steps(rng, points, MOST / (8 if kind == "gradient" else 2))
        return c
    if kind == "reduced":
        nx, ny = (int(_log(rng, 16, 256)) for _ in range(2))
        c = _cavity(precision=rng.choice(["f32", "bf16"]), nx=nx, ny=ny, nvx=8 * rng.randint(2, 6),
                    nvy=rng.choice([16, 24, 32, 40, 48, rng.randint(16, 48)]), kn=_log(rng, 0.01, 1.0),
                    lid=_log(rng, 0.02, 0.27), wall=rng.choice(["diffuse", "diffuse", "specular"]),
                    cfl=rng.choice([0.5, 0.9]), conservative=rng.choice([1, 1, 0]))
        c["steps"] = _steps(rng, nx * ny * c["nvx"] * c["nvy"], MOST)
        return c
    if kind == "batch":
        return dict(kind="batch", precision="f32", instances=rng.randint(1, 1 << 30), cavities=rng.randint(2, 24),
                    shocks=rng.randint(1, 12), steps=rng.randint(1, 20))
    nv = [rng.randint(10, 32) for _ in range(3)]
    mach = rng.uniform(1.2, 3.0)
    vt = 4.0 + 2.2 * mach
    c = _shock3v(nx=int(_log(rng, 48, 1500)), nvx=nv[0], nvy=nv[1], nvz=nv[2], vx0=-vt, vx1=vt + 1.0, vt=vt, mach=mach,
                 conservative=rng.choice([1, 1, 0]), relax_exact=rng.choice([1, 1, 0]), dt=rng.choice([0.02, 0.05]))
    c["steps"] = _steps(rng, c["nx"] * nv[0] * nv[1] * nv[2], MOST / 8, 40)
    return c


# --------------------------------------------------------------------------
# grids and configurations
# --------------------------------------------------------------------------
def _centres(lo, hi, n):
    return lo + (torch.arange(n, device=DEV, dtype=F64) + 0.5) * ((hi - lo) / n)


def _from_workload(w):
    """A case dict for one raw entry of the batched workload."""
    if w["kind"] == "shock":
        return _shock(precision=w["precision"], nx=w["nx"], nvx=w["nvx"], vbox=w["vx"][1], length=w["length"],
                      mach=w["mach"], omega=w["omega"], cfl=w["cfl"])
    return _cavity(precision=w["precision"], nx=w["n"], ny=w["n"], nvx=w["nv"], nvy=w["nv"], vbox=w["vbox"][1],
                   kn=w["kn"], lid=w["lid_mach"] * math.sqrt(GAMMA / 2.0), omega=w["omega"], cfl=w["cfl"])


def _instances(case):
    return W.batch_instances(case["instances"], case["cavities"], case["shocks"])


def _ends(mach):
    """Rankine-Hugoniot states (n, u, theta) upstream and downstream, speeds in sqrt(2 R T0)."""
    m2 = mach * mach
    dens = 4.0 * m2 / (m2 + 3.0)
    u = mach * math.sqrt(0.5 * GAMMA)
    return (1.0, u, 1.0), (dens, u / dens, (5.0 * m2 - 1.0) * (m2 + 3.0) / (16.0 * m2))


def _lengths(c):
    """Domain sides of a cavity: 1 / Kn along y, square cells."""
    side = 1.0 / c["kn"]
    return side * c["nx"] / c["ny"], side


def _config(c):
    common = dict(omega=c["omega"], cfl=c["cfl"], conservative=c["conservative"], relax_exact=c["relax_exact"],
                  precision=PRECISIONS[c["precision"]])
    if c["kind"] == "shock":
        up, down = _ends(c["mach"])
        bc = [(B.BGK_BC_INFLOW, s[0], s[1], 0.0, s[2]) for s in (up, down)]
        return B.make_config(dim=1, nx=c["nx"], ny=1, x0=-0.5 * c["length"], lx=c["length"], nvx=c["nvx"], nvy=1,
                             vx=(-c["vbox"], c["vbox"]), bc=bc, **common)
    kind = B.BGK_BC_DIFFUSE if c["wall"] == "diffuse" else B.BGK_BC_SPECULAR
    rest, lid = (kind, 1.0, 0.0, 0.0, 1.0), (kind, 1.0, c["lid"], 0.0, 1.0)
    lx, ly = _lengths(c)
    return B.make_config(dim=2, nx=c["nx"], ny=c["ny"], lx=lx, ly=ly, nvx=c["nvx"], nvy=c["nvy"],
                         vx=(-c["vbox"], c["vbox"]), vy=(-c["vbox"], c["vbox"]), bc=[rest, rest, rest, lid], **common)


def _config3v(c):
    up, down = ((s[0], s[1], 0.0, 0.0, s[2]) for s in _ends(c["mach"]))
    return B.make_config3v(nx=c["nx"], x0=-0.5 * c["length"], lx=c["length"], nv=(c["nvx"], c["nvy"], c["nvz"]),
                           vmin=(c["vx0"], -c["vt"], -c["vt"]), vmax=(c["vx1"], c["vt"], c["vt"]), omega=c["omega"],
                           dt=c["dt"], conservative=c["conservative"], relax_exact=c["relax_exact"],
                           inflow=(up, down))


# --------------------------------------------------------------------------
# initial states
# --------------------------------------------------------------------------
def _noise(g, t, amp=1e-3):
    """t times (1 + amp xi), xi uniform in [-1, 1), in place."""
    return t.mul_(torch.rand(t.shape, generator=g, device=DEV, dtype=F64).mul_(2.0 * amp).add_(1.0 - amp))


def _profile(c, g):
    """Weight of the downstream state along a shock: a smooth step, its place and width from the seed."""
    r = torch.rand(2, generator=g, device=DEV, dtype=F64)
    x = _centres(-0.5, 0.5, c["nx"]) * c["length"]
    return 0.5 * (1.0 + torch.tanh((x - (4.0 * r[0] - 2.0)) / (1.0 + 3.0 * r[1])))


def _waves(c, g, amp):
    """A smooth random field of the size of amp over the cells (ny, nx, 1, 1)."""
    x, y = _centres(0.0, 1.0, c["nx"]), _centres(0.0, 1.0, c["ny"])[:, None]
    f = torch.zeros(c["ny"], c["nx"], device=DEV, dtype=F64)
    for k in range(1, 4):
        r = torch.rand(4, generator=g, device=DEV, dtype=F64)
        f += (r[0] - 0.5) * torch.sin(math.pi * k * x + 6.28 * r[1]) * torch.cos(math.pi * k * y + 6.28 * r[2]) / k
    return (amp * f)[:, :, None, None]


def _initial(c, seed):
    """FP64 initial state in the state layout (cells, velocities, 2), or (cells, velocities) on the full grid."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    if c["kind"] == "shock":
        s = _profile(c, g)[:, None]
        cx = _centres(-c["vbox"], c["vbox"], c["nvx"])
        f = torch.empty(c["nx"], c["nvx"], 2, device=DEV, dtype=F64)
        m = [n / math.sqrt(math.pi * th) * torch.exp(-(cx - u) ** 2 / th) for n, u, th in _ends(c["mach"])]
        f[..., 0] = (1.0 - s) * m[0] + s * m[1]
        f[..., 1] = (1.0 - s) * m[0] + s * m[1] * _ends(c["mach"])[1][2]
        return _noise(g, f)
    if c["kind"] == "shock3v":
        s = _profile(c, g)[:, None, None, None]
        cx = _centres(c["vx0"], c["vx1"], c["nvx"])
        cy, cz = _centres(-c["vt"], c["vt"], c["nvy"])[:, None], _centres(-c["vt"], c["vt"], c["nvz"])[:, None, None]
        m = [n * (math.pi * th) ** -1.5 * torch.exp(-((cx - u) ** 2 + cy ** 2 + cz ** 2) / th)
             for n, u, th in _ends(c["mach"])]
        return _noise(g, (1.0 - s) * m[0] + s * m[1]).reshape(c["nx"], -1)
    cx, cy = _centres(-c["vbox"], c["vbox"], c["nvx"]), _centres(-c["vbox"], c["vbox"], c["nvy"])[:, None]
    n = 1.0 + _waves(c, g, 0.05)
    ux, uy = _waves(c, g, c["lid"]), _waves(c, g, c["lid"])
    tx, ty, tz = (1.0 + _waves(c, g, 0.05) for _ in range(3))
    f = torch.empty(c["ny"], c["nx"], c["nvy"], c["nvx"], 2, device=DEV, dtype=F64)
    f[..., 0] = (n / (math.pi * torch.sqrt(tx * ty)) * torch.exp(-(cy - uy) ** 2 / ty)) * torch.exp(-(cx - ux) ** 2 / tx)
    f[..., 1] = 0.5 * tz * f[..., 0]
    return _noise(g, f).reshape(c["ny"] * c["nx"], -1, 2)


# --------------------------------------------------------------------------
# what is run
# --------------------------------------------------------------------------
def prepare(case, seed):
    st = {"case": case, "kind": case["kind"]}
    if case["kind"] == "batch":
        ws = _instances(case)
        st["batch"] = S.Batch(ws, perturb=False)
        st["f0"] = [_initial(_from_workload(w), seed + 1000 * i) for i, w in enumerate(ws)]
        st["out"] = [torch.empty_like(f) for f in st["f0"]]
        st["mom"] = [torch.empty(f.shape[0], 4, device=DEV, dtype=F64) for f in st["f0"]]
        return st
    f0 = _initial(case, seed)
    st["f0"] = f0
    if case["kind"] == "gradient":
        st["f0"] = f0.requires_grad_()
        st["kn"] = torch.tensor(case["kn"], dtype=F64, requires_grad=True)
        st["lid"] = torch.tensor(case["lid"], dtype=F64, requires_grad=True)
        w = dict(n=case["nx"], nv=case["nvx"], vbox=(-case["vbox"], case["vbox"]), omega=case["omega"],
                 cfl=case["cfl"], conservative=case["conservative"])
        st["spec"] = A.cavity_spec(w, case["steps"], 0)
        return st
    st["out"] = torch.empty_like(f0)
    st["mom"] = torch.empty(f0.shape[0], 5 if case["kind"] == "shock3v" else 4, device=DEV, dtype=F64)
    if case["kind"] == "single":
        st["cfg"] = _config(case)
    elif case["kind"] == "shock3v":
        st["solver"] = S.Solver3v(_config3v(case))
    else:
        st["solver"] = S.Solver(_config(case))
    return st


def run(st):
    kind = st["kind"]
    if kind == "single":
        B.bgk_step_noalloc(st["cfg"], st["f0"], st["out"], st["mom"])
        return [st["out"], st["mom"]]
    if kind == "gradient":
        J = A.lid_shear_fn(st["f0"], st["kn"], st["lid"], st["spec"])
        return [J.detach(), *torch.autograd.grad(J, (st["f0"], st["kn"], st["lid"]))]
    steps = st["case"]["steps"]
    if kind == "batch":
        b = st["batch"]
        for s, f0 in zip(b.solvers, st["f0"]):
            s.set_state(f0)
        b.step(steps)
        for s, out, mom in zip(b.solvers, st["out"], st["mom"]):
            s.get_state(out)
            s.moments(0, mom)
        return st["out"] + st["mom"]
    s = st["solver"]
    s.set_state(st["f0"])
    s.step(steps)
    s.get_state(st["out"])
    s.moments(0, st["mom"])
    return [st["out"], st["mom"]]


def _work(c):
    pts = c["nx"] * c["nvx"] * (1 if c["kind"] == "shock" else c["nvy"]) * (c["nvz"] if c["kind"] == "shock3v" else 1)
    pts *= 1 if c["kind"] in ("shock", "shock3v") else c["ny"]
    n = c["steps"]
    if c["kind"] == "gradient":
        # forward: read and write f; reverse: read f and the adjoint, write the adjoint
        return {"bytes": pts * n * (32 + 48), "flops": pts * n * (24 + 37)}
    if c["kind"] == "single":
        return {"bytes": pts * 32, "flops": pts * 24}
    if c["kind"] == "shock3v":
        # the caller's state in and out, a read and a write of the state per step
        return {"bytes": pts * 8 * 2 * (1 + n), "flops": pts * 16 * n}
    stored = STATE_BYTES[c["precision"]]
    return {"bytes": pts * (2 * 16 + 2 * stored * n), "flops": pts * (18 if c["kind"] == "shock" else 24) * n}


def work(case):
    if case["kind"] != "batch":
        return _work(case)
    parts = [_work(dict(_from_workload(w), steps=case["steps"])) for w in _instances(case)]
    return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}


def tolerance(case):
    # about four times what the library and exact() differ by (2-norm): 6.5e-15 (gradient), 4e-15 (FP64),
    # 3e-7 (FP32), 1.1e-4 (BF16 deviations, whose stores are rounded stochastically); single values of a
    # state lie up to some tens of times further off, against the root mean square
    if case["kind"] == "gradient":
        return {"rel": 4e-14, "max": 2e-12}
    if case["precision"] == "f64":
        return {"rel": 2e-14, "max": 1e-12}
    if case["precision"] == "bf16":
        return {"rel": 5e-4, "max": 2e-2}
    return {"rel": 1.5e-6, "max": 5e-5}


# --------------------------------------------------------------------------
# the same in plain FP64 torch
# --------------------------------------------------------------------------
def _axis_sums(c, u, inv):
    """Gaussian of one axis (cells, n) and its sums of 1, d, d^2."""
    d = c - u[:, None]
    e = torch.exp(-d * d * inv[:, None])
    return e, e.sum(1), (d * e).sum(1), (d * d * e).sum(1)


def _effective(q, axes, dv, hidden):
    """Parameters p = (n, u..., theta) whose discrete moments equal q; ``hidden``: integrated-out components."""
    p = list(q)
    for _ in range(20):
        inv = 1.0 / p[-1]
        dens, th = p[0] * (math.pi * p[-1]) ** (-0.5 * len(axes)) * dv, 0.5 * hidden * p[-1]
        mean = []
        for c, u in zip(axes, p[1:-1]):
            _, s0, s1, s2 = _axis_sums(c, u, inv)
            dens, m = dens * s0, s1 / s0
            mean.append(u + m)
            th = th + s2 / s0 - m * m
        r = [a - b for a, b in zip(q, [dens, *mean, (2.0 / 3.0) * th])]
        p = [a + b for a, b in zip(p, r)]
        if max(float(x.abs().max()) for x in r) < 1e-15:
            break
    return p


def _weights(c, n, th, dt):
    nu = n * th ** (1.0 - c["omega"])
    return 1.0 - torch.exp(-nu * dt) if c["relax_exact"] else nu * dt


def _grid2d(c, kn=None, lid=None):
    """Numbers of one cavity; kn and lid may be tensors that carry a gradient."""
    p = dict(c, cx=_centres(-c["vbox"], c["vbox"], c["nvx"]), cy=_centres(-c["vbox"], c["vbox"], c["nvy"]))
    lx, ly = _lengths(c)
    top = [float(p[k].abs().max()) for k in ("cx", "cy")]
    dx, dy = lx / c["nx"], ly / c["ny"]
    dt = c["cfl"] / (top[0] / dx + top[1] / dy)
    p.update(ax=p["cx"].abs() * dt / dx, ay=p["cy"].abs() * dt / dy, dv=(2.0 * c["vbox"]) ** 2 / (c["nvx"] * c["nvy"]))
    scale = 1.0 if kn is None else c["kn"] / kn  # lengths and the time step together
    p.update(dt=dt * scale, dx=dx * scale, u_lid=c["lid"] if lid is None else lid)
    return p


def _wall(p, u):
    """Unit-density wall Maxwellian (nvy, nvx, 2) at tangential speed u along x, theta = 1."""
    g = torch.exp(-p["cy"][:, None] ** 2 - (p["cx"] - u) ** 2) / math.pi
    return torch.stack([g, 0.5 * g], -1)


def _outside(p, f, axis, sign):
    """Boundary values beyond one face for its cells' states f (cells, nvy, nvx, 2); sign: of the inward normal."""
    if p["wall"] == "specular":
        return f.flip(2 if axis == "x" else 1)
    cn = sign * (p["cx"].expand(p["nvy"], -1) if axis == "x" else p["cy"][:, None].expand(-1, p["nvx"]))
    wall = _wall(p, p["u_lid"] if (axis, sign) == ("y", -1) else 0.0)
    inc = ((-cn).clamp(min=0.0) * f[..., 0]).sum((1, 2))
    nw = inc / (cn.clamp(min=0.0) * wall[..., 0]).sum()
    return nw[:, None, None, None] * wall


def _moments2d(p, f):
    """n, ux, uy, theta per cell of f (cells, nvy, nvx, 2)."""
    g = f[..., 0]
    gx, gy = g.sum(1), g.sum(2)
    s0, sx, sy = gx.sum(1), (gx * p["cx"]).sum(1), (gy * p["cy"]).sum(1)
    se = (gx * p["cx"] ** 2).sum(1) + (gy * p["cy"] ** 2).sum(1) + f[..., 1].sum((1, 2))
    ux, uy = sx / s0, sy / s0
    return [s0 * p["dv"], ux, uy, (2.0 / 3.0) * (se / s0 - ux * ux - uy * uy)]


def _step2d(p, f):
    """One step of the (ny, nx, nvy, nvx, 2) state."""
    ny, nx = p["ny"], p["nx"]
    lo, hi = _outside(p, f[:, 0], "x", 1)[:, None], _outside(p, f[:, -1], "x", -1)[:, None]
    right = (p["cx"] > 0)[:, None]
    fx = torch.where(right, torch.cat([lo, f[:, :-1]], 1), torch.cat([f[:, 1:], hi], 1))
    ft = f + p["ax"][:, None] * (fx - f)
    del fx
    lo, hi = _outside(p, f[0], "y", 1)[None], _outside(p, f[-1], "y", -1)[None]
    upward = (p["cy"] > 0)[:, None, None]
    fy = torch.where(upward, torch.cat([lo, f[:-1]], 0), torch.cat([f[1:], hi], 0))
    ft = (ft + p["ay"][:, None, None] * (fy - f)).reshape(ny * nx, p["nvy"], p["nvx"], 2)
    del fy
    q = _moments2d(p, ft)
    a = _weights(p, q[0], q[3], p["dt"])[:, None, None]
    e = q
    if p["conservative"]:
        with torch.no_grad():
            exact_p = _effective([x.detach() for x in q], [p["cx"], p["cy"]], p["dv"], 1)
        e = [x + (y - x.detach()) for x, y in zip(q, exact_p)]  # the map's derivative is the identity
    inv = 1.0 / e[3]
    px = torch.exp(-(p["cx"] - e[1][:, None]) ** 2 * inv[:, None])
    py = torch.exp(-(p["cy"] - e[2][:, None]) ** 2 * inv[:, None]) * (e[0] * inv / math.pi)[:, None]
    phi = px[:, None, :] * py[:, :, None]
    kappa = (0.5 * e[3])[:, None, None]
    out = torch.stack([ft[..., 0] + a * (phi - ft[..., 0]), ft[..., 1] + a * (kappa * phi - ft[..., 1])], -1)
    return out.reshape(ny, nx, p["nvy"], p["nvx"], 2)


def _lid_shear(p, f):
    top = f[-1]
    nw_wall = _outside(p, top, "y", -1)
    crossing = torch.where((p["cy"] > 0)[:, None], top[..., 0], nw_wall[..., 0])
    return p["dx"] * p["dv"] * (crossing * p["cx"] * -p["cy"][:, None]).sum()


def _exact1d(c, f):
    cx = _centres(-c["vbox"], c["vbox"], c["nvx"])
    dx = c["length"] / c["nx"]
    dt = c["cfl"] * dx / float(cx.abs().max())
    dv = 2.0 * c["vbox"] / c["nvx"]
    courant = cx * dt / dx
    shift, far = courant.trunc(), torch.where(cx > 0, 1.0, -1.0)
    r = (courant - shift).abs()[:, None]
    ends = []
    for n, u, th in _ends(c["mach"]):
        g = n / math.sqrt(math.pi * th) * torch.exp(-(cx - u) ** 2 / th)
        ends.append(torch.stack([g, th * g], -1)[None])
    i1 = (torch.arange(c["nx"], device=DEV)[:, None] - shift.long()).clamp(-1, c["nx"]) + 1
    i2 = (torch.arange(c["nx"], device=DEV)[:, None] - (shift + far).long()).clamp(-1, c["nx"]) + 1
    j = torch.arange(c["nvx"], device=DEV)
    for _ in range(c["steps"]):
        wide = torch.cat([ends[0], f, ends[1]], 0)
        ft = (1.0 - r) * wide[i1, j] + r * wide[i2, j]
        s0, s1 = ft[..., 0].sum(1), (cx * ft[..., 0]).sum(1)
        u = s1 / s0
        th = (2.0 / 3.0) * (((cx * cx) * ft[..., 0] + ft[..., 1]).sum(1) / s0 - u * u)
        q = [s0 * dv, u, th]
        a = _weights(c, q[0], th, dt)[:, None]
        p = _effective(q, [cx], dv, 2) if c["conservative"] else q
        phi = (p[0] / torch.sqrt(math.pi * p[2]))[:, None] * torch.exp(-(cx - p[1][:, None]) ** 2 / p[2][:, None])
        f = torch.stack([ft[..., 0] + a * (phi - ft[..., 0]), ft[..., 1] + a * (p[2][:, None] * phi - ft[..., 1])], -1)
    s0, u = f[..., 0].sum(1), (cx * f[..., 0]).sum(1) / f[..., 0].sum(1)
    th = (2.0 / 3.0) * (((cx * cx) * f[..., 0] + f[..., 1]).sum(1) / s0 - u * u)
    return [f, torch.stack([s0 * dv, u, torch.zeros_like(u), th], 1)]


def _moments3v(ax, dv, f):
    """n, ux, uy, uz, theta of f (cells, nvz, nvy, nvx)."""
    m = [f.sum((1, 2)), f.sum((1, 3)), f.sum((2, 3))]
    s0 = m[0].sum(1)
    u = [(x * c).sum(1) / s0 for x, c in zip(m, ax)]
    e = sum((x * c * c).sum(1) for x, c in zip(m, ax)) / s0
    return [s0 * dv, *u, (2.0 / 3.0) * (e - u[0] ** 2 - u[1] ** 2 - u[2] ** 2)]


def _exact3v(c, f):
    ax = [_centres(c["vx0"], c["vx1"], c["nvx"]), _centres(-c["vt"], c["vt"], c["nvy"]),
          _centres(-c["vt"], c["vt"], c["nvz"])]
    nx, dx, dt = c["nx"], c["length"] / c["nx"], c["dt"]
    dv = (c["vx1"] - c["vx0"]) / c["nvx"] * (2.0 * c["vt"]) ** 2 / (c["nvy"] * c["nvz"])
    courant = [float(x) * dt / dx for x in ax[0]]
    ends = []
    for n, u, th in _ends(c["mach"]):
        ends.append(n * (math.pi * th) ** -1.5 * torch.exp(
            -((ax[0] - u) ** 2 + ax[1][:, None] ** 2 + ax[2][:, None, None] ** 2) / th))
    f = f.reshape(nx, c["nvz"], c["nvy"], c["nvx"])
    cells = torch.arange(nx, device=DEV)
    for _ in range(c["steps"]):
        wide = torch.cat([ends[0][None], f, ends[1][None]], 0)
        ft = torch.empty_like(f)
        for j, k in enumerate(courant):
            s = math.trunc(k)
            i1, i2 = ((cells - m).clamp(-1, nx) + 1 for m in (s, s + (1 if k > 0 else -1)))
            ft[..., j] = (1.0 - abs(k - s)) * wide[i1, :, :, j] + abs(k - s) * wide[i2, :, :, j]
        q = _moments3v(ax, dv, ft)
        a = _weights(c, q[0], q[4], dt)
        p = _effective(q, ax, dv, 0) if c["conservative"] else q
        e = [torch.exp(-(x - u[:, None]) ** 2 / p[4][:, None]) for x, u in zip(ax, p[1:4])]
        e[0] = e[0] * (a * p[0] * (math.pi * p[4]) ** -1.5)[:, None]
        f = ft.mul_((1.0 - a)[:, None, None, None]).add_(
            e[0][:, None, None, :] * e[1][:, None, :, None] * e[2][:, :, None, None])
    return [f.reshape(nx, -1), torch.stack(_moments3v(ax, dv, f), 1)]


def _exact2d(c, f):
    p = _grid2d(c)
    f = f.reshape(c["ny"], c["nx"], c["nvy"], c["nvx"], 2)
    for _ in range(c["steps"]):
        f = _step2d(p, f)
    cells = f.reshape(c["ny"] * c["nx"], c["nvy"], c["nvx"], 2)
    return [cells.reshape(c["ny"] * c["nx"], -1, 2), torch.stack(_moments2d(p, cells), 1)]


def _exact_single(c, f):
    """One step's state and the moments of its streamed state (relaxation off: the step's relaxation keeps n and U)."""
    p = _grid2d(c)
    f = f.reshape(c["ny"], c["nx"], c["nvy"], c["nvx"], 2)
    out = _step2d(p, f)
    still = _step2d(dict(p, dt=0.0, conservative=0), f)  # a = 0: streaming alone
    cells = still.reshape(c["ny"] * c["nx"], c["nvy"], c["nvx"], 2)
    return [out.reshape(c["ny"] * c["nx"], -1, 2), torch.stack(_moments2d(p, cells), 1)]


def _exact_gradient(c, f0):
    kn = torch.tensor(c["kn"], device=DEV, dtype=F64, requires_grad=True)
    lid = torch.tensor(c["lid"], device=DEV, dtype=F64, requires_grad=True)
    f0.requires_grad_()
    f = f0.reshape(c["ny"], c["nx"], c["nvy"], c["nvx"], 2)

    def one(x, k, u):
        return _step2d(_grid2d(c, k, u), x)

    for _ in range(c["steps"]):
        f = checkpoint(one, f, kn, lid, use_reentrant=False)
    J = _lid_shear(_grid2d(c, kn, lid), f)
    gf, gk, gl = torch.autograd.grad(J, (f0, kn, lid))
    return [J.detach(), gf, gk.cpu(), gl.cpu()]


def exact(case, seed):
    if case["kind"] == "batch":
        states, moms = [], []
        for i, w in enumerate(_instances(case)):
            c = dict(_from_workload(w), steps=case["steps"])
            f, m = (_exact1d if c["kind"] == "shock" else _exact2d)(c, _initial(c, seed + 1000 * i))
            states.append(f)
            moms.append(m)
        return states + moms
    f0 = _initial(case, seed)
    if case["kind"] == "gradient":
        return _exact_gradient(case, f0)
    with torch.no_grad():
        if case["kind"] == "single":
            return _exact_single(case, f0)
        if case["kind"] == "shock":
            return _exact1d(case, f0)
        if case["kind"] == "shock3v":
            return _exact3v(case, f0)
        return _exact2d(case, f0)
