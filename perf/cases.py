"""The calls that users of this framework make, as cases that can be timed and checked.

Kinds of case:

- frame: one control frame of a living scene.  The controller sets the tools'
  target poses, steps a few sub-steps and reads the whole state on the device.
  The tools swing to and fro (0.2 s a cycle), so that a scene can be stepped
  for as long as one likes.
- batch: the same for many environments behind one handle (reinforcement
  learning), each with its own size, material and tool.
- reset: the start of an episode: a saved state is loaded, the tool is put in
  its place, one short rollout runs and the state is read.
- grad: a differentiable rollout and its gradients with respect to the
  material, the tool poses and the initial state.
- surface: the triangles of the tissue's surface, once per rendered frame.

A body is a box of tissue on the floor of the grid: `aspect` times as wide and
deep as it is high, with `ppc` particles per grid cell (bodies at 8 and more on
a jittered lattice, the others at random places).  It starts in motion: smooth
velocities with their gradient as C, smooth deformations as F.
"""
import ctypes as ct
import math

import numpy as np
import torch

from paper_2402_01181_gb300 import autodiff, mpm

RHO, BOUND, G = 1e3, 3, (0.0, -9.8, 0.0)
DT = {32: 1e-4, 64: 5e-5, 128: 2e-5, 256: 2e-5}
RADIUS, HALF = 0.02, 0.15            # the capsule tool
BOX = (0.04, 0.01, 0.03)             # half extents of the plate tool
CYCLE, PRESS, DRAG = 0.2, 0.008, 0.01        # the tools' swing: seconds, depth and sideways in metres
FIELD_RES = 256                      # samples per axis of the sampled grasper
ENV_E, ENV_NU = (8e3, 2e4), (0.2, 0.42)


def listed():
    frame = {"kind": "frame", "E": 1e4, "nu": 0.35, "friction": 0.3, "tools": "capsule", "substeps": 25}
    return [
        # the innermost loop of a haptic controller: a small patch of tissue, a few sub-steps a call
        dict(frame, name="servo_2k", particles=2003, grid=32, ppc=16.0, aspect=1.0, substeps=4),
        # a small scene at a frame's usual length
        dict(frame, name="frame_8k", particles=8192, grid=32, ppc=16.0, aspect=1.0, E=2e4, nu=0.3),
        # the tissue slab of the paper's scale under a capsule instrument
        dict(frame, name="frame_30k", particles=30000, grid=64, ppc=3.18, aspect=6.0),
        # the same slab under a grasper given as a sampled distance field
        dict(frame, name="frame_30k_sdf", particles=30000, grid=64, ppc=3.18, aspect=6.0, tools="sampled"),
        # a finer slab, an odd count, two instruments, a frame of odd length
        dict(frame, name="frame_200k_two_tools", particles=200003, grid=128, ppc=3.3, aspect=6.0, tools="capsule+box",
             substeps=17, friction=0.2),
        # an organ-sized block of a million particles
        dict(frame, name="frame_1m", particles=1000000, grid=128, ppc=8.0, aspect=1.0, E=5e4, nu=0.3),
        # the largest scene: 8 million particles on the 256^3 grid
        dict(frame, name="frame_8m", particles=8000000, grid=256, ppc=8.0, aspect=1.0, E=5e4, nu=0.3),
        # reinforcement learning: 256 slabs of 5 to 40 thousand particles stepped together
        {"name": "batch_256", "kind": "batch", "envs": 256, "n_min": 5000, "n_max": 40000, "grid": 64, "ppc": 3.18,
         "aspect": 6.0, "friction": 0.3, "substeps": 25},
        # the start of an episode at the paper's scale
        dict(frame, name="reset_30k", kind="reset", particles=30000, grid=64, ppc=3.18, aspect=6.0),
        # system identification and trajectory optimisation at the paper's scale
        dict(frame, name="grad_30k", kind="grad", particles=30000, grid=64, ppc=3.18, aspect=6.0, substeps=100,
             checkpoint=25),
        # the surface for the renderer, of a slab on the 128^3 grid
        {"name": "surface_300k", "kind": "surface", "particles": 300000, "grid": 128, "ppc": 4.0, "aspect": 6.0},
    ]


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "frame", "batch", "reset", "grad", "surface"])

    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "batch":
        n_min = log(1000, 8000)
        return {"kind": "batch", "envs": log(8, 200), "n_min": n_min, "n_max": n_min * rng.randint(2, 5), "grid": 64,
                "ppc": round(rng.uniform(2.5, 4.0), 2), "aspect": 6.0, "friction": rng.choice([0.0, 0.3]),
                "substeps": rng.randint(5, 30)}
    grid = rng.choice([64, 128] if kind == "surface" else [32, 64] if kind == "grad" else [32, 64, 128, 256])
    most = {32: 20000, 64: 120000, 128: 1500000, 256: 6000000}[grid]
    least = {32: 1000, 64: 6000, 128: 60000, 256: 500000}[grid]
    c = {"kind": kind, "particles": log(least, min(most, 40000) if kind == "grad" else most), "grid": grid}
    c["ppc"] = round(rng.uniform(2.0, 6.0) if rng.random() < 0.5 else rng.uniform(8.0, 12.0), 2)
    if grid == 32:
        c["ppc"] = round(rng.uniform(8.0, 16.0), 2)
    c["aspect"] = rng.choice([1.0, 3.0, 6.0])
    while _box(c)[1][0] > 0.8 or _box(c)[1][1] > 0.5:        # the body has to fit the grid
        c["particles"] = int(c["particles"] * 0.8)
    if kind == "surface":
        return c
    c["nu"] = round(rng.uniform(0.2, 0.4), 3)
    c["E"] = float(round(rng.uniform(1.0, 4.0) * max(1e4, 4 * RHO * 9.8 * _box(c)[1][1])))
    c["friction"] = rng.choice([0.0, 0.2, 0.4])
    c["tools"] = "capsule" if kind == "grad" else rng.choice(["capsule", "capsule", "box", "capsule+box", "sampled"])
    c["substeps"] = rng.randint(20, 100) if kind == "grad" else rng.randint(1, 25)
    if kind == "grad":
        c["checkpoint"] = rng.randint(10, 50)
    return c


# ------------------------------------------------------------------ inputs

def _box(case, particles=None):
    """Lower corner and size of the body, in metres (the grid covers the unit cube)."""
    dx = 1.0 / case["grid"]
    volume = (particles or case["particles"]) / case["ppc"] * dx ** 3
    h = (volume / case["aspect"] ** 2) ** (1.0 / 3.0)
    w = case["aspect"] * h
    return (0.5 - w / 2, BOUND * dx, 0.5 - w / 2), (w, h, w)


def _body(case, seed, particles=None):
    """x, v, F, C of one body (CUDA, 32 bits) and its particles' volume."""
    n = particles or case["particles"]
    lo, size = _box(case, n)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    x = torch.rand((n, 3), generator=gen, device="cuda", dtype=torch.float32)
    if case["ppc"] >= 8:             # a jittered lattice, layer by layer from the floor
        s = 1.0 / case["grid"] / case["ppc"] ** (1.0 / 3.0)
        nx = max(1, round(size[0] / s))
        p = torch.arange(n, device="cuda")
        x = (x + torch.stack([p % nx, p // (nx * nx), p // nx % nx], 1)) * (size[0] / nx)
    else:
        x = x * torch.tensor(size, device="cuda")
    x = x + torch.tensor(lo, device="cuda")
    # smooth fields: a_i sin(k_i . x + b_i) for each component of v, then of F - I
    r = np.random.default_rng(seed)
    k = torch.tensor(r.uniform(-12.0, 12.0, (12, 3)), device="cuda", dtype=torch.float32)
    b = torch.tensor(r.uniform(0.0, 6.28, 12), device="cuda", dtype=torch.float32)
    phase = x @ k.T + b
    v = 0.1 * torch.sin(phase[:, :3])
    C = 0.1 * torch.cos(phase[:, :3])[:, :, None] * k[:3]
    F = torch.eye(3, device="cuda") + 0.02 * torch.sin(phase[:, 3:]).reshape(n, 3, 3)
    return x.contiguous(), v.contiguous(), F.reshape(n, 9).contiguous(), C.reshape(n, 9).contiguous(), \
        size[0] * size[1] * size[2] / n


def _shape(kind):
    s = np.zeros(8, np.float32)
    if kind == "capsule":
        s[:3] = (mpm.MPM_TOOL_CAPSULE, RADIUS, HALF)
    elif kind == "box":
        s[:4] = (mpm.MPM_TOOL_BOX, *BOX)
    else:
        s[0] = mpm.MPM_TOOL_SAMPLED
    return s


def _pose(case, seed, tool, t, particles=None):
    """Pose (T, rotation vector) of tool number `tool` at simulated time t: pressed into the top of the body, swinging."""
    lo, size = _box(case, particles)
    kind = _tools(case)[tool]
    reach = {"capsule": RADIUS + HALF, "box": BOX[1], "sampled": 0.19}[kind]
    r = np.random.default_rng([seed, 77, tool])
    side = 0.15 * size[0]
    a, off = 2 * math.pi * t / CYCLE, r.uniform(-side, side, 2)
    if tool == 1:
        off[0] += 0.25 * size[0]
    top = lo[1] + size[1] + reach - PRESS * (1.0 + 0.5 * math.sin(a))
    return np.array([0.5 + off[0] + DRAG * math.sin(0.7 * a), top, 0.5 + off[1], 0.03, 0.2 + 0.1 * math.sin(a), 0.05])


def _tools(case):
    return case.get("tools", "capsule").split("+")


def _grasper():
    """Distances to a grasper (a shaft and two jaws below it) on a cubic lattice: samples[z, y, x], origin, spacing."""
    res, side = FIELD_RES, 0.39
    h = side / (res - 6.6)
    o = torch.tensor([-0.5 * side - 3.3 * h, -0.19 - 3.3 * h, -0.5 * side - 3.3 * h], device="cuda", dtype=torch.float64)
    a = torch.arange(res, device="cuda", dtype=torch.float64) * h
    z, y, x = torch.meshgrid(a + o[2], a + o[1], a + o[0], indexing="ij")
    d = torch.sqrt(x ** 2 + (y - y.clamp(-0.12, 0.18)) ** 2 + z ** 2) - RADIUS
    for cx in (0.024, -0.024):
        q = [(x - cx).abs() - 0.012, (y + 0.16).abs() - 0.03, z.abs() - 0.02]
        out = torch.sqrt(sum(c.clamp(min=0) ** 2 for c in q))
        d = torch.minimum(d, out + torch.maximum(torch.maximum(q[0], q[1]), q[2]).clamp(max=0))
    return d.float().contiguous(), o.cpu().numpy(), h


def _grad_poses(case, seed):
    dt = DT[case["grid"]]
    return np.stack([_pose(case, seed, 0, dt * (k + 1)) for k in range(case["substeps"])])[:, None, :]


def _grad_weights(case, seed):
    """dL/d(final x, v, F, C) of the loss."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + 1)
    n = case["particles"]
    w = [torch.rand((n, c), generator=gen, device="cuda") - 0.25 for c in (3, 3, 9, 9)]
    return [w[0], 1e-3 * w[1], 1e-3 * w[2], 1e-6 * w[3]]


def _envs(case, seed):
    sizes, r = np.random.default_rng(case["envs"]), np.random.default_rng(seed)
    return [{"particles": int(sizes.integers(case["n_min"], case["n_max"] + 1)), "seed": int(r.integers(1 << 30)),
             "E": float(r.uniform(*ENV_E)), "nu": float(r.uniform(*ENV_NU))} for _ in range(case["envs"])]


def _new_sim(case, n, **kw):
    cfg = mpm.make_config(case["grid"], DT[case["grid"]], case.get("E", 1e4), case.get("nu", 0.3), RHO, gravity=G,
                          bound=BOUND, friction=case.get("friction", 0.0), max_particles=n, **kw)
    return mpm.Sim(cfg)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case, "seed": seed, "frame": 0}
    if kind == "batch":
        envs = _envs(case, seed)
        bodies = [_body(case, e["seed"], e["particles"]) for e in envs]
        n = sum(e["particles"] for e in envs)
        sim = _new_sim(case, n, n_envs=len(envs))
        for i, e in enumerate(envs):
            sim.set_env_material(i, e["E"], e["nu"], RHO)
        parts = [torch.cat([b[q] for b in bodies]) for q in range(4)]
        vol = np.array([b[4] for b in bodies], np.float32)
        counts = (ct.c_int64 * len(envs))(*[e["particles"] for e in envs])
        mpm.check(mpm.mpm_load_batch(sim.h, counts, *[ct.c_void_p(p.data_ptr()) for p in parts],
                                     vol.ctypes.data_as(ct.POINTER(ct.c_float)), 1))
        torch.cuda.synchronize()
        sim.n = n
        s.update(sim=sim, envs=envs, shape=_shape("capsule"))
        for i, e in enumerate(envs):
            sim.set_env_tool(i, 0, _pose(case, e["seed"], 0, 0.0, e["particles"]), s["shape"])
    else:
        x, v, F, C, vol = _body(case, seed)
        n = case["particles"]
        sim = _new_sim(case, n)
        s.update(sim=sim, body=(x, v, F, C), vol=vol, tools=[_shape(k) for k in _tools(case)])
        for shape in s["tools"]:
            if shape[0] == mpm.MPM_TOOL_SAMPLED:
                shape[1] = sim.add_field(*_grasper())
        if kind != "grad":
            sim.load(x, vol, v, F, C)
            _place(s)
        if kind == "grad":
            s.update(E=torch.tensor(case["E"], dtype=torch.float64, requires_grad=True),
                     nu=torch.tensor(case["nu"], dtype=torch.float64, requires_grad=True),
                     poses=torch.tensor(_grad_poses(case, seed), requires_grad=True),
                     start=[p.clone().requires_grad_(True) for p in (x, v, F, C)], weights=_grad_weights(case, seed))
    if kind == "surface":            # the renderer's vertex buffer
        s["triangles"] = torch.zeros((_room(case), 3, 3), device="cuda")
    else:
        s["out"] = [torch.empty((n, c), device="cuda") for c in (3, 3, 9, 9)]
    torch.cuda.synchronize()
    return s


def _place(s):
    """Put every tool at its starting pose, at rest."""
    for i, shape in enumerate(s["tools"]):
        s["sim"].set_tool(i, np.zeros(6), [mpm.MPM_TOOL_NONE] + [0.0] * 7)
        s["sim"].set_tool(i, _pose(s["case"], s["seed"], i, 0.0), shape)


def _aim(s):
    """Give every tool its target at the end of the next frame."""
    case = s["case"]
    s["frame"] += 1
    t = s["frame"] * case["substeps"] * DT[case["grid"]]
    if case["kind"] == "batch":
        for i, e in enumerate(s["envs"]):
            s["sim"].set_env_tool(i, 0, _pose(case, e["seed"], 0, t, e["particles"]), s["shape"])
    else:
        for i, shape in enumerate(s["tools"]):
            s["sim"].set_tool(i, _pose(case, s["seed"], i, t), shape)


# --------------------------------------------------------------- the calls

def run(s):
    case, sim = s["case"], s["sim"]
    if case["kind"] == "surface":
        tri, count = s["triangles"], ct.c_int64()
        mpm.check(mpm.mpm_extract_surface(sim.h, 0, 0.5, ct.c_void_p(tri.data_ptr()), len(tri), ct.byref(count), 1))
        return [tri, count.value]
    if case["kind"] == "grad":
        _place(s)
        x, v, F, C = s["start"]
        out = autodiff.rollout(sim, s["E"], s["nu"], s["poses"], x, s["vol"], v, F, C, case["checkpoint"])
        grads = torch.autograd.grad(out, [s["E"], s["nu"], s["poses"], x, v, F, C], s["weights"])
        return list(out) + [g.float() for g in grads]
    if case["kind"] == "reset":
        x, v, F, C = s["body"]
        sim.load(x, s["vol"], v, F, C)
        _place(s)
        s["frame"] = 0
    _aim(s)
    sim.step(case["substeps"])
    sim.read_device(*s["out"])
    return s["out"]


# ------------------------------------------------------------ their work

# FP32 operations of one particle and sub-step: P2G (27 nodes, about 17 each), G2P with the moments (27 nodes, about
# 20 each), the F update and the stress (about 200); the reverse of a sub-step takes about twice that
FLOPS = 1200.0


def _area(case):
    """Surface of the body in grid cells; each gives about 10 triangles."""
    _, size = _box(case)
    return (2 * size[0] ** 2 + 4 * size[0] * size[1]) * case["grid"] ** 2


def _room(case):
    return int(20 * _area(case)) + 1000


def work(case):
    n = (case["n_min"] + case["n_max"]) / 2 * case["envs"] if case["kind"] == "batch" else case["particles"]
    if case["kind"] == "surface":
        return {"bytes": 4.0 * case["grid"] ** 3 + 36.0 * 10 * _area(case), "flops": 300.0 * _area(case)}
    w = {"bytes": 2 * 96.0 * n, "flops": FLOPS * n * case["substeps"]}
    if case["kind"] == "grad":       # the rollout, its repetition from the checkpoints, and the reverse
        w = {"bytes": 4 * 96.0 * n, "flops": 4 * w["flops"]}
    return w


# ------------------------------------------- the same in 64 bits, in torch

def _rotation(r):
    """exp of the rotation vector r (not zero)."""
    a = torch.linalg.norm(r)
    z = torch.zeros_like(a)
    K = torch.stack([z, -r[2], r[1], r[2], z, -r[0], -r[1], r[0], z]).reshape(3, 3)
    return torch.eye(3, dtype=r.dtype, device=r.device) + torch.sin(a) / a * K + (1 - torch.cos(a)) / a ** 2 * (K @ K)


def _frame(p0, p1, s, span):
    """R, T, u, w of a tool a share s into a uniform motion from pose p0 to p1 over `span` seconds."""
    R0 = _rotation(p0[3:])
    M = _rotation(p1[3:]) @ R0.T
    q = 0.5 * torch.stack([M[2, 1] - M[1, 2], M[0, 2] - M[2, 0], M[1, 0] - M[0, 1]])   # sin(a) times the axis
    s2 = (q * q).sum()
    phi = q * (1 + s2 / 6 + 3 * s2 ** 2 / 40 + 15 * s2 ** 3 / 336)                     # asin's series: a is small
    a = torch.sqrt((phi.detach() ** 2).sum())
    if s == 1:
        R = _rotation(p1[3:])
    else:
        R = (_rotation(s * phi) if float(a) > 1e-12 else torch.eye(3, dtype=p0.dtype, device=p0.device)) @ R0
    return R, p0[:3] + s * (p1[:3] - p0[:3]), (p1[:3] - p0[:3]) / span, phi / span


def _distance(kind, p, field):
    """Distance and unit normal at the tool-frame points p."""
    if kind == "capsule":
        q = torch.stack([p[:, 0], p[:, 1] - p[:, 1].clamp(-HALF, HALF), p[:, 2]], 1)
        L = torch.linalg.norm(q, dim=1)
        return L - RADIUS, q / L[:, None]
    if kind == "box":
        q = p.abs() - torch.tensor(BOX, dtype=p.dtype, device=p.device)
        sign = torch.where(p < 0, -1.0, 1.0).to(p.dtype)
        o = q.clamp(min=0)
        on = torch.linalg.norm(o, dim=1)
        inner = torch.nn.functional.one_hot(q.argmax(1), 3).to(p.dtype)
        outside = (on > 0)[:, None]
        return torch.where(on > 0, on, q.max(1).values), sign * torch.where(outside, o / on.clamp(min=1e-300)[:, None], inner)
    f, o, h = field
    res = f.shape[0]
    c = torch.floor((p - torch.tensor(o, dtype=p.dtype, device=p.device)) / h)
    ok = ((c >= 0) & (c < res)).all(1)
    c = c.clamp(0, res - 1).long()
    g = []
    for a in range(3):
        hi, lo = c.clone(), c.clone()
        hi[:, a] = (hi[:, a] + 1).clamp(max=res - 1)
        lo[:, a] = (lo[:, a] - 1).clamp(min=0)
        g.append((f[hi[:, 2], hi[:, 1], hi[:, 0]].to(p.dtype) - f[lo[:, 2], lo[:, 1], lo[:, 0]].to(p.dtype))
                 / (hi[:, a] - lo[:, a]))
    g = torch.stack(g, 1)
    d = f[c[:, 2], c[:, 1], c[:, 0]].to(p.dtype)
    return torch.where(ok, d, torch.full_like(d, 1e30)), g / torch.linalg.norm(g, dim=1).clamp(min=1e-300)[:, None]


def _mul(a, b):
    return (a[:, :, :, None] * b[:, None]).sum(2)


def _det(F):
    return (F[:, 0] * torch.linalg.cross(F[:, 1], F[:, 2])).sum(1)


def _stencil(x, n):
    base = torch.floor(x.detach() * n - 0.5).long().clamp(0, n - 3)
    f = x * n - base
    return base, f, torch.stack([0.5 * (1.5 - f) ** 2, 0.75 - (f - 1) ** 2, 0.5 * (f - 0.5) ** 2])


def _scatter(x, v, C, F, E, nu, vol, n, dt):
    """Mass and momentum of the n^3 nodes."""
    mu, lam = E / (2 * (1 + nu)), E * nu / ((1 + nu) * (1 - 2 * nu))
    eye = torch.eye(3, dtype=x.dtype, device=x.device)
    m = RHO * vol
    tau = mu * (_mul(F, F.transpose(1, 2)) - eye) + (lam * torch.log(_det(F)))[:, None, None] * eye
    A = m * C - dt * vol * 4 * n * n * tau
    base, f, w = _stencil(x, n)
    grid = torch.zeros((n ** 3, 4), dtype=x.dtype, device=x.device)
    for o in range(27):
        off = torch.tensor([o % 3, o // 3 % 3, o // 9], device=x.device)
        wo = w[o % 3, :, 0] * w[o // 3 % 3, :, 1] * w[o // 9, :, 2]
        mom = m * v + (A * ((off - f) / n)[:, None, :]).sum(2)
        node = base + off
        grid = grid.index_add(0, (node[:, 0] * n + node[:, 1]) * n + node[:, 2],
                              wo[:, None] * torch.cat([torch.full_like(mom[:, :1], m), mom], 1))
    return grid, base, f, w


def _substep(x, v, C, F, E, nu, vol, n, dt, fric, tools):
    """tools: (kind, (R, T, u, w), field) each."""
    grid, base, f, w = _scatter(x, v, C, F, E, nu, vol, n, dt)
    live = torch.nonzero(grid[:, 0].detach() > 0)[:, 0]
    ijk = torch.stack([live // (n * n), live // n % n, live % n], 1)
    val = grid[live]
    vel = val[:, 1:] / val[:, :1] + dt * torch.tensor(G, dtype=x.dtype, device=x.device)
    pos = ijk.to(x.dtype) / n
    best = torch.full((len(live),), 1e30, dtype=x.dtype, device=x.device)
    normal, vco = torch.zeros_like(vel), torch.zeros_like(vel)
    for kind, (R, T, u, om), field in tools:
        rel = pos - T
        d, nr = _distance(kind, rel @ R, field)
        near = d.detach() < best
        best = torch.where(near, d.detach(), best)
        normal = torch.where(near[:, None], nr @ R.T, normal)
        vco = torch.where(near[:, None], u + torch.linalg.cross(om.expand_as(rel), rel), vco)
    hit = torch.nonzero((best < 0) & (((vel - vco) * normal).sum(1).detach() < 0))[:, 0]
    nh, ch = normal[hit], vco[hit]
    vr = vel[hit] - ch
    vn = (vr * nh).sum(1, keepdim=True)
    vt = vr - vn * nh
    tn = torch.linalg.norm(vt, dim=1, keepdim=True).clamp(min=1e-300)
    vel = vel.index_put((hit,), (1 + fric * vn / tn).clamp(min=0) * vt + ch)
    inside = ((ijk >= BOUND) & (ijk < n - BOUND)).all(1)
    vel = torch.where(inside[:, None], vel, torch.zeros_like(vel))
    vg = torch.zeros((n ** 3, 3), dtype=x.dtype, device=x.device).index_put((live,), vel)
    v, B = torch.zeros_like(v), torch.zeros_like(C)
    for o in range(27):
        off = torch.tensor([o % 3, o // 3 % 3, o // 9], device=x.device)
        node = base + off
        g = (w[o % 3, :, 0] * w[o // 3 % 3, :, 1] * w[o // 9, :, 2])[:, None] \
            * vg[(node[:, 0] * n + node[:, 1]) * n + node[:, 2]]
        v = v + g
        B = B + g[:, :, None] * ((off - f) / n)[:, None, :]
    C = 4 * n * n * B
    return x + dt * v, v, C, F + dt * _mul(C, F)


def _as64(body):
    n = len(body[0])
    x, v, F, C = (p.double() for p in body[:4])
    return x, v, C.reshape(n, 3, 3), F.reshape(n, 3, 3)


def _out(x, v, C, F):
    n = len(x)
    return [x, v, F.reshape(n, 9), C.reshape(n, 9)]


def _exact_frame(case, seed, body, E, nu, particles=None):
    """One frame of one body from its starting state."""
    n, S = case["grid"], case["substeps"]
    dt = float(np.float32(DT[n]))
    field = _grasper() if "sampled" in _tools(case) else None
    ends = [[torch.tensor(_pose(case, seed, i, t, particles)) for t in (0.0, S * DT[n])] for i in range(len(_tools(case)))]
    state = _as64(body)
    mat = (float(np.float32(E)), float(np.float32(nu)), float(np.float32(body[4])))
    for k in range(S):
        tools = [(kind, [q.cuda() for q in _frame(*ends[i], (k + 1) / S, S * dt)], field) for i, kind in enumerate(_tools(case))]
        state = _substep(*state, *mat, n, dt, float(np.float32(case["friction"])), tools)
    return _out(*state)


def _exact_grad(case, seed):
    n = case["grid"]
    dt = float(np.float32(DT[n]))
    body = _body(case, seed)
    vol = float(np.float32(body[4]))
    leaves = [p.double().requires_grad_(True) for p in body[:4]]
    E, nu = (torch.tensor(float(np.float32(case[k])), dtype=torch.float64, requires_grad=True) for k in ("E", "nu"))
    poses = torch.tensor(_grad_poses(case, seed), requires_grad=True)
    state = _as64(leaves)
    last = torch.tensor(_pose(case, seed, 0, 0.0))
    for k in range(case["substeps"]):
        frame = [q.cuda() for q in _frame(last, poses[k, 0], 1, dt)]
        state = _substep(*state, E.cuda(), nu.cuda(), vol, n, dt, float(np.float32(case["friction"])), [("capsule", frame, None)])
        last = poses[k, 0]
    out = _out(*state)
    weights = [w.double() for w in _grad_weights(case, seed)]
    return [p.detach() for p in out] + list(torch.autograd.grad(out, [E, nu, poses] + leaves, weights))


def _exact_surface(case, seed):
    """Marching tetrahedra of density 0.5: six tetrahedra around each cell's diagonal, in cell order (x fastest)."""
    n, body = case["grid"], _body(case, seed)
    vol = float(np.float32(body[4]))
    grid = _scatter(*_as64(body), 1e4, 0.3, vol, n, DT[n])[0]
    f = (grid[:, 0] * (n ** 3 / RHO)).reshape(n, n, n).permute(2, 1, 0)              # [z, y, x]
    corner = [(c & 1, c >> 1 & 1, c >> 2) for c in range(8)]
    cells = torch.stack([f[z:n - 1 + z, y:n - 1 + y, x:n - 1 + x].reshape(-1) for x, y, z in corner], 1)
    ins = cells >= 0.5
    idx = torch.nonzero(ins.any(1) & ~ins.all(1))[:, 0]
    cells, m = cells[idx], n - 1
    org = torch.stack([idx % m, idx // m % m, idx // (m * m)], 1).double()
    offs = torch.tensor(corner, dtype=torch.float64, device="cuda")
    tris, keys = [], []

    def emit(sel, q, t, edges):
        a, b = (torch.stack(e) for e in zip(*edges))                                 # (3, cells) corner numbers
        a, b = torch.minimum(a, b), torch.maximum(a, b)
        r = torch.arange(len(sel), device="cuda").expand_as(a)
        fa, fb = cells[sel][r, a], cells[sel][r, b]
        s = ((0.5 - fa) / (fb - fa))[:, :, None]
        tris.append(((org[sel] + offs[a] + s * (offs[b] - offs[a])) / n).permute(1, 0, 2))
        keys.append(idx[sel] * 12 + 2 * q + t)

    for q, (pa, pb) in enumerate(((1, 3), (1, 5), (2, 3), (2, 6), (4, 5), (4, 6))):
        t = [0, pa, pb, 7]
        if np.linalg.det(np.array([corner[c] for c in t[1:]], float)) < 0:
            t[1], t[2] = t[2], t[1]
        inside = cells[:, t] >= 0.5
        for code in range(1, 15):
            bits = [code >> r & 1 for r in range(4)]
            sel = torch.nonzero((inside == torch.tensor(bits, device="cuda", dtype=torch.bool)).all(1))[:, 0]
            c = [torch.full((len(sel),), v, device="cuda") for v in t]
            if sum(bits) != 2:
                lone = bits.index(1 if sum(bits) == 1 else 0)
                p = ((0, 1, 2, 3), (1, 0, 3, 2), (2, 0, 1, 3), (3, 0, 2, 1))[lone]
                e = [(c[p[0]], c[p[k]]) for k in (1, 2, 3)]
                emit(sel, q, 0, e if sum(bits) == 1 else [e[0], e[2], e[1]])
            else:
                p = [r for r in range(4) if bits[r]] + [r for r in range(4) if not bits[r]]
                if sum(p[i] > p[j] for i in range(4) for j in range(i + 1, 4)) & 1:
                    p[2], p[3] = p[3], p[2]
                P, Q, R, S = (c[r] for r in p)
                emit(sel, q, 0, [(P, R), (P, S), (Q, S)])
                emit(sel, q, 1, [(P, R), (Q, S), (Q, R)])
    tris = torch.cat(tris)[torch.argsort(torch.cat(keys))]
    return [torch.cat([tris, torch.zeros((_room(case) - len(tris), 3, 3), dtype=torch.float64, device="cuda")]), len(tris)]


def exact(case, seed):
    if case["kind"] == "surface":
        return _exact_surface(case, seed)
    if case["kind"] == "grad":
        return _exact_grad(case, seed)
    if case["kind"] == "batch":
        if case["envs"] * case["substeps"] > 2000:
            return None              # a sub-step of one environment takes about 10 ms this way
        envs = _envs(case, seed)
        outs = [_exact_frame(case, e["seed"], _body(case, e["seed"], e["particles"]), e["E"], e["nu"], e["particles"])
                for e in envs]
        return [torch.cat(p) for p in zip(*outs)]
    return _exact_frame(case, seed, _body(case, seed), case["E"], case["nu"])
