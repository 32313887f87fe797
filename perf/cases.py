"""The workloads whose speed is tracked, as a user's program runs them.

Every case goes through the public entry points (``Scene``, ``Mlp``,
``sph_marching_cubes``).  A pass that advances a scene loads its state, steps
and reads the state back, so that it is a function of the inputs alone
however often it is repeated.  Five kinds:

``step``
    one scene: load, n steps, read the state and the usual fields; from the
    4,096-particle dam-break to the 2,097,152-particle tank, with cubic and
    narrow cells, plain and graph-replayed steps, device and host buffers,
    the diagnostic fields, both coupling modes and obstacles.
``batch``
    many independent tanks of uneven size in one handle, graph-replayed.
``forces``
    the fluid force on every boid of a state, by one of the four modes.
``mlp``
    the boid-force network: inference, gradients, training steps.
``surface``
    the voxel density of a state, or marching cubes of a corner grid.

The states are made from the seed alone: jittered lattices (the dam-breaks
early in their collapse) and a fluid compressed towards the floor (the tank
after its settling), each under a smooth flow with a little noise.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2311_15088_gb300 import scenes
from paper_2311_15088_gb300.sph import (SPH_BOID_EXACT, SPH_BOID_EXACT_LOCAL, SPH_BOID_SURROGATE,
                                        SPH_BOID_SURROGATE_FALLBACK, Mlp, Scene, sph_marching_cubes,
                                        sph_mc_workspace_size)

DEV = "cuda"
H = scenes.default_params()["h"]
RHO0 = 1000.0
MODES = {"exact": SPH_BOID_EXACT, "local": SPH_BOID_EXACT_LOCAL, "surrogate": SPH_BOID_SURROGATE,
         "gated": SPH_BOID_SURROGATE_FALLBACK}
# cell sizes along (y and z, x) in units of h: the default, cubic h cells
# (the paper's), the batched scenes' and the large tank's
CELLS = {"half": (0.5, 0.0), "full": (1.0, 0.0), "full_halfx": (1.0, 0.5), "narrow": (0.5, 0.125)}
# the network: 272 inputs, three hidden layers of 256, 16 outputs (three
# force components, the error head, padding)
LAYERS = ((272, 256), (256, 256), (256, 256), (256, 16))
F_SCALE = 20.0  # the force one unit of network output stands for
# the input-range gate: boids faster than this along an axis fall back
GATE_SPEED = 0.95


def listed():
    return [
        # the smallest use: the paper-sized dam-break of the parity suite and
        # of an interactive loop, ten frames; launches and latency count
        dict(name="step_small", kind="step", layout="dam", n=4096, boids=16, spacing=0.5 * H, bx=1.0, by=1.0, bz=1.0,
             cells="half", steps=10, graph=False, host=False, diag=False, literal=False, const_set=0, spheres=0),
        # a debugging or analysis run of odd size: the paper's cubic cells and
        # literal coupling, obstacles, diagnostic fields read
        dict(name="step_diag", kind="step", layout="dam", n=33331, boids=77, spacing=0.5 * H, bx=1.0, by=1.0, bz=1.0,
             cells="full", steps=2, graph=False, host=False, diag=True, literal=True, const_set=0, spheres=5),
        # the dam-break column the surrogate's data is logged from
        dict(name="step_column", kind="step", layout="dam", n=262144, boids=1024, spacing=1.0 / 64.0,
             bx=2.0, by=1.0, bz=1.0, cells="half", steps=4, graph=True, host=False, diag=False, literal=False,
             const_set=0, spheres=0),
        # the same column driven from host memory, a step per round trip
        dict(name="step_host", kind="step", layout="dam", n=262144, boids=1024, spacing=1.0 / 64.0,
             bx=2.0, by=1.0, bz=1.0, cells="half", steps=1, graph=False, host=True, diag=False, literal=False,
             const_set=0, spheres=0),
        # the benchmark's tank, settled: the headline workload
        dict(name="step_tank", kind="step", layout="settled", n=2097152, boids=16384, spacing=0.0,
             bx=4.0, by=2.0, bz=2.0, cells="narrow", steps=2, graph=False, host=False, diag=False, literal=False,
             const_set=0, spheres=0),
        # independent scenes of uneven size, one graph (an RL farm's step)
        dict(name="batch_tanks", kind="batch", scenes=256, n_min=2048, n_max=65536, cells="full_halfx", steps=4,
             graph=True),
        # boid forces by the network with its gate, replayed (control loop)
        dict(name="forces_gated", kind="forces", layout="dam", n=262144, boids=1024, spacing=1.0 / 64.0,
             bx=2.0, by=1.0, bz=1.0, cells="half", mode="gated", graph=True),
        # exact boid forces of the tank from the needed densities alone
        dict(name="forces_local", kind="forces", layout="settled", n=2097152, boids=16384, spacing=0.0,
             bx=4.0, by=2.0, bz=2.0, cells="narrow", mode="local", graph=False),
        # bulk evaluation of the network: the held-out queries
        dict(name="mlp_infer", kind="mlp", op="infer", batch=65536),
        # training: eight Adam steps of the default batch from a checkpoint
        dict(name="mlp_train", kind="mlp", op="train", batch=2048, steps=8, phase=0),
        # the surface of the tank: the corner grid's voxel density ...
        dict(name="surface_voxel", kind="surface", op="voxel", layout="settled", n=2097152, boids=16384, spacing=0.0,
             bx=4.0, by=2.0, bz=2.0, cells="narrow", grid=0.5, radius=1.0),
        # ... and its triangles
        dict(name="surface_mc", kind="surface", op="mc", nx=182, ny=94, nz=94),
    ]


def _logu(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_scene(rng, n_max):
    n = _logu(rng, 1500, n_max)
    boids = min(max(1, _logu(rng, max(1, n // 1000), max(2, n // 64))), 16384)
    if n >= 60000 and rng.random() < 0.5:
        # the settled tank at the size that keeps the neighbours of the full one
        f = (n / 2097152.0) ** (1.0 / 3.0)
        return dict(layout="settled", n=n, boids=boids, spacing=0.0, bx=round(4.0 * f, 4), by=round(2.0 * f, 4),
                    bz=round(2.0 * f, 4), cells=rng.choice(["narrow", "half", "full_halfx"]))
    spacing = rng.choice([0.5 * H, 1.0 / 64.0, rng.uniform(0.3, 0.55) * H])
    side = math.ceil(n ** (1.0 / 3.0)) * spacing
    wide = round(max(1.0, 1.05 * side), 4)
    return dict(layout="dam", n=n, boids=boids, spacing=spacing, bx=round(max(1.0, 2.0 * side), 4), by=wide, bz=wide,
                cells=rng.choice(["half", "half", "full", "full_halfx", "narrow"]))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "batch", "forces", "forces", "mlp", "mlp", "surface"])
    if kind == "step":
        c = _draw_scene(rng, 2000000)
        diag = c["n"] < 300000 and rng.random() < 0.25
        c.update(kind="step", steps=max(1, min(10, 600000 // c["n"])), graph=rng.random() < 0.4,
                 host=rng.random() < 0.15, diag=diag, literal=rng.random() < 0.2, const_set=int(rng.random() < 0.15),
                 spheres=rng.randint(1, 6) if diag and rng.random() < 0.5 else 0)
        return c
    if kind == "batch":
        n_max = _logu(rng, 3000, 65536)
        return dict(kind="batch", scenes=_logu(rng, 2, 200), n_min=2048, n_max=n_max,
                    cells=rng.choice(["half", "full", "full_halfx"]), steps=rng.randint(1, 4), graph=True)
    if kind == "forces":
        c = _draw_scene(rng, 1000000)
        c.update(kind="forces", mode=rng.choice(["exact", "local", "surrogate", "gated"]), graph=rng.random() < 0.5)
        return c
    if kind == "mlp":
        op = rng.choice(["infer", "infer", "grad", "train", "train"])
        if op == "infer":
            return dict(kind="mlp", op="infer", batch=_logu(rng, 100, 65536))
        if op == "grad":
            return dict(kind="mlp", op="grad", batch=_logu(rng, 100, 8192))
        return dict(kind="mlp", op="train", batch=128 * _logu(rng, 1, 64), steps=rng.randint(1, 8),
                    phase=int(rng.random() < 0.25))
    if rng.random() < 0.5:
        c = _draw_scene(rng, 1000000)
        c.update(kind="surface", op="voxel", grid=rng.uniform(0.4, 0.9), radius=rng.uniform(0.7, 1.2))
        return c
    return dict(kind="surface", op="mc", **{k: _logu(rng, 20, 150) for k in ("nx", "ny", "nz")})


# ------------------------------------------------------------------ inputs

def _gen(seed, salt=0):
    return torch.Generator(device=DEV).manual_seed((int(seed) * 1000003 + salt) % (1 << 62))


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _pack(xyz):
    out = torch.zeros((xyz.shape[0], 4), dtype=torch.float32, device=DEV)
    out[:, :3] = xyz
    return out


def _box(case):
    return case["bx"], case["by"], case["bz"]


def _mean_neighbors(case):
    """Expected neighbours of a fluid particle of the layout."""
    ball = 4.0 / 3.0 * math.pi * float(H) ** 3
    if case["layout"] == "dam":
        return ball / case["spacing"] ** 3
    _, lo, hi = _settled_profile(case)
    return ball * 0.5 * (lo + hi) / RHO0 * _number_density(case)


def _number_density(case):
    """Particles per volume at the rest density: the tank's 40 % fill."""
    return case["n"] / (0.4 * case["bx"] * case["by"] * case["bz"])


def _settled_profile(case):
    """(depth of the settled fluid, density at its surface, at the floor) of
    an exponential profile holding the tank's 40 % fill in 25 % of its height."""
    by = case["by"]
    depth, a = 0.25 * by, 3.0 / by
    c = RHO0 * 0.4 * by * a * 2.0 / (1.0 - math.exp(-2.0 * a * depth))
    return depth, c * math.exp(-2.0 * a * depth), c


def _params(case):
    cell, cell_x = CELLS[case["cells"]]
    over = dict(box_max=_box(case), cell_size=cell * H, cell_size_x=cell_x * H,
                const_set=case.get("const_set", 0), coupling_mode=int(case.get("literal", False)))
    if case["layout"] == "dam":
        over["mass"] = RHO0 * case["spacing"] ** 3
    else:
        over["mass"] = RHO0 / _number_density(case)
    return scenes.default_params(**over)


def _lattice(g, idx, width, spacing, origin):
    """Points idx of a lattice width x * x width (x, z fastest last), jittered
    by a tenth of the spacing; idx, width and origin per point."""
    w = width
    i, k, j = idx % w, (idx // w) % w, idx // (w * w)
    base = torch.stack([i, j, k], 1).double() + 0.5
    return origin + (base + 0.2 * (_rand(g, idx.shape[0], 3) - 0.5)) * spacing


def _flow(g, pos, box, speed, noise):
    """A smooth flow of the tank (one sloshing mode per axis) with noise."""
    x = pos / torch.tensor(box, device=DEV, dtype=torch.float64)
    ph = _rand(g, 3)
    u = torch.stack([torch.sin(math.pi * x[:, 0]) * torch.cos(math.pi * x[:, 1] + ph[0]),
                     -0.6 * torch.cos(math.pi * x[:, 0]) * torch.sin(math.pi * x[:, 1]),
                     0.3 * torch.sin(2.0 * math.pi * x[:, 2] + ph[1]) * torch.cos(math.pi * x[:, 0] + ph[2])], 1)
    return speed * u + noise * _randn(g, pos.shape[0], 3)


def _headings(g, n):
    d = _randn(g, n, 3)
    return d / d.norm(dim=1, keepdim=True)


def _fluid(case, seed):
    n, box = case["n"], _box(case)
    g = _gen(seed, 1)
    i = torch.arange(n, device=DEV)
    if case["layout"] == "dam":
        w = math.ceil(n ** (1.0 / 3.0) - 1e-9)
        pos = _lattice(g, i, w, case["spacing"], 0.0)
        vel = _flow(g, pos, box, 0.6, 0.02)
    else:
        # a low-discrepancy sequence (even, without lattice directions), its
        # y mapped to the exponential profile
        phi = 1.2207440846057596
        u = torch.stack([(i.double() * (1.0 / phi ** (a + 1)) + _rand(g, 1)) % 1.0 for a in range(3)], 1)
        u = (u + 0.3 * n ** (-1.0 / 3.0) * (_rand(g, n, 3) - 0.5)).clamp(1e-5, 1.0 - 1e-5)
        depth, _, _ = _settled_profile(case)
        a2 = 6.0 / box[1]
        y = -torch.log1p(-u[:, 1] * (1.0 - math.exp(-a2 * depth))) / a2
        # 2 mm off the side walls: a pass moves the fluid by less, so that only
        # the floor reflects (at a far wall one rounding of x decides which way
        # a particle goes, in any precision)
        pos = torch.stack([0.002 + u[:, 0] * (box[0] - 0.004), y, 0.002 + u[:, 2] * (box[2] - 0.004)], 1)
        vel = _flow(g, pos, box, 0.8, 0.05)
    return _pack(pos), _pack(vel)


def _boids(case, seed):
    n, box = case["boids"], torch.tensor(_box(case), device=DEV, dtype=torch.float64)
    g = _gen(seed, 2)
    if case["layout"] == "dam":
        pos = 1e-3 + _rand(g, n, 3) * (box - 2e-3)
        return _pack(pos), _pack(_headings(g, n))
    # eight schools released in the lower 40 %
    school = torch.arange(n, device=DEV) % 8
    span = box * torch.tensor([1.0, 0.4, 1.0], device=DEV, dtype=torch.float64)
    centre = 0.1 + _rand(g, 8, 3) * (span - 0.2).clamp_min(0.0)
    pos = centre[school] + _headings(g, n) * 0.1 * _rand(g, n, 1) ** (1.0 / 3.0)
    head = _headings(g, 8)[school] + 0.1 * _headings(g, n)
    return _pack(pos), _pack(0.5 * head / head.norm(dim=1, keepdim=True))


def _spheres(case, seed):
    k = case.get("spheres", 0)
    if not k:
        return None
    g = _gen(seed, 3)
    c = 0.2 + 0.6 * _rand(g, k, 3) * torch.tensor(_box(case), device=DEV, dtype=torch.float64)
    return torch.cat([c, 0.1 + 0.15 * _rand(g, k, 1)], 1).float().cpu().numpy()


def _batch(case, seed):
    """Per-scene counts and the concatenated state of the batched tanks."""
    S = case["scenes"]
    g = _gen(seed, 4)
    r = np.random.default_rng(20231118 + 977 * S + case["n_max"])
    # the sizes belong to the case (a handle is laid out for them once)
    nf = np.exp(r.uniform(math.log(case["n_min"]), math.log(case["n_max"]), S)).astype(np.int64)
    nb = r.integers(8, 257, S)
    cell, cell_x = CELLS[case["cells"]]
    s = 0.5 * H
    p = scenes.default_params(mass=RHO0 * s ** 3, cell_size=cell * H, cell_size_x=cell_x * H)
    w = np.minimum(np.ceil(nf ** (1.0 / 3.0) - 1e-9), math.floor(0.92 / s)).astype(np.int64)
    cnt = torch.from_numpy(nf).to(DEV)
    first = torch.cumsum(cnt, 0) - cnt
    scene = torch.repeat_interleave(torch.arange(S, device=DEV), cnt)
    idx = torch.arange(int(nf.sum()), device=DEV) - first[scene]
    pos = _lattice(g, idx, torch.from_numpy(w).to(DEV)[scene], s, 0.0)
    pos[:, 1].clamp_(max=0.999)
    vel = _flow(g, pos, (1.0, 1.0, 1.0), 0.6, 0.02)
    B = int(nb.sum())
    bpos = 1e-3 + 0.998 * _rand(g, B, 3)
    bscene = torch.repeat_interleave(torch.arange(S, device=DEV), torch.from_numpy(nb).to(DEV))
    return p, nf.tolist(), nb.tolist(), (_pack(pos), _pack(vel), _pack(bpos), _pack(_headings(g, B))), scene, bscene


def _net(seed):
    """Packed FP32 parameters of the network as a trained one has them in
    size (uniform in +-1 / sqrt(fan in), small biases)."""
    g = _gen(seed, 5)
    parts = []
    for n_in, n_out in LAYERS:
        parts += [(2.0 * _rand(g, n_out * n_in) - 1.0) / math.sqrt(n_in), 0.1 * (2.0 * _rand(g, n_out) - 1.0)]
    return torch.cat(parts).float()


def _rows(seed, n, salt):
    """Network inputs as the features come: per stencil cell a count around
    one (or an empty cell) and a mean velocity, then the boid's own columns."""
    g = _gen(seed, salt)
    x = 0.4 * _randn(g, n, 272)
    full = (_rand(g, n, 64) > 0.3).double()
    x[:, 0:256:4] = full * (1.0 + 0.2 * _randn(g, n, 64))
    for a in range(1, 4):
        x[:, a:256:4] *= full
    x[:, 262:264] = 1.0 + 0.3 * _randn(g, n, 2)
    x[:, 270:] = 0.0
    return x.to(torch.bfloat16)


def _targets(seed, n, salt):
    g = _gen(seed, salt)
    t = torch.zeros((n, 4), device=DEV)
    t[:, :3] = _randn(g, n, 3)
    t[:, 3] = -1.0 + 0.5 * _randn(g, n)
    return t


def _moments(seed):
    """Adam moments of a run under way (step 1000)."""
    g = _gen(seed, 6)
    n = sum(a * b + b for a, b in LAYERS)
    m2 = (1e-6 * (0.2 + _rand(g, n))).float()
    return (2e-4 * _randn(g, n)).float(), m2


def _field(case, seed):
    """Corner values of a wavy free surface with drops above it, as the
    voxel density gives them: -r .. R around the surface, R in the air."""
    g = _gen(seed, 7)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    s = 0.5 * H
    x, y, z = (torch.arange(k, device=DEV, dtype=torch.float64) * s for k in (nx, ny, nz))
    a = 2.0 * math.pi * _rand(g, 4)
    lx, lz = nx * s, nz * s
    level = 0.35 * ny * s * (1.0 + 0.3 * torch.sin(2 * math.pi * x[None, :] / lx * 2 + a[0]) *
                             torch.cos(2 * math.pi * z[:, None] / lz + a[1]) +
                             0.06 * torch.sin(2 * math.pi * x[None, :] / lx * 17 + a[2]) *
                             torch.cos(2 * math.pi * z[:, None] / lz * 9 + a[3]))
    phi = y[None, :, None] - level[:, None, :]
    for c in _rand(g, 12, 4).cpu().tolist():
        d = ((x[None, None, :] - c[0] * lx) ** 2 + (y[None, :, None] - (0.5 + 0.4 * c[1]) * ny * s) ** 2 +
             (z[:, None, None] - c[2] * lz) ** 2).sqrt() - (2.0 + 4.0 * c[3]) * s
        phi = torch.minimum(phi, d)
    phi = phi + 0.02 * s * _randn(g, nz, ny, nx)
    return phi.clamp(-0.25 * float(H), float(H)).float().reshape(-1).contiguous()


# ------------------------------------------------------------------ passes

def prepare(case, seed):
    kind = case["kind"]
    st = {"case": dict(case)}
    if kind == "batch":
        p, nf, nb, state, _, _ = _batch(case, seed)
        st["scene"] = Scene([p] * case["scenes"], nf, nb, device=DEV)
        st["state"] = state
        st["stream"] = torch.cuda.Stream()
    elif kind == "mlp":
        B, op = case["batch"], case["op"]
        st["mlp"] = Mlp(B, device=DEV)
        st["mlp"].set_params(_net(seed))
        if op == "infer":
            st["x"] = _rows(seed, B, 10)
        elif op == "grad":
            st["x"], st["dy"] = _rows(seed, B, 10), _grad_rows(seed, B)
        else:
            st["x"] = [_rows(seed, B, 10 + k) for k in range(case["steps"])]
            st["t"] = [_targets(seed, B, 30 + k) for k in range(case["steps"])]
            m1, m2 = _moments(seed)
            st["ckpt"] = {"params": _net(seed), "adam_m1": m1, "adam_m2": m2, "adam_step": torch.tensor(1000)}
    elif kind == "surface" and case["op"] == "mc":
        st["phi"] = _field(case, seed)
        dims = (case["nx"], case["ny"], case["nz"])
        # a real-time loop keeps its triangle buffer and workspace
        st["dims"], st["cap"] = dims, 4 * dims[0] * dims[2] + 20000
        st["ws_bytes"] = sph_mc_workspace_size(dims)
        st["ws"] = torch.empty(st["ws_bytes"], dtype=torch.uint8, device=DEV)
        st["tris"] = torch.zeros((st["cap"], 3, 3), dtype=torch.float32, device=DEV)
        st["total"] = torch.zeros(1, dtype=torch.int32, device=DEV)
    else:
        s = Scene(_params(case), case["n"], case["boids"], device=DEV, diagnostics=bool(case.get("diag")))
        st["scene"] = s
        st["state"] = (*_fluid(case, seed), *_boids(case, seed))
        if case.get("host"):
            st["state"] = tuple(t.cpu().pin_memory() for t in st["state"])
            st["out"] = [torch.empty_like(t).pin_memory() for t in st["state"]]
        sph = _spheres(case, seed)
        if sph is not None:
            s.set_obstacles(spheres=sph)
        if case.get("graph"):
            st["stream"] = torch.cuda.Stream()
        if kind == "forces":
            if case["mode"] in ("surrogate", "gated"):
                mlp = Mlp(max(case["boids"], 128), device=DEV)
                mlp.set_params(_net(seed))
                lo = torch.full((272,), -1e30)
                hi = torch.full((272,), 1e30)
                lo[256:259], hi[256:259] = -GATE_SPEED, GATE_SPEED
                s.set_surrogate(mlp, F_SCALE, 1e30, (lo, hi))
            if case["graph"]:
                s.set_state(*st["state"])  # the state whose forces are asked for
    torch.cuda.synchronize()
    return st


def _grad_rows(seed, n):
    return (_randn(_gen(seed, 8), n, 16) / n).float()


def _on_stream(st, body):
    """Run body on the program's own stream (graphs need one), ordered with
    the caller's."""
    if "stream" not in st:
        return body()
    cur = torch.cuda.current_stream()
    st["stream"].wait_stream(cur)
    with torch.cuda.stream(st["stream"]):
        out = body()
    cur.wait_stream(st["stream"])
    for t in out.values():
        if t.is_cuda:
            t.record_stream(cur)
    return out


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind in ("step", "batch"):
        return _on_stream(st, lambda: _run_steps(st, case))
    if kind == "forces":
        return _on_stream(st, lambda: _run_forces(st, case))
    if kind == "mlp":
        return _run_mlp(st, case)
    if case["op"] == "voxel":
        s = st["scene"]
        s.set_state(*st["state"])
        phi, cnt, _, _ = s.voxel_density(case["grid"] * H, case["radius"] * H, 0.25 * H)
        return {"phi": phi, "count": cnt}
    sph_marching_cubes(st["phi"].data_ptr(), st["dims"], (0.0, 0.0, 0.0), 0.5 * H, 0.0, st["ws"].data_ptr(),
                       st["ws_bytes"], st["tris"].data_ptr(), st["cap"], st["total"].data_ptr(),
                       torch.cuda.current_stream().cuda_stream)
    return {"tris": st["tris"], "total": st["total"]}


def _run_steps(st, case):
    s = st["scene"]
    if case.get("host"):
        s.set_state_host(*st["state"])
    else:
        s.set_state(*st["state"])
    if case["graph"]:
        s.graph_step(case["steps"])
    else:
        s.step(case["steps"])
    out = {"rho": s.field("rho"), "nbr_count": s.field("nbr_count"), "fb": s.field("fb")}
    if case.get("diag"):
        out.update(acc=s.field("acc"), touched=s.field("touched"), influence=s.field("influence"), stats=s.stats())
    if case.get("host"):
        s.get_state_host(st["out"])
        state = st["out"]
    else:
        state = s.get_state()
    out.update(zip(("fluid_pos", "fluid_vel", "boid_pos", "boid_vel"), state))
    return out


def _run_forces(st, case):
    s = st["scene"]
    if case["graph"]:
        return {"fb": s.graph_boid_forces(MODES[case["mode"]])}
    s.set_state(*st["state"])
    return {"fb": s.boid_forces(MODES[case["mode"]])}


def _run_mlp(st, case):
    m = st["mlp"]
    if case["op"] == "infer":
        return {"y": m.forward(st["x"])}
    if case["op"] == "grad":
        return {"grads": m.gradients(st["x"], st["dy"])}
    m.load_state_dict(st["ckpt"])
    losses = [m.train_step(x, t, 1e-3, phase=case["phase"]).clone() for x, t in zip(st["x"], st["t"])]
    g, m1, m2, _ = m.optimizer_state()
    # phase 1 trains the error head alone: the other gradients are left over
    # from whatever ran before and belong to no output
    out = {"loss": torch.cat(losses), "params": m.get_params(), "adam_m1": m1, "adam_m2": m2}
    if case["phase"] == 0:
        out["grads"] = g
    return out


# -------------------------------------------------------------------- work

def work(case):
    kind = case["kind"]
    if kind == "step":
        n, b = case["n"], case["boids"]
        nb = _mean_neighbors(case)
        per = 32 + 32 + 4 + 4 + (36 if case["diag"] else 0)
        # per neighbour: distance (8), density (4), force (30)
        return {"bytes": (n + b) * per + b * 80, "flops": case["steps"] * n * nb * 42}
    if kind == "batch":
        # mean of the log-uniform sizes
        lo, hi = case["n_min"], case["n_max"]
        n = case["scenes"] * (hi - lo) / math.log(hi / lo)
        nb = 4.0 / 3.0 * math.pi * 8.0
        return {"bytes": n * 72, "flops": case["steps"] * n * nb * 42}
    if kind == "forces":
        n, b = case["n"], case["boids"]
        nb = _mean_neighbors(case)
        # in: the particles' positions and velocities; out: the forces
        f = b * nb * 30
        if case["mode"] in ("exact", "local"):
            f += min(n, b * nb) * nb * 12
        else:
            f += b * 2 * sum(i * o for i, o in LAYERS)
        return {"bytes": n * 32 + b * 48, "flops": f}
    if kind == "mlp":
        B = case["batch"]
        mac = sum(i * o for i, o in LAYERS)
        npar = sum(i * o + o for i, o in LAYERS)
        if case["op"] == "infer":
            return {"bytes": B * (544 + 64) + 4 * npar, "flops": 2 * B * mac}
        if case["op"] == "grad":
            return {"bytes": B * (544 + 64) + 8 * npar, "flops": 2 * B * (3 * mac - 272 * 256)}
        per = 2 * B * (3 * mac - 272 * 256) if case["phase"] == 0 else 2 * B * (mac + 256 * 16)
        return {"bytes": case["steps"] * B * (544 + 16) + 28 * npar, "flops": case["steps"] * per}
    if case["op"] == "voxel":
        n = case["n"]
        s = case["grid"] * float(H)
        corners = 1.0
        for e in _box(case):
            corners *= e / s + 7
        rel = case["radius"] ** 3
        mean = _mean_neighbors(case) * rel
        # corners within the fluid's volume see the neighbours
        wet = n / max(mean, 1.0) * 4.0 / 3.0 * math.pi * (case["radius"] * float(H)) ** 3 / s ** 3
        return {"bytes": n * 16 + corners * 8, "flops": wet * mean * 20}
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    tri = 2.4 * nx * nz
    return {"bytes": 4.0 * nx * ny * nz + 36 * tri, "flops": 60.0 * tri}


# ------------------------------------------------------- values in 64 bits

def _pairs(q, p, radius, qs=None, ps=None, budget=4_000_000):
    """Index pairs (i, j) with |q_i - p_j| < radius, in chunks: points p
    binned in cells of the radius, each query's nine rows of three cells
    expanded.  qs, ps: scene of every point (pairs stay within a scene)."""
    if not len(q) or not len(p):
        return
    lo = torch.minimum(q.min(0).values, p.min(0).values) - 1e-9
    cq, cp = ((q - lo) / radius).floor().long() + 1, ((p - lo) / radius).floor().long() + 1
    dim = torch.maximum(cq.max(0).values, cp.max(0).values) + 2
    nx, ny, nz = (int(v) for v in dim)
    sq = qs if qs is not None else torch.zeros(len(q), dtype=torch.long, device=q.device)
    sp = ps if ps is not None else torch.zeros(len(p), dtype=torch.long, device=p.device)
    key = ((sp * nz + cp[:, 2]) * ny + cp[:, 1]) * nx + cp[:, 0]
    key, order = key.sort()
    qkey = ((sq * nz + cq[:, 2]) * ny + cq[:, 1]) * nx + cq[:, 0]
    rows = torch.tensor([(dz * ny + dy) * nx for dz in (-1, 0, 1) for dy in (-1, 0, 1)], device=q.device)
    first = torch.searchsorted(key, (qkey[:, None] + rows - 1).reshape(-1)).view(-1, 9)
    last = torch.searchsorted(key, (qkey[:, None] + rows + 1).reshape(-1), right=True).view(-1, 9)
    total = torch.cumsum((last - first).sum(1), 0).cpu()
    a, n = 0, len(q)
    while a < n:
        base = int(total[a - 1]) if a else 0
        b = int(torch.searchsorted(total, base + budget, right=True))
        b = min(max(b, a + 1), n)
        cnt = (last[a:b] - first[a:b]).reshape(-1)
        off = torch.cumsum(cnt, 0) - cnt
        src = torch.repeat_interleave(torch.arange(len(cnt), device=q.device), cnt)
        j = order[first[a:b].reshape(-1)[src] + torch.arange(len(src), device=q.device) - off[src]]
        i = a + src // 9
        near = ((q[i] - p[j]) ** 2).sum(1) < radius * radius
        yield i[near], j[near]
        a = b


def _constants(p):
    h = p["h"]
    if p["const_set"] == 1:
        return 30.0 / (math.pi * h ** 4), 40.0 / (math.pi * h ** 4)
    return (45.0 / (math.pi * h ** 5),) * 2


def _density64(p, x, att, scene=None, want=None):
    """Densities of the particles x (of those in `want`, an index list) and
    their neighbour counts; pairs of attached particles are left out."""
    h = p["h"]
    c6 = p["mass"] * 315.0 / (64.0 * math.pi * h ** 9)
    idx = want if want is not None else torch.arange(len(x), device=x.device)
    s = torch.full((len(idx),), h ** 6, dtype=torch.float64, device=x.device)
    cnt = torch.zeros(len(idx), dtype=torch.long, device=x.device)
    for i, j in _pairs(x[idx], x, h, None if scene is None else scene[idx], scene):
        gi = idx[i]
        ok = (gi != j) & ~(att[gi] & att[j])
        i, j, gi = i[ok], j[ok], gi[ok]
        t = h * h - ((x[gi] - x[j]) ** 2).sum(1)
        s.index_add_(0, i, t ** 3)
        cnt.index_add_(0, i, torch.ones_like(i))
    return c6 * s, cnt


def _accel64(p, x, v, rho, att, scene=None, want=None):
    """(1 / rho_i) sum_j f_ij without gravity, and the part from attached j."""
    h = p["h"]
    cp, cv = _constants(p)
    idx = want if want is not None else torch.arange(len(x), device=x.device)
    acc = torch.zeros((len(idx), 3), dtype=torch.float64, device=x.device)
    infl = torch.zeros_like(acc)
    for i, j in _pairs(x[idx], x, h, None if scene is None else scene[idx], scene):
        gi = idx[i]
        d = x[gi] - x[j]
        r = d.norm(dim=1)
        ok = (gi != j) & (r > 0) & ~(att[gi] & att[j])
        i, j, gi, d, r = i[ok], j[ok], gi[ok], d[ok], r[ok]
        w = 1.0 - r / h
        pres = cp * 0.5 * p["k"] * (rho[gi] + rho[j] - 2.0 * p["rho0"]) * w * w * h / r
        f = (p["mass"] / rho[j])[:, None] * (pres[:, None] * d - (cv * p["mu"] * w)[:, None] * (v[gi] - v[j]))
        acc.index_add_(0, i, f)
        a = att[j]
        infl.index_add_(0, i[a], f[a])
    return acc / rho[idx][:, None], infl / rho[idx][:, None]


def _obstacle64(p, spheres, pb):
    """w_obst times the weighted mean normal of the obstacle cells in sight."""
    d = float(p["boid_cell_size"])
    mn, mx = (torch.tensor(p[k], dtype=torch.float64, device=DEV) for k in ("box_min", "box_max"))
    dim = torch.ceil((mx - mn) / d).long().clamp_min(1)
    c = torch.stack(torch.meshgrid(*[torch.arange(int(k), device=DEV) for k in dim], indexing="ij"), -1).reshape(-1, 3)
    c = (c.double() + 0.5) * d + mn
    s = torch.from_numpy(spheres).to(DEV).double()
    u = c[:, None] - s[None, :, :3]
    r = u.norm(dim=2)
    on = ((r - s[None, :, 3]).abs() <= 0.866025403784 * d) & (r > 0)
    cnt = on.sum(1)
    normal = (torch.where(on[..., None], u / r.clamp_min(1e-300)[..., None], torch.zeros_like(u)).sum(1) /
              cnt.clamp_min(1)[:, None])
    c, normal = c[cnt > 0], normal[cnt > 0]
    r = (pb[:, None] - c[None]).norm(dim=2)
    w = torch.where(r < p["r_sep"], 2.0, 1.0) * (r < p["r_vis"])
    n = (r < p["r_vis"]).sum(1)
    return 0.05 * (w[..., None] * normal[None]).sum(1) / n.clamp_min(1)[:, None].double()


def _step64(p, fx, fv, bx, bv, va, fscene=None, bscene=None, spheres=None):
    """One step in 64 bits: new (fx, fv, bx, bv, va) and the step's fields."""
    nb = len(bx)
    x, v = torch.cat([bx, fx]), torch.cat([va, fv])
    att = torch.arange(len(x), device=DEV) < nb
    scene = None if fscene is None else torch.cat([bscene, fscene])
    rho, cnt = _density64(p, x, att, scene)
    acc, infl = _accel64(p, x, v, rho, att, scene)
    grav = torch.tensor([p["gx"], p["gy"], p["gz"]], dtype=torch.float64, device=DEV)
    fb = acc[:nb].clone()
    # boid rules on the snapshot
    cl, vs, ps = (torch.zeros_like(bx) for _ in range(3))
    nv = torch.zeros(nb, dtype=torch.float64, device=DEV)
    for i, j in _pairs(bx, bx, p["r_vis"], bscene, bscene):
        ok = i != j
        i, j = i[ok], j[ok]
        d = bx[i] - bx[j]
        w = (1.0 - d.norm(dim=1) / p["r_sep"]).clamp(0.0, 1.0)
        cl.index_add_(0, i, d * w[:, None])
        vs.index_add_(0, i, bv[j])
        ps.index_add_(0, i, -d)
        nv.index_add_(0, i, torch.ones_like(w))
    u = bv + p["w_sep"] * cl
    seen = (nv > 0)[:, None]
    nn = nv.clamp_min(1)[:, None]
    u = torch.where(seen, u + p["w_align"] * (vs / nn - u), u)
    u = torch.where(seen, u + p["w_coh"] * ps / nn, u)
    if p["coupling_mode"] == 1:
        va = va + p["dt"] * (fb + grav)
        u = u + p["sph_factor"] * va
    else:
        u = u + p["sph_factor"] * p["dt"] * fb
    if spheres is not None:
        u = u + _obstacle64(p, spheres, bx)
    lo, hi = (torch.tensor(p[k], dtype=torch.float64, device=DEV) for k in ("box_min", "box_max"))
    u = u + p["edge_turn"] * ((bx < lo).double() - (bx > hi).double())
    sp = u.norm(dim=1, keepdim=True)
    u = u * torch.where(sp > p["v_max"], p["v_max"] / sp,
                        torch.where((sp > 0) & (sp < p["v_min"]), p["v_min"] / sp.clamp_min(1e-300),
                                    torch.ones_like(sp)))
    bx = bx + p["dt"] * u
    if p["coupling_mode"] == 0:
        va = u
    # integration and walls
    facc = acc[nb:] + grav
    fv = fv + p["dt"] * facc
    fx = fx + p["dt"] * fv
    below, above = fx < lo, fx > hi
    fx = torch.where(below, 2 * lo - fx, torch.where(above, 2 * hi - fx, fx))
    fv = torch.where(below | above, -p["wall_restitution"] * fv, fv)
    fx = torch.minimum(torch.maximum(fx, lo), hi)
    infl[:nb] = 0.0
    return (fx, fv, bx, u, va), dict(rho=rho, cnt=cnt, fb=fb, acc=torch.cat([fb, facc]), infl=infl)


def _pad4(t):
    return torch.cat([t, torch.zeros_like(t[:, :1])], 1)


def _stats64(p, x, state, f, nb):
    fv = state[1]
    c = []
    for a in range(3):
        s = p["cell_size_x"] if a == 0 and p["cell_size_x"] > 0 else p["cell_size"]
        dim = max(1, math.ceil((p["box_max"][a] - p["box_min"][a]) / s))
        c.append(((x[:, a] - p["box_min"][a]) / s).floor().clamp(0, dim - 1).long())
    _, occ = torch.unique((c[2] * 100000 + c[1]) * 100000 + c[0], return_counts=True)
    n, rho = f["cnt"][nb:].double(), f["rho"][nb:]
    v2 = (fv * fv).sum(1)
    m = p["mass"]
    return torch.stack([torch.tensor(float(len(fv)), dtype=torch.float64, device=DEV), n.mean(), n.max(),
                        occ.max().double(), *(m * fv.sum(0)), 0.5 * m * v2.sum(), rho.min(), rho.max(), rho.mean(),
                        v2.max().sqrt()])[None]


def _forward64(P, x):
    """The network with its weights in BF16, everything else in 64 bits."""
    off, a, keep = 0, x.double(), []
    for l, (n_in, n_out) in enumerate(LAYERS):
        W = P[off:off + n_in * n_out].view(n_out, n_in).to(torch.bfloat16).double()
        b = P[off + n_in * n_out:off + n_in * n_out + n_out].double()
        off += n_in * n_out + n_out
        z = a @ W.T + b
        keep.append((a, W, z))
        a = z if l == 3 else 0.5 * z * (1.0 + torch.erf(z / math.sqrt(2.0)))
    return a, keep


def _backward64(keep, dy, head_only=False):
    grads, d = [], dy
    for l in (3, 2, 1, 0):
        a, W, z = keep[l]
        if l < 3:
            phi = torch.exp(-0.5 * z * z) / math.sqrt(2.0 * math.pi)
            d = d * (0.5 * (1.0 + torch.erf(z / math.sqrt(2.0))) + z * phi)
        if head_only and l < 3:
            grads.append(torch.zeros(W.numel() + W.shape[0], dtype=torch.float64, device=DEV))
        else:
            grads.append(torch.cat([(d.T @ a).reshape(-1), d.sum(0)]))
        d = d @ W
    return torch.cat(grads[::-1])


def _train64(case, seed):
    B, phase = case["batch"], case["phase"]
    P = _net(seed).double()
    m1, m2 = (t.double() for t in _moments(seed))
    sizes = [i * o + o for i, o in LAYERS]
    w4 = sum(sizes[:3])
    head = torch.zeros(len(P), dtype=torch.bool, device=DEV)
    head[w4 + 3 * 256:w4 + 4 * 256] = True
    head[w4 + 16 * 256 + 3] = True
    upd = head if phase == 1 else ~head
    losses = []
    for k in range(case["steps"]):
        x, t = _rows(seed, B, 10 + k), _targets(seed, B, 30 + k).double()
        y, keep = _forward64(P.float(), x)
        dy = torch.zeros_like(y)
        cols = slice(3, 4) if phase == 1 else slice(0, 3)
        d = y[:, cols] - t[:, cols]
        dy[:, cols] = d / B
        losses.append(0.5 * (d * d).sum() / B)
        g = _backward64(keep, dy, head_only=phase == 1)
        step = 1001 + k
        a = torch.where(upd, 0.9 * m1 + 0.1 * g, m1)
        b = torch.where(upd, 0.999 * m2 + 0.001 * g * g, m2)
        m1, m2 = a, b
        new = P - 1e-3 * (m1 / (1 - 0.9 ** step)) / ((m2 / (1 - 0.999 ** step)).sqrt() + 1e-8)
        P = torch.where(upd, new, P)
    out = {"loss": torch.stack(losses), "params": P, "adam_m1": m1, "adam_m2": m2}
    if phase == 0:
        out["grads"] = g
    return out


def _features64(p, fx, fv, bx, bv):
    h, m = p["h"], p["mass"]
    lo = torch.tensor(p["box_min"], dtype=torch.float64, device=DEV)
    t = (bx - lo) / h
    c0 = (t - 1.5).floor()
    x = torch.zeros((len(bx), 272), dtype=torch.float64, device=DEV)
    # stencil cells: sums per feature cell, then gathered
    fc = ((fx - lo) / h).floor().long() + 4
    hi = torch.tensor(p["box_max"], dtype=torch.float64, device=DEV)
    dim = [int(v) for v in (((hi - lo) / h).ceil().long() + 9)]
    grid = torch.zeros((dim[0] * dim[1] * dim[2], 4), dtype=torch.float64, device=DEV)
    grid.index_add_(0, (fc[:, 2] * dim[1] + fc[:, 1]) * dim[0] + fc[:, 0],
                    torch.cat([torch.ones_like(fx[:, :1]), fv], 1))
    for q in range(64):
        o = torch.tensor([q & 3, (q >> 2) & 3, q >> 4], device=DEV)
        c = c0.long() + 4 + o
        inside = ((c >= 0) & (c < torch.tensor(dim, device=DEV))).all(1)
        c = c.clamp_min(0)
        k = ((c[:, 2] * dim[1] + c[:, 1]) * dim[0] + c[:, 0]).clamp_max(len(grid) - 1)
        s = grid[k] * inside[:, None]
        x[:, 4 * q] = s[:, 0] * m / (h ** 3 * p["rho0"])
        x[:, 4 * q + 1:4 * q + 4] = s[:, 1:] / s[:, :1].clamp_min(1)
    x[:, 256:259] = bv
    x[:, 259:262] = t - c0 - 2.0
    x[:, 262] = h ** 6
    for i, j in _pairs(bx, fx, h):
        d = bx[i] - fx[j]
        r = d.norm(dim=1)
        w = 1.0 - r / h
        x[:, 262].index_add_(0, i, (h * h - r * r) ** 3)
        x[:, 263].index_add_(0, i, w)
        x[:, 264:267] = x[:, 264:267].index_add(0, i, w[:, None] * (fv[j] - bv[i]))
        x[:, 267:270] = x[:, 267:270].index_add(0, i, (w * w / r.clamp_min(1e-300))[:, None] * d)
    x[:, 262] *= m * 315.0 / (64.0 * math.pi * h ** 9) / p["rho0"]
    x[:, 263:270] *= m / (p["rho0"] * h ** 3)
    return x


def _forces64(case, seed):
    p = _params(case)
    fx, fv, bx, bv = (t[:, :3].double() for t in (*_fluid(case, seed), *_boids(case, seed)))
    nb = len(bx)
    out = torch.zeros((nb, 4), dtype=torch.float64, device=DEV)
    flag = torch.ones(nb, dtype=torch.bool, device=DEV)
    if case["mode"] in ("surrogate", "gated"):
        y, _ = _forward64(_net(seed), _features64(p, fx, fv, bx, bv))
        out[:, :3] = y[:, :3] * F_SCALE
        flag = ((bv.to(torch.bfloat16).double().abs() > float(np.float32(GATE_SPEED))).any(1)
                if case["mode"] == "gated" else ~flag)
        out[:, 3] = 0.0
    if flag.any():
        x, v = torch.cat([bx, fx]), torch.cat([bv, fv])
        att = torch.arange(len(x), device=DEV) < nb
        who = torch.nonzero(flag).view(-1)
        need = torch.zeros(len(x), dtype=torch.bool, device=DEV)
        need[who] = True
        for _, j in _pairs(x[who], x, p["h"]):
            need[j] = True
        idx = torch.nonzero(need).view(-1)
        rho = torch.full((len(x),), p["rho0"], dtype=torch.float64, device=DEV)
        rho[idx] = _density64(p, x, att, want=idx)[0]
        out[who, :3] = _accel64(p, x, v, rho, att, want=who)[0]
        if case["mode"] == "gated":
            out[who, 3] = 1.0
    return {"fb": out}


def _voxel64(case, seed):
    p = _params(case)
    fx = _fluid(case, seed)[0][:, :3].double()
    s, R, r = (np.float32(k) for k in (case["grid"] * H, case["radius"] * H, 0.25 * H))
    pad = math.ceil(np.float32(R / s)) + 1
    axes = []
    for a in range(3):
        ext = np.float32(p["box_max"][a]) - np.float32(p["box_min"][a])
        n = int(math.floor(float(ext) / float(s)) + 1 + 2 * pad)
        o = np.float32(p["box_min"][a]) - np.float32(pad) * s
        # a corner is at fl(origin + fl(i spacing)): its place is float32 by definition
        axes.append(torch.from_numpy((np.arange(n, dtype=np.float32) * s + o).astype(np.float64)).to(DEV))
    z, y, x = torch.meshgrid(axes[2], axes[1], axes[0], indexing="ij")
    q = torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1)
    ks = torch.zeros(len(q), dtype=torch.float64, device=DEV)
    kd = torch.zeros((len(q), 3), dtype=torch.float64, device=DEV)
    for i, j in _pairs(q, fx, float(R)):
        d = fx[j] - q[i]
        k = (1.0 - (d * d).sum(1) / float(R) ** 2) ** 3
        ks.index_add_(0, i, k)
        kd.index_add_(0, i, k[:, None] * d)
    phi = torch.where(ks > 0, kd.norm(dim=1) / ks.clamp_min(1e-300) - float(r), torch.full_like(ks, float(R)))
    return {"phi": phi, "count": None}


def exact(case, seed):
    """What run returns, in 64 bits; whole numbers, and the triangles (their
    order and number belong to the corner values' signs), have none."""
    kind = case["kind"]
    if kind == "mlp":
        if case["op"] == "infer":
            return {"y": _forward64(_net(seed), _rows(seed, case["batch"], 10))[0]}
        if case["op"] == "grad":
            _, keep = _forward64(_net(seed), _rows(seed, case["batch"], 10))
            return {"grads": _backward64(keep, _grad_rows(seed, case["batch"]).double())}
        return _train64(case, seed)
    if kind == "surface":
        return _voxel64(case, seed) if case["op"] == "voxel" else None
    if kind == "forces":
        return _forces64(case, seed)
    fscene = bscene = spheres = None
    if kind == "batch":
        p, _, _, inputs, fscene, bscene = _batch(case, seed)
    else:
        p = _params(case)
        inputs = (*_fluid(case, seed), *_boids(case, seed))
        spheres = _spheres(case, seed)
    state = tuple(t[:, :3].double() for t in inputs)
    state = (*state, state[3])  # the attached particles start with their boids' velocities
    for _ in range(case["steps"]):
        before = torch.cat([state[2], state[0]])
        state, f = _step64(p, *state, fscene, bscene, spheres)
    out = {"rho": f["rho"], "nbr_count": None, "fb": _pad4(f["fb"])}
    if case.get("diag"):
        out.update(acc=_pad4(f["acc"]), touched=None, influence=_pad4(f["infl"]),
                   stats=_stats64(p, before, state, f, len(state[2])))
    out.update(zip(("fluid_pos", "fluid_vel", "boid_pos", "boid_vel"), (_pad4(t) for t in state[:4])))
    if case.get("host"):
        for k in ("fluid_pos", "fluid_vel", "boid_pos", "boid_vel"):
            out[k] = out[k].cpu()
    return out
