"""The framework's work, as its users have it done: one pass of each case is a
whole call on fields that the caller holds: set the state, take the steps, get
the state back (or, for the gradient cases, a differentiable rollout and its
backward pass). Meshes and handles are built once, in ``prepare``, as a
program that runs a model again and again keeps them.

A case is a dict of plain values:
  family     which flow: "stoker" (1D dam break), "drop" (Gaussian hump in a
             square basin), "mounds" (dam break over dry mounds), "humps"
             (wet/dry bed humps, or fully wet), "sinusoid" (radial dam break
             over a rough bed, per-cell roughness), "ensemble" (independent
             dam breaks)
  nx, ny     quads of the jittered grid (2 nx ny triangles); for an ensemble
             the number of scenarios is `scenarios` and nx is unused
  precision  "f64" (the default arithmetic) or "f32"
  mode       "run" (steps), "advance" (to t_end), "grad" (rollout and
             backward over steps), "adjoint" (backward alone, of a recorded
             tape)
  io         "device" (CUDA tensors) or "host" (page-locked FP32 arrays)
"""
import math

import numpy as np
import torch

from paper_1807_00672_gb300 import grad as swe_grad
from paper_1807_00672_gb300 import swe

G, COURANT, H_EPS = 9.81, 0.7, 1e-6


def listed():
    return [
        # The smallest job: a classroom dam break run to its end time. 128
        # steps of a mesh that fits in a few tiles; latency is all of it.
        dict(name="stoker_2500_f64_advance", family="stoker", nx=50, ny=25, precision="f64",
             mode="advance", t_end=2.0, io="device"),
        # A dam break with drying and wetting, to an end time, in the paper's
        # precision: a model study on a small mesh.
        dict(name="mounds_20k_f64_advance", family="mounds", nx=160, ny=64, precision="f64",
             mode="advance", t_end=1.0, io="device"),
        # The paper's second test grid size in single precision: a small mesh
        # stepped many times.
        dict(name="drop_10k_f32_run", family="drop", nx=71, ny=71, precision="f32", mode="run",
             steps=200, io="device"),
        # The paper's third test grid size in its own precision.
        dict(name="drop_105k_f64_run", family="drop", nx=229, ny=229, precision="f64", mode="run",
             steps=50, io="device"),
        # A mesh a user keeps in reverse Cuthill-McKee order, odd sizes.
        dict(name="humps_250k_rcm_f32_run", family="humps", nx=501, ny=249, precision="f32",
             mode="run", steps=50, io="device", order="rcm"),
        # Half a million cells in the paper's precision, ragged.
        dict(name="humps_499k_f64_run", family="humps", nx=613, ny=407, precision="f64",
             mode="run", steps=20, io="device"),
        # The 1M wet/dry workload in single precision, fields in host memory.
        dict(name="humps_1m_f32_host", family="humps", nx=1000, ny=500, precision="f32",
             mode="run", steps=100, io="host"),
        # The paper's fourth test grid size, FP32 with the depth residual
        # that long runs use to keep their mass.
        dict(name="drop_1057k_f32_residual", family="drop", nx=727, ny=727, precision="f32",
             mode="run", steps=60, io="device", residual=True),
        # Many scenarios at once, in the shape the autotuner picks for them.
        dict(name="ensemble_32_f32_run", family="ensemble", scenarios=32, nx=0, ny=0, t_min=5_000,
             t_max=300_000, precision="f32", mode="run", steps=50, io="device", tile=256,
             halo_schedule=1),
        # The headline workload: 10M triangles, single precision.
        dict(name="sinusoid_10m_f32_run", family="sinusoid", nx=3163, ny=1581, precision="f32",
             mode="run", steps=20, io="device"),
        # Calibration: gauges, forward and backward through the PyTorch call.
        dict(name="calibration_1m_f32_grad", family="humps", nx=1000, ny=500, precision="f32",
             mode="grad", steps=100, every=50, gauges=64, wet=True, tile=256, io="device"),
        # The backward sweep alone, of a recorded run, in double precision
        # (several losses of one run).
        dict(name="humps_80k_f64_adjoint", family="humps", nx=283, ny=141, precision="f64",
             mode="adjoint", steps=40, every=10, gauges=16, wet=True, tile=256, io="device"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["f64", "f64", "f32", "f32", "f32", "ensemble", "grad"])
    if kind == "ensemble":
        c = dict(family="ensemble", scenarios=rng.randint(2, 64), nx=0, ny=0, t_min=5_000,
                 t_max=rng.choice([20_000, 50_000, 100_000]), precision="f32", mode="run",
                 steps=rng.randint(20, 60), io="device")
        if rng.random() < 0.5:
            c.update(tile=256, halo_schedule=1)
        return c
    if kind == "grad":
        prec = rng.choice(["f32", "f64"])
        ny = _log(rng, 20, 400 if prec == "f32" else 140)
        c = dict(family="humps", nx=2 * ny + rng.randint(-7, 7), ny=ny, precision=prec,
                 mode=rng.choice(["grad", "adjoint"]), steps=rng.randint(12, 60),
                 every=rng.choice([1, 7, 10, 25, 50]), gauges=rng.choice([1, 16, 64]), wet=True,
                 io="device")
        if rng.random() < 0.8:
            c["tile"] = 256
        return c
    family = rng.choice(["stoker", "drop", "mounds", "humps", "sinusoid"])
    cells = _log(rng, 1_000, 400_000 if kind == "f64" else 4_000_000)
    ny = max(8, int(round(math.sqrt(cells / (2.0 if family == "drop" else 4.0)))))
    nx = ny if family == "drop" else 2 * ny + rng.randint(-3, 3)
    c = dict(family=family, nx=nx, ny=ny, precision=kind, mode="run",
             steps=max(10, min(200, int((2.0e7 if kind == "f64" else 1.0e8) / cells))),
             io="device")
    if kind == "f32":
        c["io"] = rng.choice(["device", "device", "host"])
        option = rng.choice(["none", "none", "none", "residual", "rcm"])
        if option == "residual":
            c["residual"] = True
        elif option == "rcm" and cells < 500_000:
            c["order"] = "rcm"
    elif rng.random() < 0.2 and cells < 200_000:
        c["order"] = "rcm"
    return c


# --- inputs: meshes and initial fields, made on the GPU from the seed -------

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _grid(nx, ny, lx, ly, jitter, seed):
    """A jittered nx x ny grid of quads, each cut along its shorter diagonal
    (an unjittered grid by a coin): xy [V, 2] float64, tri [T, 3] int64."""
    dev = _device()
    gen = torch.Generator(device=dev).manual_seed(seed)
    x = torch.arange(nx + 1, dtype=torch.float64, device=dev) * (lx / nx)
    y = torch.arange(ny + 1, dtype=torch.float64, device=dev) * (ly / ny)
    X = x[None, :].repeat(ny + 1, 1)
    Y = y[:, None].repeat(1, nx + 1)
    if jitter > 0 and nx > 1 and ny > 1:
        j = torch.rand((2, ny - 1, nx - 1), generator=gen, dtype=torch.float64, device=dev) * 2 - 1
        X[1:-1, 1:-1] += j[0] * (jitter * lx / nx)
        Y[1:-1, 1:-1] += j[1] * (jitter * ly / ny)
    xy = torch.stack([X.reshape(-1), Y.reshape(-1)], 1)
    a = (torch.arange(ny, device=dev)[:, None] * (nx + 1) + torch.arange(nx, device=dev)).reshape(-1)
    b, c, d = a + 1, a + nx + 2, a + nx + 1
    lac = (xy[a] - xy[c]).square().sum(1)
    lbd = (xy[b] - xy[d]).square().sum(1)
    coin = torch.rand(a.shape[0], generator=gen, device=dev) < 0.5
    ac = torch.where(lac == lbd, coin, lac < lbd)[:, None] if jitter > 0 else coin[:, None]
    t1 = torch.where(ac, torch.stack([a, b, c], 1), torch.stack([a, b, d], 1))
    t2 = torch.where(ac, torch.stack([a, c, d], 1), torch.stack([b, c, d], 1))
    return xy, torch.stack([t1, t2], 1).reshape(-1, 3)


def _current(cx, cy, lx, ly, rng, speed):
    """A smooth velocity field of a few random waves, about `speed` m/s."""
    out = []
    for _ in range(2):
        v = torch.full_like(cx, rng.uniform(-0.4, 0.4) * speed)
        for _ in range(3):
            kx, ky = rng.uniform(-4, 4) * 2 * math.pi / lx, rng.uniform(-4, 4) * 2 * math.pi / ly
            v += rng.uniform(0.1, 0.4) * speed * torch.sin(kx * cx + ky * cy + rng.uniform(0, 6.28))
        out.append(v)
    return out


def _one(case, seed, nx, ny):
    """Mesh and fields (xy, tri, h, hu, hv, z, n) of one flow, float64."""
    fam = case["family"]
    rng = np.random.default_rng(seed)
    # Jitter 0.2: triangles of a mesh generator's quality. With 0.3 a mesh of
    # 1M quads has near-flat triangles in which the explicit scheme itself
    # amplifies a rounding error from step to step.
    if fam == "stoker":
        lx, ly, jitter = 2.0 * nx, 2.0 * ny, 0.0
    elif fam == "drop":
        lx, ly, jitter = 10_000.0, 10_000.0, 0.15
    elif fam == "mounds":
        lx, ly, jitter = 80.0, 32.0, 0.2
    elif fam == "humps":
        lx, ly, jitter = 10_000.0, 5_000.0, 0.2
    elif fam == "sinusoid":
        lx, ly, jitter = 100_000.0, 50_000.0, 0.2
    else:  # one scenario of an ensemble
        lx, ly, jitter = 10.0 * nx, 10.0 * ny, 0.2
    xy, tri = _grid(nx, ny, lx, ly, jitter, int(rng.integers(1 << 31)))
    cen = (xy[tri[:, 0]] + xy[tri[:, 1]] + xy[tri[:, 2]]) / 3.0
    cx, cy = cen[:, 0].contiguous(), cen[:, 1].contiguous()
    zero = torch.zeros_like(cx)
    z, n, speed = zero, 0.0, 0.3
    if fam == "stoker":
        h = torch.where(cx < 0.5 * lx, rng.uniform(8, 12), rng.uniform(0.8, 1.2)) + zero
        speed = 0.0
    elif fam == "drop":
        s = rng.uniform(400, 600)
        r2 = (cx - 0.5 * lx).square() + (cy - 0.5 * ly).square()
        h = 10.0 + rng.uniform(0.8, 1.2) * torch.exp(-r2 / (2 * s * s))
    elif fam == "mounds":
        for mx, my, height, radius in ((32.0, 8.0, 1.2, 9.0), (32.0, 24.0, 1.2, 9.0),
                                       (52.0, 16.0, 2.8, 11.0)):
            d = torch.hypot(cx - mx, cy - my)
            z = torch.maximum(z, height * (1.0 - d / radius).clamp(min=0.0))
        h = torch.where(cx < rng.uniform(17, 21), (rng.uniform(1.8, 2.2) - z).clamp(min=0.0), zero)
        n, speed = 0.02, 0.1
    elif fam == "humps":
        for _ in range(3):
            a, s = rng.uniform(0.5, 2.0), rng.uniform(300.0, 800.0)
            x0, y0 = rng.uniform(0, lx), rng.uniform(0, ly)
            z = z + a * torch.exp(-((cx - x0).square() + (cy - y0).square()) / (2 * s * s))
        top = float(z.max())
        inside = ((cx - lx / 2).abs() <= 500.0) & ((cy - ly / 2).abs() <= 500.0)
        if case.get("wet"):
            eta = top + 1.0 + inside.double()
        else:  # the highest hump's top stays dry
            z = z + (2.3 - top)
            eta = 2.0 + inside.double()
        h = (eta - z).clamp(min=0.0)
        n = 0.03
    elif fam == "sinusoid":
        w = rng.uniform(0.0, 1.0, size=8)
        w = 3.0 * w / w.sum()
        for k in range(8):
            lam, th, ph = rng.uniform(2_000, 50_000), rng.uniform(0, 6.283), rng.uniform(0, 6.283)
            z = z + w[k] * torch.sin((2 * math.pi / lam) * (math.cos(th) * cx + math.sin(th) * cy) + ph)
        h = torch.where(torch.hypot(cx - lx / 2, cy - ly / 2) < 5_000.0, 5.0, 1.0) + zero
        n = torch.from_numpy(rng.uniform(0.02, 0.05, size=h.shape[0])).to(h.device)
    else:
        h = torch.where(cx < 0.5 * lx, rng.uniform(2, 10), 1.0) + zero
        n = rng.uniform(0.01, 0.05)
    if speed > 0:
        u, v = _current(cx, cy, lx, ly, rng, speed)
        q = h * (h / 0.5).clamp(max=1.0)  # slower towards a shore
        hu, hv = q * u, q * v
    else:
        hu, hv = zero.clone(), zero.clone()
    return xy, tri, h, hu, hv, z + zero, torch.zeros_like(h) + n


def _flows(case, seed):
    if case["family"] != "ensemble":
        return [_one(case, seed, case["nx"], case["ny"])]
    rng = np.random.default_rng(seed + 77)
    size = np.random.default_rng(case["scenarios"])  # the sizes go with the case
    out = []
    for _ in range(case["scenarios"]):
        t = math.exp(size.uniform(math.log(case["t_min"]), math.log(case["t_max"])))
        ny = max(1, int(round(math.sqrt(t / 4.0))))
        out.append(_one(case, int(rng.integers(1 << 31)), 2 * ny, ny))
    return out


def _gauges(case, n_cells):
    return np.sort(np.random.default_rng(n_cells).choice(n_cells, case["gauges"], replace=False)).astype(np.int32)


def _seeds(case, seed, like):
    """dL/d(final h, hu, hv) and dL/d(gauge depths) of some smooth loss."""
    gen = torch.Generator(device=like.device).manual_seed(seed + 5)
    T = like.shape[0]
    ramp = torch.arange(T, dtype=torch.float64, device=like.device) / T
    a = torch.rand(8, generator=gen, dtype=torch.float64, device=like.device)
    gh = 0.5 + a[0] + a[1] * torch.sin(6.28 * (ramp + a[2]))
    ghu = a[3] * torch.cos(6.28 * (ramp + a[4])) + 0.2
    ghv = a[5] * torch.cos(6.28 * (ramp + a[6])) - 0.2
    gg = 0.5 + torch.rand((case["steps"], case["gauges"]), generator=gen, dtype=torch.float64,
                          device=like.device)
    return gh, ghu, ghv, gg


def _n_cells(case):
    if case["family"] != "ensemble":
        return 2 * case["nx"] * case["ny"]
    size = np.random.default_rng(case["scenarios"])
    total = 0
    for _ in range(case["scenarios"]):
        t = math.exp(size.uniform(math.log(case["t_min"]), math.log(case["t_max"])))
        total += 4 * max(1, int(round(math.sqrt(t / 4.0)))) ** 2
    return total


def prepare(case, seed):
    flows = _flows(case, seed)
    meshes = [(f[0].cpu().numpy(), f[1].to(torch.int32).cpu().numpy()) for f in flows]
    h, hu, hv, z, n = (torch.cat([f[k] for f in flows]) if len(flows) > 1 else flows[0][k]
                       for k in range(2, 7))
    del flows
    kw = dict(precision=case["precision"], order=case.get("order", "morton"),
              tile=case.get("tile", 0), halo_schedule=case.get("halo_schedule", 0),
              compensated_depth=bool(case.get("residual", False)))
    # One stream for the library and for the caller's own tensors.
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        return _prepare_on(side, case, seed, meshes, (h, hu, hv, z, n), kw)


def _prepare_on(side, case, seed, meshes, fields, kw):
    stream = side.cuda_stream
    h, hu, hv, z, n = (x.clone() for x in fields)  # this stream's own
    if case["family"] == "ensemble":
        mesh = swe.Mesh.ensemble(meshes, stream=stream, **kw)
    else:
        mesh = swe.Mesh(*meshes[0], stream=stream, **kw)
    s = dict(case=case, mesh=mesh, f32=case["precision"] == "f32", side=side)
    if case["mode"] == "grad":
        dt = torch.float32 if s["f32"] else torch.float64
        s["inputs"] = [x.to(dt).requires_grad_(True) for x in (h, hu, hv, z, n)]
        s["seeds"] = [x.to(dt) for x in _seeds(case, seed, h)]
        s["gauges"] = _gauges(case, mesh.T)
        return s
    fields = [h, hu, hv, z, n]
    state = swe.State.from_device(mesh, *(x.data_ptr() for x in fields), stream=stream)
    s["state"] = state
    if case["mode"] == "adjoint":
        s["tape"] = swe.Tape(state, case["steps"], case["every"], _gauges(case, mesh.T),
                             host_gauges=False)
        s["seeds"] = list(_seeds(case, seed, h))
        s["keep"] = fields
        return s
    if case["io"] == "host":  # page-locked FP32 arrays, as a solver's driver keeps them
        s["inputs"] = [x.float().cpu().pin_memory() for x in (h, hu, hv)]
        s["outputs"] = [torch.empty(mesh.T, dtype=torch.float32, pin_memory=True) for _ in range(3)]
    else:
        s["inputs"] = [h, hu, hv]
    if case["mode"] == "run":
        state.run(0)  # captures the step graph, as a driver does before its time loop
    return s


def run(s):
    with torch.cuda.stream(s["side"]):
        return _run_on(s, s["case"], s["side"].cuda_stream)


def _run_on(s, case, stream):
    if case["mode"] == "grad":
        outs = swe_grad.rollout(s["mesh"], *s["inputs"], case["steps"], case["every"], s["gauges"])
        grads = torch.autograd.grad(outs, s["inputs"], s["seeds"])
        return dict(out=list(o.detach() for o in outs), grad=list(grads))
    T = s["mesh"].T
    if case["mode"] == "adjoint":
        grads = [torch.empty(T, dtype=torch.float64, device="cuda") for _ in range(5)]
        s["tape"].grad_device([x.data_ptr() for x in s["seeds"]], [x.data_ptr() for x in grads],
                              stream=stream)
        return dict(grad=grads)
    state = s["state"]
    if case["io"] == "host":
        state.set_f32(*(x.numpy() for x in s["inputs"]))
    else:
        state.set_device(*(x.data_ptr() for x in s["inputs"]), stream=stream)
    if case["mode"] == "advance":
        state.advance(case["t_end"])
    else:
        state.run(case["steps"], sync=False)
    if case["io"] == "host":
        out = s["outputs"]
        t, mass = state.copy_out_f32(*(x.numpy() for x in out))
    else:
        out = [torch.empty(T, dtype=torch.float64, device="cuda") for _ in range(3)]
        t, mass = state.copy_out_device(*(x.data_ptr() for x in out), stream=stream)
        if s["f32"]:
            out = [x.float() for x in out]  # an FP32 state's fields, handed on as FP32 tensors
    return dict(h=out[0], hu=out[1], hv=out[2], t=t, mass=mass)


# What one step reads and writes per cell, each value once: the cell's h, hu,
# hv, z, 1/area and n, its share (1.5 edges) of the edges' normal, length and
# two cell numbers, and the new h, hu, hv. 200 operations: about 95 per edge
# and 60 per cell.
_FLOPS = 200.0


def work(case):
    T = _n_cells(case)
    w = 4 if case["precision"] == "f32" else 8
    step = T * (13.5 * w + 12.0 + (8.0 if case.get("residual") else 0.0))
    K = case.get("steps")
    if K is None:  # advance: about as many CFL steps as the listed sizes take
        K = 128 if case["family"] == "stoker" else 200
    # A mesh and state that fit in the 129 MB L2 need not cross HBM each step.
    fits = step < 129e6
    if case["mode"] in ("grad", "adjoint"):
        adj = T * (23.5 * w + 12.0)  # U^n, U^n+1, lambda, the cell's constants, edges, outputs
        fwd = step * (1 if fits else K) if case["mode"] == "grad" else 0.0
        tape = T * 4.0 * w * K       # each step's state is read back (stored or recomputed)
        return {"bytes": fwd + (adj + tape if fits else adj * K) + T * 8 * 8.0,
                "flops": T * K * _FLOPS * (4.0 if case["mode"] == "grad" else 3.0)}
    io = T * (24.0 if case["io"] == "host" else 48.0)
    return {"bytes": (step if fits else step * K) + io, "flops": T * K * _FLOPS}


# --- the same scheme in plain torch, 64 bits --------------------------------

def _topology(flows):
    """Cells and edges of the concatenated flows, float64: areas, perimeters,
    each edge's left (lower) and right cell, outward normal and length, and
    each cell's three edges."""
    tri, xy, scen, v0 = [], [], [], 0
    for i, f in enumerate(flows):
        tri.append(f[1] + v0)
        xy.append(f[0])
        scen.append(torch.full((f[1].shape[0],), i, dtype=torch.int64, device=f[0].device))
        v0 += f[0].shape[0]
    tri, xy, scen = torch.cat(tri), torch.cat(xy), torch.cat(scen)
    T, dev = tri.shape[0], tri.device
    p = xy[tri]
    area = 0.5 * ((p[:, 1, 0] - p[:, 0, 0]) * (p[:, 2, 1] - p[:, 0, 1])
                  - (p[:, 2, 0] - p[:, 0, 0]) * (p[:, 1, 1] - p[:, 0, 1]))
    a = tri.reshape(-1)
    b = tri[:, [1, 2, 0]].reshape(-1)
    key, order = torch.sort(torch.minimum(a, b) * v0 + torch.maximum(a, b), stable=True)
    first = torch.ones(3 * T, dtype=torch.bool, device=dev)
    first[1:] = key[1:] != key[:-1]
    eid = torch.cumsum(first, 0) - 1
    E = int(eid[-1]) + 1
    edge = torch.empty(3 * T, dtype=torch.int64, device=dev)
    edge[order] = eid
    half = order[first]  # the lower cell's half-edge (the sort is stable)
    left = half // 3
    right = torch.full((E,), -1, dtype=torch.int64, device=dev)
    right[eid[~first]] = order[~first] // 3
    d = xy[b[half]] - xy[a[half]]
    ln = d.square().sum(1).sqrt()
    edge = edge.reshape(T, 3)
    perim = ln[edge[:, 0]] + ln[edge[:, 1]] + ln[edge[:, 2]]
    is_left = left[edge] == torch.arange(T, device=dev)[:, None]
    return dict(T=T, area=area, perim=perim, left=left, right=right, nx=d[:, 1] / ln,
                ny=-d[:, 0] / ln, ln=ln, edge=edge, is_left=is_left, scen=scen, n=len(flows))


def _safe_sqrt(x):
    pos = x > 0
    return torch.where(pos, torch.where(pos, x, torch.ones_like(x)).sqrt(), torch.zeros_like(x))


def _velocity(h, q):
    wet = h > H_EPS
    return torch.where(wet, q / torch.where(wet, h, torch.ones_like(h)), torch.zeros_like(h))


def _rate(m, h, hu, hv):
    """The CFL time step of each scenario, and of each cell."""
    speed = (hu * hu + hv * hv).sqrt() / h.clamp(min=1e-300) + (G * h).sqrt()
    r = torch.where(h > H_EPS, speed * (m["perim"] / m["area"]), torch.zeros_like(h))
    top = torch.zeros(m["n"], dtype=torch.float64, device=h.device)
    top = top.scatter_reduce(0, m["scen"], r, "amax")
    return COURANT / top


def _step(m, h, hu, hv, z, n, dt):
    """One explicit step with the time step `dt` per cell; differentiable,
    each max/min taking its first argument on a tie."""
    zero = torch.zeros((), dtype=torch.float64, device=h.device)
    L, R, nx, ny, ln = m["left"], m["right"], m["nx"], m["ny"], m["ln"]
    wall = R < 0
    Rc = torch.where(wall, L, R)
    u, v = _velocity(h, hu), _velocity(h, hv)
    hA, zA, hB, zB = h[L], z[L], h[Rc], z[Rc]
    uA, vA, uB, vB = u[L], v[L], u[Rc], v[Rc]
    unA, utA = uA * nx + vA * ny, vA * nx - uA * ny
    unB = torch.where(wall, -unA, uB * nx + vB * ny)
    utB = torch.where(wall, utA, vB * nx - uB * ny)
    zs = torch.where(zA >= zB, zA, zB)
    xA, xB = hA + (zA - zs), hB + (zB - zs)
    wA, wB = xA > H_EPS, xB > H_EPS
    hAs, hBs = torch.where(wA, xA, zero), torch.where(wB, xB, zero)
    cA, cB = _safe_sqrt(G * hAs), _safe_sqrt(G * hBs)
    us = (unA + unB) / 2 + cA - cB
    cs = (cA + cB) / 2 + (unA - unB) / 4
    a1, a2, b1, b2 = unA - cA, us - cs, unB + cB, us + cs
    SA = torch.where(wA & wB, torch.where(a1 <= a2, a1, a2), torch.where(wA, a1, unB - 2 * cB))
    SB = torch.where(wA & wB, torch.where(b1 >= b2, b1, b2), torch.where(wA, unA + 2 * cA, b1))
    Sm, Sp = torch.where(SA < 0, SA, zero), torch.where(SB > 0, SB, zero)
    live = wA | wB
    inv = 1.0 / torch.where(live, Sp - Sm, torch.ones_like(Sp))
    qA, qB = hAs * unA, hBs * unB
    fA, fB = qA * unA + G / 2 * hAs * hAs, qB * unB + G / 2 * hBs * hBs
    F0 = torch.where(live, (Sp * qA - Sm * qB + Sm * Sp * (hBs - hAs)) * inv, zero)
    F1 = torch.where(live, (Sp * fA - Sm * fB + Sm * Sp * (qB - qA)) * inv, zero)
    F2 = F0 * torch.where(F0 >= 0, utA, utB)
    F0, F2 = torch.where(wall, zero, F0), torch.where(wall, zero, F2)
    pA, pB = G / 2 * (hA * hA - hAs * hAs), G / 2 * (hB * hB - hBs * hBs)
    c0, fx, fy = ln * F0, F1 * nx - F2 * ny, F1 * ny + F2 * nx
    A1, A2 = ln * (fx + pA * nx), ln * (fy + pA * ny)
    B1, B2 = ln * (fx + pB * nx), ln * (fy + pB * ny)
    edge, isl = m["edge"], m["is_left"]
    R0 = torch.where(isl, c0[edge], -c0[edge]).sum(1)
    R1 = torch.where(isl, A1[edge], -B1[edge]).sum(1)
    R2 = torch.where(isl, A2[edge], -B2[edge]).sum(1)
    k = dt / m["area"]
    h1, qx, qy = h - k * R0, hu - k * R1, hv - k * R2
    h1 = torch.where(h1 > 0, h1, zero)
    wet = h1 > H_EPS
    q = _safe_sqrt(qx * qx + qy * qy)
    hs = torch.where(wet, h1, torch.ones_like(h1))
    d = 1 + dt * G * n * n * q / hs.pow(7.0 / 3.0)
    return h1, torch.where(wet, qx / d, zero), torch.where(wet, qy / d, zero)


def exact(case, seed):
    flows = _flows(case, seed)
    m = _topology(flows)
    h, hu, hv, z, n = (torch.cat([f[k] for f in flows]) for k in range(2, 7))
    if case["mode"] in ("grad", "adjoint"):
        return _exact_grad(case, seed, m, h, hu, hv, z, n)
    t_end = case.get("t_end", math.inf)
    t = torch.zeros(m["n"], dtype=torch.float64, device=h.device)
    k = 0
    while k < case.get("steps", 1 << 30):
        dt = torch.minimum(_rate(m, h, hu, hv), t_end - t)
        h, hu, hv = _step(m, h, hu, hv, z, n, dt[m["scen"]])
        t = t + dt
        k += 1
        if t_end < math.inf and float((t_end - t).min()) <= 1e-14 * t_end:
            break
    return dict(h=h, hu=hu, hv=hv, t=float(t[0]), mass=float((m["area"] * h).sum()))


def _exact_grad(case, seed, m, h, hu, hv, z, n):
    K = case["steps"]
    gauges = torch.from_numpy(_gauges(case, m["T"])).to(h.device).long()
    gh, ghu, ghv, gg = _seeds(case, seed, h)
    states, dts, depths = [(h, hu, hv)], [], []
    with torch.no_grad():
        for k in range(K):
            dts.append(_rate(m, *states[-1])[m["scen"]])
            states.append(_step(m, *states[-1], z, n, dts[-1]))
            depths.append(states[-1][0][gauges])
    lam = [gh, ghu, ghv]
    dz, dn = torch.zeros_like(z), torch.zeros_like(n)
    for k in reversed(range(K)):
        lam[0] = lam[0].clone()
        lam[0].index_add_(0, gauges, gg[k])
        ins = [x.detach().requires_grad_(True) for x in (*states[k], z, n)]
        outs = _step(m, *ins, dts[k])
        got = torch.autograd.grad(outs, ins, lam)
        lam = list(got[:3])
        dz, dn = dz + got[3], dn + got[4]
    grads = [*lam, dz, dn]
    if case["mode"] == "adjoint":
        return dict(grad=grads)
    return dict(out=[*states[-1], torch.stack(depths)], grad=grads)
