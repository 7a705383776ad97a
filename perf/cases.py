"""Timed work of the library: what its users call, over the sizes they call it at.

Every case goes through the public binding (bsgd_forward_project,
bsgd_back_project, Projector, bsgd_solve, State.block_step, Server). Images are
seeded ellipse / ellipsoid phantoms, sinograms their exact line integrals with
Poisson counting noise, which is what a scanner hands over.

listed()  the cases; draw(rng) one more of the same ranges
prepare() inputs on the GPU and the handle a program keeps (geometry, state, server)
run()     one pass; work() its compulsory bytes and multiply-adds
exact()   the same outputs in FP64 by plain torch, where that takes seconds
"""
import math

import numpy as np
import torch

from paper_1903_11874_gb300 import binding as B
from paper_1903_11874_gb300.autograd import Projector

KAPPA = 0.01       # attenuation per mm of unit density
COUNTS = 1e4       # unattenuated photons per pixel
_STORE = {"f32": B.F32, "bf16": B.BF16, "f16": B.F16}
_TORCH = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


# ---------------------------------------------------------------------------
# The cases

def _case(name, op, kind, n, views, nu, **more):
    c = dict(op=op, kind=kind, nx=n, ny=n, nz=1 if kind != "cone3d" else n, voxel=1.0, views=views,
             nu=nu, nv=1 if kind != "cone3d" else nu, pixel=1.0, dso=0.0, dsd=0.0, M=1, N=1,
             storage="f32", batch=1, epochs=1, iters=1, kM=1, kN=1, pairs="uniform", cells="none",
             tv=0.0)
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    cone = dict(voxel=1.0, pixel=1.6, dso=500.0, dsd=1000.0)
    return [
        # one projection of a 64^2 slice: the smallest call there is, all launch latency
        _case("forward_par2d_64", "forward", "par2d", 64, 90, 96, M=4, N=4),
        # filtered-back-projection sized fan-beam slice, back projected
        _case("backward_fan2d_256", "backward", "fan2d", 256, 360, 384, pixel=2.0, dso=500.0,
              dsd=1000.0, M=4, N=4),
        # a whole slice reconstruction: many short dependent iterations
        _case("solve_par2d_64", "solve", "par2d", 64, 90, 96, M=4, N=4, epochs=10),
        # a training step through the autograd projector: forward, loss, gradient
        _case("train_cone_128", "train", "cone3d", 128, 180, 192, batch=4, **cone),
        # simulation of a full scan from a 16-bit volume
        _case("forward_cone_256_bf16", "forward", "cone3d", 256, 360, 256, M=8, N=8, storage="bf16",
              **cone),
        # the adjoint of a full scan
        _case("backward_cone_256", "backward", "cone3d", 256, 360, 256, M=8, N=8, **cone),
        # a small ragged reconstruction stepped iteration by iteration: odd sides,
        # uneven slabs and row blocks, partly filled detector tiles
        _case("step_cone_odd", "step", "cone3d", 50, 43, 67, ny=47, nz=37, nv=53, M=5, N=3, iters=30,
              voxel=1.1, pixel=1.7, dso=160.0, dsd=320.0),
        # the headline reconstruction: one epoch of residual-weighted block pairs
        _case("solve_cone_256", "solve", "cone3d", 256, 360, 256, M=8, N=8, pairs="residual", **cone),
        # the method's two-slab scan set-up: two column blocks per iteration, long source distance
        _case("step_cone_256_two", "step", "cone3d", 256, 360, 400, M=5, N=8, kN=2, iters=5,
              pixel=1.0, dso=1536.0, dsd=2536.0),
        # importance sampling by detector quadrants, four column blocks per iteration
        _case("step_cone_256_cells", "step", "cone3d", 256, 360, 512, M=5, N=8, kN=4, iters=5,
              cells="geometric", pixel=1.0, dso=1000.0, dsd=1536.0),
        # the largest: a 512^3 volume in 16-bit storage with total-variation regularisation
        _case("solve_cone_512_bf16_tv", "solve", "cone3d", 512, 720, 512, M=16, N=16, storage="bf16",
              tv=1e-3, voxel=0.5, pixel=0.8, dso=500.0, dsd=1000.0),
        # a mixed queue of small and mid-size requests served together from host buffers
        _case("serve_mix", "serve", "cone3d", 128, 180, 128, M=8, N=8, epochs=2, batch=6, voxel=2.0,
              pixel=3.2, dso=500.0, dsd=1000.0),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["forward", "backward", "train", "solve", "step"])
    store = rng.choice(["f32", "f32", "bf16", "f16"])
    if op != "train" and rng.random() < 0.25:
        n = log_int(32, 512)
        kind = rng.choice(["par2d", "fan2d"])
        more = dict(pixel=rng.uniform(0.7, 1.3)) if kind == "par2d" else \
            dict(pixel=rng.uniform(1.4, 2.6), dso=2.0 * n, dsd=4.0 * n)
        return _case("", op, kind, n, log_int(36, 720), int(n * rng.uniform(0.8, 1.6)),
                     ny=max(16, int(n * rng.uniform(0.7, 1.0))), M=rng.randint(1, 6), N=rng.randint(1, 6),
                     storage=store, epochs=2, iters=8, **more)
    n = log_int(24, 160 if op == "train" else 256)
    h = 256.0 / n
    nu = int(n * rng.uniform(0.8, 1.4))
    views = log_int(24, 180 if op == "train" else 360)
    far = rng.random() < 0.3
    more = {}
    if op in ("solve", "step"):
        more["kN"] = rng.choice([1, 1, 1, 2, 4])
        if more["kN"] == 1 and rng.random() < 0.4:
            more["pairs"] = "residual"
        elif rng.random() < 0.3:
            more["cells"] = rng.choice(["geometric", "uniform"])
    return _case("", op, "cone3d", n, views, nu, ny=max(16, int(n * rng.uniform(0.8, 1.0))),
                 nz=max(8, int(n * rng.uniform(0.5, 1.0))), nv=max(8, int(nu * rng.uniform(0.6, 1.0))),
                 M=rng.randint(1, 8), N=rng.choice([4, 5, 7, 8]), voxel=h,
                 pixel=(420.0 if far else 410.0) / nu, dso=1000.0 if far else 500.0,
                 dsd=1536.0 if far else 1000.0, storage="f32" if op == "train" else store,
                 batch=rng.randint(1, 3) if op == "train" else 1,
                 iters=8 if op == "step" else 1, **more)


# ---------------------------------------------------------------------------
# Geometry, phantoms and data (torch on the GPU, FP64 geometry)

def _geo(c):
    return dict(kind=c["kind"], nx=c["nx"], ny=c["ny"], nz=c["nz"], dx=c["voxel"], dy=c["voxel"],
                dz=c["voxel"], n_views=c["views"], nu=c["nu"], nv=c["nv"], du=c["pixel"],
                dv=c["pixel"], dso=c["dso"], dsd=c["dsd"])


def _cos_sin(c, a):
    b = a * ((math.pi if c["kind"] == "par2d" else 2.0 * math.pi) / c["views"])
    k = round(b / (0.5 * math.pi))
    if abs(b - k * 0.5 * math.pi) <= 1e-9:      # axis-aligned views are exactly aligned
        return ((1.0, 0.0), (0.0, 1.0), (-1.0, 0.0), (0.0, -1.0))[k % 4]
    return math.cos(b), math.sin(b)


def _ends(c, a, dev="cuda"):
    """Both ends of the rays of view a, in mm, FP64: xy ends per column u and
    z ends per row v."""
    cs, sn = _cos_sin(c, a)
    u = (torch.arange(c["nu"], device=dev, dtype=torch.float64) - 0.5 * (c["nu"] - 1)) * c["pixel"]
    v = (torch.arange(c["nv"], device=dev, dtype=torch.float64) - 0.5 * (c["nv"] - 1)) * c["pixel"]
    if c["kind"] == "par2d":
        R = 0.5 * c["voxel"] * math.hypot(c["nx"], c["ny"]) + 1.0
        p = (-R * cs - u * sn, -R * sn + u * cs)
        q = (R * cs - u * sn, R * sn + u * cs)
        return p, q, v * 0.0, v * 0.0
    back = c["dsd"] - c["dso"]
    one = torch.ones_like(u)
    p = (c["dso"] * cs * one, c["dso"] * sn * one)
    q = (-back * cs - u * sn, -back * sn + u * cs)
    return p, q, v * 0.0, v


def _blobs(c, seed):
    """Ellipsoids (ellipses for a slice): centre, half axes, rotation, density, in mm."""
    rng = np.random.default_rng(seed)
    half = 0.5 * c["voxel"] * np.array([c["nx"], c["ny"], c["nz"]])
    out = []
    for _ in range(8):
        ctr = rng.uniform(-0.6, 0.6, 3) * half
        ax = rng.uniform(0.08, 0.4, 3) * half
        if c["nz"] == 1:
            ctr[2], ax[2] = 0.0, 1e9
        phi, rho = rng.uniform(0.0, math.pi), rng.uniform(0.1, 1.0) * KAPPA
        out.append((ctr, ax, math.cos(phi), math.sin(phi), rho))
    return out


def _volume(c, blobs):
    def axis(n):
        return (torch.arange(n, device="cuda", dtype=torch.float32) - 0.5 * (n - 1)) * c["voxel"]
    x, y, z = axis(c["nx"])[None, None], axis(c["ny"])[None, :, None], axis(c["nz"])[:, None, None]
    vol = torch.zeros(c["nz"], c["ny"], c["nx"], device="cuda")
    for ctr, ax, cp, sp, rho in blobs:
        xr = cp * (x - ctr[0]) + sp * (y - ctr[1])
        yr = -sp * (x - ctr[0]) + cp * (y - ctr[1])
        vol += rho * ((xr / ax[0]) ** 2 + (yr / ax[1]) ** 2 + ((z - ctr[2]) / ax[2]) ** 2 <= 1.0)
    return vol


def _line_integrals(c, blobs):
    """Exact line integrals of the ellipsoids: [views, nv, nu] float32."""
    y = torch.zeros(c["views"], c["nv"], c["nu"], device="cuda")
    many = max(1, (1 << 24) // (c["nv"] * c["nu"]))      # views at a time
    for a in range(0, c["views"], many):
        b = min(c["views"], a + many)
        ends = [_ends(c, k, "cpu") for k in range(a, b)]
        px, py, qx, qy = (torch.stack([e[m][k] for e in ends]).float().cuda()[:, None, :]
                          for m in (0, 1) for k in (0, 1))
        pz, qz = (torch.stack([e[m] for e in ends]).float().cuda()[:, :, None] for m in (2, 3))
        dx, dy, dz = qx - px, qy - py, qz - pz
        length = torch.sqrt(dx * dx + dy * dy + dz * dz)
        for ctr, ax, cp, sp, rho in blobs:
            ox, oy, oz = px - ctr[0], py - ctr[1], (pz - ctr[2]) / ax[2]
            ux, uy = (cp * ox + sp * oy) / ax[0], (-sp * ox + cp * oy) / ax[1]
            ex, ey, ez = (cp * dx + sp * dy) / ax[0], (-sp * dx + cp * dy) / ax[1], dz / ax[2]
            A = ex * ex + ey * ey + ez * ez
            h = (ux * ex + uy * ey + oz * ez) / A
            # squared distance of the centre from the line, in half axes
            fx, fy, fz = ux - h * ex, uy - h * ey, oz - h * ez
            y[a:b] += rho * length * 2.0 * torch.sqrt(((1.0 - fx * fx - fy * fy - fz * fz) / A).clamp_min(0.0))
    return y


def _scan(c, blobs, seed):
    """Log data of a photon-counting scan: -ln(max(N, 1) / I0), N ~ Poisson."""
    y = _line_integrals(c, blobs)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return -torch.log(torch.poisson(y.neg_().exp_().mul_(COUNTS), generator=g).clamp_min_(1.0) / COUNTS)


def _step_size(c):
    """A quarter of the Lipschitz step, from the row-sum times column-sum bound of ||A^J||^2."""
    h = c["voxel"]
    iso = c["pixel"] * (c["dso"] / c["dsd"] if c["kind"] != "par2d" else 1.0)
    row = h * 1.3 * max(c["nx"], c["ny"])
    col = c["views"] * (h * h / iso if c["kind"] != "cone3d" else h ** 3 / iso ** 2) * 1.3
    return 0.25 / (row * col)


def _params(c, seed, **more):
    cells = {"none": B.CELLS_NONE, "geometric": B.CELLS_GEOMETRIC, "uniform": B.CELLS_UNIFORM}[c["cells"]]
    return B.SolveParams(alpha=c["kM"] / c["M"], gamma=c["kN"] / c["N"], epochs=c["epochs"],
                         step_rule=B.STEP_FIXED, mu=_step_size(c), seed=seed,
                         pair_sampling=B.PAIRS_RESIDUAL if c["pairs"] == "residual" else B.PAIRS_UNIFORM,
                         cells=cells, n_cells=1 if c["cells"] == "none" else (4 if c["nv"] > 1 else 2),
                         tv_lambda=c["tv"], storage=_STORE[c["storage"]], **more)


# the queue of the served case: sizes (voxels a side), views, storage
_QUEUE = [(64, 90, "f32"), (128, 180, "f32"), (64, 180, "bf16"), (64, 90, "f32"), (128, 90, "bf16"),
          (64, 180, "f32")]


def _request(c, k):
    n, views, store = _QUEUE[k % len(_QUEUE)]
    h = 256.0 / n
    return dict(c, nx=n, ny=n, nz=n, nu=n, nv=n, views=views, voxel=h, pixel=1.6 * h, storage=store)


class _Served:
    """A server and the requests a pass hands to it; closed with the state."""

    def __init__(self, c, seed):
        self.server = B.Server(budget_bytes=16 << 30, max_slots=8)
        self.requests = []
        for k in range(c["batch"]):
            q = _request(c, k)
            y = _scan(q, _blobs(q, seed + k), seed + k).reshape(-1).cpu().numpy()
            self.requests.append((_geo(q), q["M"], q["N"], _params(q, seed + k), y))

    def __del__(self):
        self.server.close()


def prepare(case, seed):
    c = case
    s = {"case": c}
    if c["op"] == "serve":
        s["served"] = _Served(c, seed)
        return s
    blobs = _blobs(c, seed)
    s["geom"] = B.Geometry(M=c["M"], N=c["N"], **_geo(c))
    if c["op"] == "forward":
        s["x"] = _volume(c, blobs).to(_TORCH[c["storage"]])
        s["y"] = torch.zeros(c["views"], c["nv"], c["nu"], device="cuda")
    elif c["op"] == "backward":
        s["r"] = _scan(c, blobs, seed).to(_TORCH[c["storage"]])
        s["x"] = torch.zeros(c["nz"], c["ny"], c["nx"], device="cuda")
    elif c["op"] == "train":
        # the network's current volumes and the measured scans of other objects
        s["x"] = torch.stack([_volume(c, _blobs(c, seed + 100 + k)) for k in range(c["batch"])])
        s["x"].requires_grad_(True)
        s["target"] = torch.stack([_scan(c, _blobs(c, seed + k), seed + k) for k in range(c["batch"])])
    else:
        s["y"] = _scan(c, blobs, seed)
        s["x"] = torch.zeros(c["nz"], c["ny"], c["nx"], device="cuda", dtype=_TORCH[c["storage"]])
        if c["op"] == "step":
            s["state"] = B.State(s["geom"], _params(c, seed), s["y"])
        else:
            s["params"] = _params(c, seed, zero_start=True)
    return s


def run(state):
    c = state["case"]
    op = c["op"]
    if op == "forward":
        return B.bsgd_forward_project(state["geom"], state["x"], state["y"])
    if op == "backward":
        return B.bsgd_back_project(state["geom"], state["r"], state["x"])
    if op == "train":
        x = state["x"]
        x.grad = None
        y = Projector.apply(x, state["geom"])
        (0.5 * (y - state["target"]).square().sum()).backward()
        return {"y": y.detach(), "grad": x.grad}
    if op == "solve":
        report = B.bsgd_solve(state["geom"], state["params"], state["y"], state["x"])
        return {"x": state["x"], "updates": report["updates"]}
    if op == "step":
        return state["state"].block_step(state["x"], c["iters"])
    server = state["served"].server
    ids = [server.submit(*q) for q in state["served"].requests]
    return [server.wait(i)[0] for i in ids]


# ---------------------------------------------------------------------------
# Compulsory work

def _updates(c):
    """Voxels that the rays of one scan cross: plane crossings inside the volume, on a
    sample of views, rows and columns, scaled up."""
    views = np.unique(np.linspace(0, c["views"] - 1, 9).astype(int))
    total = 0.0
    n, h = (c["nx"], c["ny"], c["nz"]), c["voxel"]
    for a in views:
        p, q, pz, qz = _ends(c, int(a), "cpu")
        us = np.unique(np.linspace(0, c["nu"] - 1, 65).astype(int))
        vs = np.unique(np.linspace(0, c["nv"] - 1, 33).astype(int))
        lo, hi, d = np.zeros((vs.size, us.size)), np.ones((vs.size, us.size)), []
        for k, (e0, e1) in enumerate(((p[0].numpy()[us][None], q[0].numpy()[us][None]),
                                      (p[1].numpy()[us][None], q[1].numpy()[us][None]),
                                      (pz.numpy()[vs][:, None], qz.numpy()[vs][:, None]))):
            dk = np.where(np.abs(e1 - e0) < 1e-12, 1e-12, e1 - e0)
            t0, t1 = (-0.5 * n[k] * h - e0) / dk, (0.5 * n[k] * h - e0) / dk
            lo, hi = np.maximum(lo, np.minimum(t0, t1)), np.minimum(hi, np.maximum(t0, t1))
            d.append(np.abs(dk) / h)
        inside = np.maximum(hi - lo, 0.0)
        total += np.mean(inside * (d[0] + d[1] + d[2]) + (inside > 0))
    return total / views.size * c["views"] * c["nu"] * c["nv"]


def work(case):
    c = case
    size = {"f32": 4, "bf16": 2, "f16": 2}[c["storage"]]
    if c["op"] == "serve":
        parts = []
        for k in range(c["batch"]):
            q = _request(c, k)
            parts.append(work(dict(q, op="solve", batch=1)))
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    vox, rays = c["nx"] * c["ny"] * c["nz"], c["views"] * c["nu"] * c["nv"]
    one = 2.0 * _updates(c)           # a multiply-add per voxel and ray, one direction
    if c["op"] == "forward":
        return {"bytes": vox * size + rays * 4, "flops": one}
    if c["op"] == "backward":
        return {"bytes": rays * size + vox * 4, "flops": one}
    if c["op"] == "train":
        return {"bytes": c["batch"] * 2 * (vox + rays) * 4, "flops": c["batch"] * 2 * one}
    # a pair's rays are traced forward and back; an iteration takes kM x kN of the M x N pairs
    share = c["kM"] * c["kN"] / (c["M"] * c["N"])
    if c["cells"] != "none":
        share *= 0.5                  # the drawn quadrant (half) holds about half a block's rays
    iters = c["iters"] if c["op"] == "step" else c["epochs"] * round(1.0 / (c["kM"] * c["kN"] / (c["M"] * c["N"])))
    if c["op"] == "step":             # the drawn rows read, the drawn slabs read and written
        data = c["iters"] * (rays * c["kM"] / c["M"] * size + 2 * vox * c["kN"] / c["N"] * size)
    else:                             # the scan read once, the image written once
        data = rays * 4 + vox * size
    return {"bytes": data, "flops": 2 * one * share * iters}


# ---------------------------------------------------------------------------
# The same results in FP64: rays cut at every x and y plane (sorted), each piece
# cut at the z planes it meets

def _pieces(c, a):
    """Cells and parameter ranges of view a's rays in the xy plane: flat cell
    [nu, S], start and end parameter [nu, S] (equal where there is no piece)."""
    p, q, _, _ = _ends(c, a)
    h = c["voxel"]
    o = [(p[k] + 0.5 * n * h) / h for k, n in ((0, c["nx"]), (1, c["ny"]))]
    d = [(q[k] - p[k]) / h for k in (0, 1)]
    lo, hi, ts, ok = 0.0, 1.0, [], True
    for k, n in ((0, c["nx"]), (1, c["ny"])):
        flat = d[k].abs() < 1e-12
        t = (torch.arange(n + 1, device="cuda", dtype=torch.float64)[None] - o[k][:, None]) / \
            torch.where(flat, torch.ones_like(d[k]), d[k])[:, None]
        inside = (o[k] >= 0) & (o[k] < n)
        t0 = torch.where(flat, torch.where(inside, 0.0, 2.0).double(), torch.minimum(t[:, 0], t[:, -1]))
        t1 = torch.where(flat, torch.where(inside, 1.0, -1.0).double(), torch.maximum(t[:, 0], t[:, -1]))
        lo, hi = torch.clamp(t0, min=lo) if k == 0 else torch.maximum(t0, lo), \
            torch.clamp(t1, max=hi) if k == 0 else torch.minimum(t1, hi)
        ts.append(torch.where(flat[:, None], torch.zeros_like(t), t))
    hi = torch.maximum(lo, hi)
    t = torch.cat(ts, 1).clamp(min=lo[:, None], max=hi[:, None]).sort(1).values
    t = torch.cat([lo[:, None], t, hi[:, None]], 1)
    t0, t1 = t[:, :-1], t[:, 1:]
    mid = 0.5 * (t0 + t1)
    ix = (o[0][:, None] + mid * d[0][:, None]).floor().long().clamp(0, c["nx"] - 1)
    iy = (o[1][:, None] + mid * d[1][:, None]).floor().long().clamp(0, c["ny"] - 1)
    keep = (t1 > t0).any(0)
    return (iy * c["nx"] + ix)[:, keep], t0[:, keep], t1[:, keep]


def _chords(c, a):
    """Yields (cell index [nv, nu, S] into z-major flat voxels, length in mm) for
    view a, until every z cell a piece meets is covered."""
    cell, t0, t1 = _pieces(c, a)
    p, q, pz, qz = _ends(c, a)
    h, plane = c["voxel"], c["nx"] * c["ny"]
    length = torch.sqrt(((q[0] - p[0]) ** 2 + (q[1] - p[1]) ** 2)[None] + ((qz - pz) ** 2)[:, None])
    zo, zd = (pz / h + 0.5 * c["nz"])[:, None, None], ((qz - pz) / h)[:, None, None]
    za, zb = zo + t0 * zd, zo + t1 * zd
    low, high = torch.minimum(za, zb), torch.maximum(za, zb)
    first, width = low.floor(), high - low
    more = int((high - first).max().ceil().item()) if cell.numel() else 0
    flat = width < 1e-13
    for k in range(max(1, more)):
        k0 = first + k
        part = (torch.minimum(high, k0 + 1) - torch.maximum(low, k0)).clamp_min(0.0) / torch.where(flat, 1.0, width)
        part = torch.where(flat, torch.full_like(part, 1.0 if k == 0 else 0.0), part)
        part = torch.where((k0 >= 0) & (k0 < c["nz"]), part, torch.zeros_like(part))
        yield k0.clamp(0, c["nz"] - 1).long() * plane + cell[None], part * (t1 - t0)[None] * length[:, :, None]


def _project64(c, x):
    y = torch.zeros(c["views"], c["nv"], c["nu"], device="cuda", dtype=torch.float64)
    flat = x.double().reshape(-1)
    for a in range(c["views"]):
        for idx, w in _chords(c, a):
            y[a] += (flat[idx] * w).sum(-1)
    return y


def _adjoint64(c, r):
    x = torch.zeros(c["nz"] * c["ny"] * c["nx"], device="cuda", dtype=torch.float64)
    r = r.double()
    for a in range(c["views"]):
        for idx, w in _chords(c, a):
            x.index_add_(0, idx.reshape(-1), (w * r[a][:, :, None]).reshape(-1))
    return x.reshape(c["nz"], c["ny"], c["nx"])


def _mix(z):
    z &= (1 << 64) - 1
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & ((1 << 64) - 1)
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & ((1 << 64) - 1)
    return z ^ (z >> 31)


def _drawn(seed, it, lane, n, k):
    """k of n blocks at iteration it: SplitMix64 counters, partial Fisher-Yates."""
    perm = list(range(n))
    for t in range(k):
        u = (_mix(seed + ((it << 20) + lane + t + 1) * 0x9E3779B97F4A7C15) >> 11) / 9007199254740992.0
        j = t + int(u * (n - t))
        perm[t], perm[j] = perm[j], perm[t]
    return sorted(perm[:k])


def _solve64(c, y, seed, iters):
    """BSGD in FP64 with an explicit sparse matrix: uniform pairs, whole views."""
    rows, cols, vals = [], [], []
    ray = torch.arange(c["nv"] * c["nu"], device="cuda").reshape(c["nv"], c["nu"], 1)
    for a in range(c["views"]):
        for idx, w in _chords(c, a):
            m = w > 0
            rows.append((a * c["nv"] * c["nu"] + ray).expand_as(w)[m])
            cols.append(idx[m])
            vals.append(w[m])
    R, C = c["views"] * c["nv"] * c["nu"], c["nx"] * c["ny"] * c["nz"]
    rows, cols, vals = torch.cat(rows), torch.cat(cols), torch.cat(vals)
    planes, size = (c["nz"], c["nx"] * c["ny"]) if c["nz"] > 1 else (c["ny"], c["nx"])
    cut = [j * planes // c["N"] * size for j in range(c["N"] + 1)]
    view_of = torch.arange(R, device="cuda") // (c["nv"] * c["nu"])
    y = y.double().reshape(-1)
    x, g = torch.zeros(C, device="cuda", dtype=torch.float64), torch.zeros(C, device="cuda", dtype=torch.float64)
    z = torch.zeros(c["N"], R, device="cuda", dtype=torch.float64)
    snap, r, mu = torch.zeros_like(z), y.clone(), _step_size(c)
    parts = []
    for j in range(c["N"]):
        m = (cols >= cut[j]) & (cols < cut[j + 1])
        A = torch.sparse_coo_tensor(torch.stack([rows[m], cols[m] - cut[j]]), vals[m],
                                    (R, cut[j + 1] - cut[j])).coalesce()
        parts.append((A.to_sparse_csr(), A.t().coalesce().to_sparse_csr()))
    for it in range(iters):
        I, J = _drawn(seed, it, 0, c["M"], c["kM"]), _drawn(seed, it, 256, c["N"], c["kN"])
        on = torch.zeros(R, device="cuda", dtype=torch.bool)
        for i in I:
            on |= view_of % c["M"] == i
        for j in J:
            z[j] = torch.where(on, parts[j][0] @ x[cut[j]:cut[j + 1]], z[j])
        r = torch.where(on, y - z.sum(0), r)
        for j in J:
            w = torch.where(on, r - snap[j], torch.zeros_like(r))
            snap[j] = torch.where(on, r, snap[j])
            g[cut[j]:cut[j + 1]] += parts[j][1] @ w
            x[cut[j]:cut[j + 1]] += mu * g[cut[j]:cut[j + 1]]
    return x.reshape(c["nz"], c["ny"], c["nx"])


def exact(case, seed):
    c = case
    pieces = c["views"] * c["nv"] * c["nu"] * (c["nx"] + c["ny"])   # of one scan, at most
    blobs = _blobs(c, seed)
    if c["op"] == "forward":
        return _project64(c, _volume(c, blobs).to(_TORCH[c["storage"]])) if pieces < 2e10 else None
    if c["op"] == "backward":
        return _adjoint64(c, _scan(c, blobs, seed).to(_TORCH[c["storage"]])) if pieces < 2e10 else None
    if c["op"] == "train":
        if c["batch"] * pieces > 1e10:
            return None
        ys, grads = [], []
        for k in range(c["batch"]):
            ys.append(_project64(c, _volume(c, _blobs(c, seed + 100 + k))))
            grads.append(_adjoint64(c, ys[-1] - _scan(c, _blobs(c, seed + k), seed + k)))
        return {"y": torch.stack(ys), "grad": torch.stack(grads)}
    if c["op"] not in ("solve", "step") or c["storage"] != "f32" or c["pairs"] != "uniform" or \
            c["cells"] != "none" or c["tv"] or pieces > 6e7:
        return None
    iters = c["iters"] if c["op"] == "step" else c["epochs"] * round(c["M"] * c["N"] / (c["kM"] * c["kN"]))
    x = _solve64(c, _scan(c, blobs, seed), seed, iters)
    return {"x": x, "updates": None} if c["op"] == "solve" else x
