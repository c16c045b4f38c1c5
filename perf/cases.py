"""The work that a user of the package has it do, as cases to be timed.

``listed()`` gives the cases, ``draw()`` further ones of the same ranges, ``prepare()`` what a program has in hand before
the call (maps on the GPU, predicted capsules, spheres, network state, kept workspaces), ``run()`` one pass through the
public entry points, ``work()`` the bytes and operations that pass cannot do without, and ``exact()`` the results in
64 bits by plain torch.  Every input follows from the seed alone.
"""
import math

import numpy as np
import torch

import paper_2201_05058_gb300 as pcdf

INF = 2 ** 31 - 1   # "no voxel of the other state" in the int32 fields
EPS = 0.2           # hinge distance (m)
BAND = 0.05         # exact-fallback band of the learned surrogate (m)
WIDTH, COLS, FEATURES = 256, 16, 13            # the surrogate network: 16 -> 256 -> 256 -> 256 -> 1, 13 columns in use
PARAMS = WIDTH * COLS + 2 * WIDTH * WIDTH + 4 * WIDTH + 1
PARAMS_PAD = -(-PARAMS // 4) * 4
DEV = "cuda"


def listed():
    return [
        # a manipulator's work cell, 64^3 voxels of 5 cm: the smallest map that is mapped anew; launches and latency count
        dict(name="field_small", kind="field", nx=64, ny=64, nz=64, boxes=10, noise=0.0),
        # the room-scale static map: 256^3 voxels of 4 cm with 60 boxes
        dict(name="field_large", kind="field", nx=256, ny=256, nz=256, boxes=60, noise=0.0),
        # a cropped sensor map: odd sizes, and speckle among the boxes
        dict(name="field_ragged", kind="field", nx=317, ny=211, nz=97, boxes=40, noise=0.002),
        # the headline map update: static field and the fields of 20 predicted time steps, 3 walking humans
        dict(name="update_large", kind="update", nx=256, ny=256, nz=256, boxes=60, T=20, H=3, cylinder=False),
        # a smaller update on odd sizes: 4 humans as the paper's cylinders, a short horizon
        dict(name="update_ragged", kind="update", nx=161, ny=115, nz=83, boxes=30, T=9, H=4, cylinder=True),
        # many planners' maps at once: environments of uneven size, horizon and number of humans in one batch
        dict(name="batch", kind="batch", envs=16, lo=64, hi=320, zhi=128, tmax=30),
        # one configuration checked: 1,024 body spheres on one field
        dict(name="cost_small", kind="cost", nx=64, ny=64, nz=64, T=1, traj=1, states=1, spheres=1024, grad=False),
        # a trajectory optimiser's iteration: hinge costs and their gradients along 256 trajectories, 20 fields
        dict(name="cost_grad", kind="cost", nx=64, ny=64, nz=64, T=20, traj=256, states=40, spheres=30, grad=True),
        # a planner's step with the learned surrogate: 1,024,000 spheres in a 12.8 x 12.8 x 3.2 m room, 3 humans
        dict(name="plan_step", kind="plan", nx=256, ny=256, nz=64, boxes=160, T=20, H=3, traj=1024, states=40, spheres=25),
        # one step of the surrogate's training at the batch that it is trained with
        dict(name="train_step", kind="train", rows=262144),
        # the network alone over a planner's queries
        dict(name="network", kind="infer", rows=1024000),
        # clean-up of a new map and the prediction module's 2-D distance map
        dict(name="map_cleanup", kind="cleanup", nx=256, ny=256, nz=256, boxes=60, noise=0.005),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(hi, zhi, most):
        while True:
            nx, ny, nz = log(32, hi), log(32, hi), log(32, zhi)
            if nx * ny * nz <= most:
                return nx, ny, nz

    kind = rng.choice(["field", "field", "update", "update", "batch", "cost", "cost", "plan", "train", "infer", "cleanup"])
    if kind in ("field", "cleanup"):
        nx, ny, nz = box(512, 320, 256 ** 3)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, boxes=rng.randint(5, 60), noise=rng.choice([0.0, 0.002, 0.005]))
    if kind == "update":
        nx, ny, nz = box(320, 256, 200 ** 3)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, boxes=rng.randint(5, 60), T=rng.randint(1, 20), H=rng.randint(1, 4),
                    cylinder=rng.random() < 0.3)
    if kind == "batch":
        lo = rng.randint(48, 128)
        return dict(kind=kind, envs=rng.randint(2, 12), lo=lo, hi=rng.randint(lo + 8, 320), zhi=rng.randint(lo + 4, 140), tmax=rng.randint(6, 30))
    if kind == "cost":
        n = log(48, 96)
        return dict(kind=kind, nx=n, ny=log(48, 96), nz=log(48, 96), T=rng.randint(1, 20), traj=log(1, 256), states=rng.randint(1, 40),
                    spheres=rng.randint(10, 30), grad=rng.random() < 0.6)
    if kind == "plan":
        nx, ny, nz = box(256, 96, 256 * 256 * 64)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, boxes=rng.randint(10, 120), T=rng.randint(5, 20), H=rng.randint(1, 3), traj=log(32, 1024),
                    states=rng.randint(10, 40), spheres=rng.randint(10, 25))
    if kind == "train":
        return dict(kind=kind, rows=log(8192, 262144))
    return dict(kind=kind, rows=log(16000, 1024000))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _boxes_map(rng, shape_xyz, vox, boxes, noise=0.0):
    """uint8 [nz, ny, nx]: boxes of 0.1 to 0.8 m per axis, centres uniform, then speckle."""
    ext = np.array(shape_xyz) * vox
    occ = np.zeros(shape_xyz[::-1], np.uint8)
    for _ in range(boxes):
        c, s = rng.uniform(0, 1, 3) * ext, rng.uniform(0.1, 0.8, 3)
        a = [max(0, math.ceil((c[k] - s[k] / 2) / vox - 0.5)) for k in range(3)]
        b = [min(shape_xyz[k], math.floor((c[k] + s[k] / 2) / vox - 0.5) + 1) for k in range(3)]
        occ[a[2]:b[2], a[1]:b[1], a[0]:b[0]] = 1
    if noise:
        occ |= (rng.random(occ.shape, np.float32) < noise).view(np.uint8)
    return torch.from_numpy(occ).to(DEV)


def _walk(rng, grid, T, H, cylinder=False):
    """int32 [T][H][7]: upright humans of 1.8 m and 0.25 m radius walking four-waypoint paths at 1.2 m/s, 0.1 s a step; as
    cylinders their radius grows by 5 mm a step."""
    ext, r, h = np.array([grid.nx, grid.ny]) * grid.vox, 0.25, 1.8
    xy = np.zeros((T, H, 2))
    for k in range(H):
        way = r + grid.vox + rng.uniform(0, 1, (4, 2)) * (ext - 2 * (r + grid.vox))
        at = np.concatenate([[0.0], np.cumsum(np.linalg.norm(np.diff(way, axis=0), axis=1))])
        s = np.minimum(0.12 * np.arange(T), at[-1])
        xy[:, k] = np.stack([np.interp(s, at, way[:, j]) for j in range(2)], -1)
    z = np.zeros((T, H, 1))
    rad = np.full((T, H), r) + (0.005 * np.arange(T)[:, None] if cylinder else 0.0)
    lo, hi = (0.0, h) if cylinder else (r, h - r)
    return pcdf.capsule_fixed(np.concatenate([xy, z + lo], -1), np.concatenate([xy, z + hi], -1), rad, grid, cylinder=cylinder)


def _spheres(rng, grid, c):
    """Body spheres of 5 to 15 cm about straight-line trajectories, and the field that each state reads."""
    ext = np.array([grid.nx, grid.ny, grid.nz]) * grid.vox
    a, b = (rng.uniform(0.1, 0.9, (c["traj"], 1, 3)) * ext for _ in range(2))
    s = np.linspace(0, 1, c["states"]).reshape(1, -1, 1)
    p = (a + s * (b - a))[:, :, None] + rng.normal(0, 0.1, (c["traj"], c["states"], c["spheres"], 3))
    if c["traj"] == 1:
        p = rng.uniform(0, 1, p.shape) * ext
    r = rng.uniform(0.05, 0.15, p.shape[:3] + (1,))
    sph = torch.from_numpy(np.concatenate([p, r], -1).astype(np.float32)).to(DEV)
    t = np.broadcast_to(np.minimum(np.arange(c["states"]), c["T"] - 1).reshape(1, -1, 1), p.shape[:3]).astype(np.int32)
    return sph, torch.from_numpy(t.copy()).to(DEV)


def _batch_sizes(c):
    """The sizes are the case's, whatever the seed: (voxels per axis, horizon, humans) of each environment."""
    rng, out = np.random.default_rng([c[k] for k in ("envs", "lo", "hi", "zhi", "tmax")]), []
    for _ in range(c["envs"]):
        n = [int(rng.integers(c["lo"], m + 1)) for m in (c["hi"], c["hi"], max(c["zhi"], c["lo"]))]
        out.append((n, int(rng.integers(5, c["tmax"] + 1)), int(rng.integers(1, 5))))
    return out


def _weights(rng):
    """FP32 parameters of a network of the surrogate's shape (W1, b1, W2, b2, W3, b3, w4, b4), as a training run holds them."""
    out = []
    for rows, cols, used in ((WIDTH, COLS, FEATURES), (WIDTH, WIDTH, WIDTH), (WIDTH, WIDTH, WIDTH), (1, WIDTH, WIDTH)):
        w = rng.normal(0, math.sqrt(2.0 / used), (rows, cols))
        w[:, used:] = 0
        out += [w * (0.05 if rows == 1 else 1.0), rng.normal(0, 0.05, rows)]
    return [a.astype(np.float32) for a in out]


def _network_case(c, seed):
    """Parameters, feature rows (BF16 [M][16]) and targets: heights, times, offsets to the capsule's ends, radius, distance."""
    rng = np.random.default_rng([seed, 11])
    w = _weights(rng)
    g = torch.Generator(DEV).manual_seed(1000 + seed)
    M = c["rows"]
    p = torch.rand(M, 3, device=DEV, generator=g) * 3.2
    a = torch.rand(M, 3, device=DEV, generator=g) * 3.2
    a[:, 2] = 0.25
    b = a + torch.tensor([0.0, 0.0, 1.3], device=DEV)
    t = torch.randint(0, 20, (M, 1), device=DEV, generator=g) / 9.5 - 1
    s = ((p[:, 2:] - 0.25) / 1.3).clamp(0, 1)
    d = (p - (a + s * (b - a))).norm(dim=1, keepdim=True) - 0.25
    zero = torch.zeros(M, 2, device=DEV)
    x = torch.cat([zero, p[:, 2:] / 2, t, (p - a) / 2, (p - b) / 2, torch.full_like(t, 0.125), d / 2, s], 1)
    x = torch.nn.functional.pad(x, (0, COLS - FEATURES)).bfloat16().contiguous()
    target = (0.03 * torch.sin(7 * d[:, 0]) + 0.01 * torch.randn(M, device=DEV, generator=g)).contiguous()
    return w, x, target


def _network(w):
    """A network that holds these parameters, some way into its training (second moments filled)."""
    net = pcdf.SurrogateMLP(DEV, seed=0)
    v = net.state[:16 * PARAMS_PAD].view(torch.float32).view(4, PARAMS_PAD)
    v.zero_()
    v[0, :PARAMS] = torch.from_numpy(np.concatenate([a.ravel() for a in w])).to(DEV)
    net.adam(0.0)       # brings the network's working copies of the weights up to date
    v[1].zero_()
    v[2].fill_(1e-4)
    net.step = 100
    return net


def _grid(c, vox):
    return pcdf.Grid(c["nx"], c["ny"], c["nz"], vox)


def _vox(c):
    return 0.05 if c["kind"] in ("cost", "plan") or c["nx"] * c["ny"] * c["nz"] <= 64 ** 3 else 0.04


def prepare(case, seed):
    c, kind = case, case["kind"]
    rng = np.random.default_rng(seed)
    s = dict(case=c)
    if kind in ("field", "update", "cleanup", "plan"):
        g = s["grid"] = _grid(c, _vox(c))
        s["occ"] = _boxes_map(rng, (g.nx, g.ny, g.nz), g.vox, c["boxes"], c.get("noise", 0.0))
    if kind == "update":
        s["caps"] = _walk(rng, g, c["T"], c["H"], c["cylinder"])
        s["ws"] = pcdf.update_workspace(g, s["caps"], s["occ"].device)
        s["out"] = dict(out_static_sq=torch.empty(g.shape, dtype=torch.int32, device=DEV), out_static_sdf=torch.empty(g.shape, device=DEV),
                        out_sq=torch.empty((c["T"],) + g.shape, dtype=torch.int32, device=DEV),
                        out_sdf=torch.empty((c["T"],) + g.shape, device=DEV))
    elif kind == "batch":
        s["envs"] = []
        for n, T, H in _batch_sizes(c):
            g = pcdf.Grid(*n, 0.04)
            occ = _boxes_map(rng, n, g.vox, math.ceil(60 * n[0] * n[1] * n[2] / 256 ** 3))
            s["envs"].append((g, occ, _walk(rng, g, T, H)))
        s["batch"] = pcdf.Batch(s["envs"])
    elif kind == "cost":
        g = s["grid"] = _grid(c, _vox(c))
        occ = _boxes_map(rng, (g.nx, g.ny, g.nz), g.vox, 10)
        s["sdf"] = pcdf.predicted_fields(occ, g, _walk(rng, g, c["T"], 1))[3]
        s["sph"], s["tidx"] = _spheres(rng, g, c)
        if c["grad"]:
            s["c"] = s["sph"][..., :3].clone().requires_grad_(True)
            s["r"] = s["sph"][..., 3].clone().requires_grad_(True)
            s["up"] = torch.from_numpy(rng.uniform(0.5, 1.5, tuple(s["tidx"].shape)).astype(np.float32)).to(DEV)
    elif kind == "plan":
        s["caps"] = _walk(rng, g, c["T"], c["H"])
        s["caps_dev"] = torch.from_numpy(s["caps"]).to(DEV)
        s["sq"], s["sdf"] = pcdf.build_static_sdf(s["occ"], g)
        s["sph"], s["tidx"] = _spheres(rng, g, c)
        s["ws"] = pcdf.composite_workspace(g, s["caps"], s["occ"].device)
        s["net"] = _network(_weights(rng))
    elif kind in ("train", "infer"):
        w, s["x"], s["target"] = _network_case(c, seed)
        s["net"] = _network(w)
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "field":
        return pcdf.build_static_sdf(s["occ"], s["grid"])
    if kind == "update":
        return pcdf.predicted_fields(s["occ"], s["grid"], s["caps"], workspace=s["ws"], **s["out"])
    if kind == "batch":
        s["batch"].run()
        return s["batch"].comp_sq
    if kind == "cost":
        if not c["grad"]:
            return pcdf.query_cost(s["sdf"], s["grid"], s["sph"], s["tidx"], EPS)
        h = pcdf.hinge_cost(s["c"], s["r"], s["sdf"], s["tidx"], EPS, s["grid"])
        return (h.detach(),) + torch.autograd.grad(h, (s["c"], s["r"]), s["up"])
    if kind == "plan":
        return pcdf.surrogate_step(s["net"], s["grid"], s["sq"], s["sdf"], s["sph"], s["tidx"], s["caps"], EPS, BAND, s["ws"],
                                   caps_dev=s["caps_dev"])
    if kind == "train":
        y, loss = s["net"].backward(s["x"], s["target"])
        s["net"].adam(1e-4)
        v = s["net"].state[:16 * PARAMS_PAD].view(torch.float32).view(4, PARAMS_PAD)
        return dict(y=y, loss=loss, params=v[0, :PARAMS], grad=v[3, :PARAMS])
    if kind == "infer":
        return s["net"].infer_tc(s["x"])
    clean = pcdf.filter_voxels(s["occ"], s["grid"])
    z1 = min(s["grid"].nz, round(1.8 / s["grid"].vox))
    return (clean,) + pcdf.edt_2d(clean, s["grid"], 0, z1)


def work(case):
    c, kind = case, case["kind"]
    if kind == "batch":
        b = 0
        for n, T, H in _batch_sizes(c):
            b += n[0] * n[1] * n[2] * (1 + 4 * T)
        return {"bytes": b, "flops": 0}
    if kind in ("train", "infer"):
        macs = WIDTH * COLS + 2 * WIDTH * WIDTH + WIDTH
        if kind == "infer":
            return {"bytes": c["rows"] * (2 * COLS + 4) + 4 * PARAMS, "flops": 2 * macs * c["rows"]}
        return {"bytes": c["rows"] * (2 * COLS + 8) + 4 * PARAMS * 7, "flops": (6 * macs - 2 * WIDTH * COLS) * c["rows"]}
    V = c["nx"] * c["ny"] * c["nz"]
    if kind == "field":
        return {"bytes": 9 * V, "flops": 0}
    if kind == "cleanup":
        return {"bytes": 2 * V + 8 * c["nx"] * c["ny"], "flops": 0}
    if kind == "update":
        return {"bytes": V * (9 + 8 * c["T"]), "flops": 0}
    n = c["traj"] * c["states"] * c["spheres"]
    if kind == "plan":   # spheres, time indices, cost and distance; the static pair once
        return {"bytes": n * (16 + 4 + 8) + 8 * V, "flops": 0}
    touched = min(4 * V * c["T"], 32 * n)
    return {"bytes": n * (16 + 4 + 4 + (20 if c["grad"] else 0)) + touched, "flops": 0}


# ---------------------------------------------------------------------------
# the results in 64 bits, by plain torch
# ---------------------------------------------------------------------------

FAR = 1 << 40


def _axis_min(g, dim):
    """min over j of g[.., j, ..] + (i - j)^2 along dim (int64)."""
    n = g.shape[dim]
    view = [1] * g.dim()
    view[dim] = n
    i = torch.arange(n, device=g.device).view(view)
    out = torch.full_like(g, FAR)
    for j in range(n):
        out = torch.minimum(out, g.narrow(dim, j, 1) + (i - j) ** 2)
    return out


def _edt(occ):
    """int64 signed squared distance to the nearest voxel of the other state; +-INF where there is none."""
    def to(sites):
        g = torch.where(sites, 0, FAR)
        for dim in range(occ.dim()):
            if occ.shape[dim] > 1:
                g = _axis_min(g, dim)
        return torch.where(g >= FAR, INF, g)
    o = occ != 0
    return torch.where(o, -to(~o), to(o))


def _metres(sq, vox):
    v = float(np.float32(vox))
    m = sq.double().abs().sqrt() * v
    m = torch.where(sq.abs() == INF, math.inf, m)
    return torch.where(sq < 0, -m, m)


def _inside(grid, caps):
    """bool [nz, ny, nx]: voxel centres in any of the primitives caps [H][7] (1/16-voxel fixed point)."""
    c = [16 * torch.arange(n, device=DEV) + 8 for n in (grid.nx, grid.ny, grid.nz)]
    p = (c[0].view(1, 1, -1), c[1].view(1, -1, 1), c[2].view(-1, 1, 1))
    out = torch.zeros(grid.shape, dtype=torch.bool, device=DEV)
    for q in caps.astype(np.int64).tolist():
        cyl, r2 = bool(q[6] & pcdf.CYLINDER), (q[6] & ~pcdf.CYLINDER) ** 2
        d = [q[3 + k] - q[k] for k in range(3)]
        L = sum(v * v for v in d)
        w = [p[k] - q[k] for k in range(3)]
        s, ww = sum(w[k] * d[k] for k in range(3)), sum(v * v for v in w)
        e = sum((p[k] - q[3 + k]) ** 2 for k in range(3))
        line = ww * L - s * s <= r2 * L
        if cyl:
            out |= (s >= 0) & (s <= L) & line
        else:
            out |= torch.where(s <= 0, ww <= r2, torch.where(s >= L, e <= r2, line))
    return out


def _composites(grid, occ, caps):
    """(int64 static, [int64 composite of each t])."""
    st = _edt(occ)
    return st, [torch.minimum(st, _edt(_inside(grid, caps[t]))) for t in range(caps.shape[0])]


def _trilinear(sdf, grid, c, tidx):
    """float64 field value at each centre, from the FP32 field that it reads."""
    t = tidx.reshape(-1).long().clamp(0, sdf.shape[0] - 1)
    lo, f = [], []
    for k, n in enumerate((grid.nx, grid.ny, grid.nz)):
        u = (c[..., k].reshape(-1) / float(np.float32(grid.vox)) - 0.5).clamp(0, n - 1)
        i = u.detach().floor().long().clamp(max=n - 2)
        lo.append(i)
        f.append(u - i)
    d = 0.0
    for corner in range(8):
        b = [(corner >> k) & 1 for k in range(3)]
        w = 1.0
        for k in range(3):
            w = w * (f[k] if b[k] else 1 - f[k])
        d = d + w * sdf[t, lo[2] + b[2], lo[1] + b[1], lo[0] + b[0]].double()
    return d.view(tidx.shape)


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "plan":
        return None   # a network's estimate for some spheres and an exact answer for others: there is no 64-bit value of the whole
    if kind in ("train", "infer"):
        w, x, target = _network_case(c, seed)
        p = [torch.from_numpy(a).to(DEV) for a in w]
        p = [(a.bfloat16() if a.dim() == 2 else a).double().requires_grad_(kind == "train") for a in p]
        ys, M = [], x.shape[0]
        for x_ in x.split(32768):
            h = x_.double()
            for k in range(3):
                h = torch.relu(h @ p[2 * k].T + p[2 * k + 1])
            y = (h @ p[6].T + p[7]).view(-1)
            if kind == "train":
                at = sum(v.numel() for v in ys)
                ((y - target[at:at + y.numel()].double()) ** 2).sum().div(M).backward()
            ys.append(y.detach())
        y = torch.cat(ys)
        if kind == "infer":
            return y
        g = torch.cat([a.grad.reshape(-1) for a in p])
        b1, b2, step = 0.9, 0.999, 101
        m, v = (1 - b1) * g / (1 - b1 ** step), (b2 * float(np.float32(1e-4)) + (1 - b2) * g * g) / (1 - b2 ** step)
        master = torch.from_numpy(np.concatenate([a.ravel() for a in w])).to(DEV).double()
        return dict(y=y, loss=((y - target.double()) ** 2).mean().view(1), params=master - 1e-4 * m / (v.sqrt() + 1e-8), grad=g)
    s = prepare(case, seed)
    if kind == "field":
        sq = _edt(s["occ"])
        return sq, _metres(sq, s["grid"].vox)
    if kind == "update":
        st, comp = _composites(s["grid"], s["occ"], s["caps"])
        comp = torch.stack(comp)
        return st, _metres(st, s["grid"].vox), comp, _metres(comp, s["grid"].vox)
    if kind == "batch":
        return [torch.stack(_composites(g, occ, caps)[1]) for g, occ, caps in s["envs"]]
    if kind == "cost":
        ctr = s["sph"][..., :3].double().requires_grad_(c["grad"])
        rad = s["sph"][..., 3].double().requires_grad_(c["grad"])
        h = torch.relu(float(np.float32(EPS)) + rad - _trilinear(s["sdf"], s["grid"], ctr, s["tidx"]))
        return h if not c["grad"] else (h.detach(),) + torch.autograd.grad(h, (ctr, rad), s["up"].double())
    occ = s["occ"] != 0
    n = torch.nn.functional.conv3d(occ.float()[None, None], torch.ones(1, 1, 3, 3, 3, device=DEV), padding=1)[0, 0] - occ.float()
    clean = (occ & (n >= 5)).to(torch.uint8)
    sq = _edt(clean[:min(s["grid"].nz, round(1.8 / s["grid"].vox))].amax(0))
    return clean, sq, _metres(sq, s["grid"].vox)
