"""The calls whose speed matters to a user of this library, as cases that can
be prepared, run, costed and checked.

Every case is one public call (or one reconstruction) on seeded synthetic
data: ellipsoid phantoms, their analytic cone-beam projections and 1 % noise,
on circular orbits like those of the repository's workloads (SOD 1000 mm, SDD
1500 mm, a detector 1.5 times the volume's edge in pixels).  Kinds:

  project      A_N x of a list of views (the forward operator alone)
  backproject  A_N^T y of a list of views, also added into a volume
  reconstruct  a solver made for the scan and run for one epoch of Algorithm 1
               from x = 0 (host loop or graph, plain or learned first step)
  batch        a kept batch of uneven volumes, one epoch of each from x = 0
  fdk          the analytic reconstruction of a list of views
  prox_tv      the TV regulariser's prox on one volume

listed() names the cases and draw() gives more of the same ranges.
"""
from __future__ import annotations

import math
import types

import numpy as np
import torch

import paper_2605_12085_gb300 as fbl

DEVICE = "cuda"
DTYPES = {"f32": (torch.float32, fbl.F32), "bf16": (torch.bfloat16, fbl.BF16), "f16": (torch.float16, fbl.F16)}
MAX_UNITS = 2.0e11       # voxel-views of the largest case
EXACT_FORWARD = 3.0e11   # voxel-views up to which exact() projects (seconds on the GPU)
EXACT_BACK = 3.0e10      # and backprojects


def _op(kind, n, sel, views, **kw):
    """An operator case: n the volume's edges, sel of views listed."""
    nx, ny, nz = n if isinstance(n, tuple) else (n, n, n)
    case = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "voxel": 1.0, "views": views, "sel": sel,
            "nu": math.ceil(1.5 * max(nx, ny)), "nv": math.ceil(1.5 * nz), "pixel": 1.5, "dtype": "f32", "tuned": False}
    case.update(kw)
    return case


def listed():
    return [
        # a mini-batch of the smallest workload: launches and latency, not arithmetic
        dict(_op("project", 64, 10, 90), name="project_64"),
        # a mini-batch of the 256^3 workload with 16-bit volume and projections, as a low-memory run keeps them
        dict(_op("project", 256, 20, 360, dtype="bf16"), name="project_256_bf16"),
        # the whole scan's forward projection at full size on a tuned geometry: the benchmark's forward half
        dict(_op("project", 512, 720, 720, tuned=True), name="project_512"),
        # a mini-batch gradient's backprojection at 256^3 with the launch a new geometry starts with
        dict(_op("backproject", 256, 20, 360), name="backproject_256"),
        # an odd-sized scan of few views in 16 bits, added into a volume that holds other views already
        dict(_op("backproject", (301, 257, 190), 31, 93, nu=449, nv=301, dtype="f16", accumulate=True),
             name="backproject_ragged_f16"),
        # the whole scan's backprojection at full size on a tuned geometry: the benchmark's other half
        dict(_op("backproject", 512, 720, 720, tuned=True), name="backproject_512"),
        # a small scan reconstructed for one epoch: many short iterations, the host in the loop
        dict(_op("reconstruct", 64, 10, 90, graph=False, learned=False), name="reconstruct_64"),
        # the production setting: 16-bit storage, learned first step, one graph per iteration
        dict(_op("reconstruct", 256, 20, 360, dtype="bf16", graph=True, learned=True), name="reconstruct_256_learned"),
        # the paper's sparse scan in shape: 560^3, 36 views, 8-view mini-batches, plain line search in FP32
        dict(_op("reconstruct", 560, 8, 36, graph=False, learned=False), name="reconstruct_560"),
        # sixteen small uneven volumes at once, where one volume alone cannot fill the GPU
        {"kind": "batch", "volumes": 16, "edge_lo": 24, "edge_hi": 80, "views_lo": 30, "views_hi": 120, "dtype": "f32",
         "name": "batch_16"},
        # the analytic reconstruction of the whole 256^3 scan (a starting point or a reference volume)
        dict(_op("fdk", 256, 360, 360), name="fdk_256"),
        # the TV regulariser's prox as one trial of a line search calls it
        {"kind": "prox_tv", "nx": 256, "ny": 256, "nz": 256, "lam": 0.05, "iters": 20, "x_max": None, "name": "prox_tv_256"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["project", "project", "backproject", "backproject", "reconstruct", "reconstruct", "batch", "fdk", "prox_tv"])
    if kind == "batch":
        lo = rng.randint(20, 40)
        return {"kind": kind, "volumes": rng.randint(3, 20), "edge_lo": lo, "edge_hi": rng.randint(lo + 8, 96), "views_lo": rng.randint(24, 40),
                "views_hi": rng.randint(60, 130), "dtype": rng.choice(["f32", "f32", "bf16", "f16"])}
    if kind == "prox_tv":
        return {"kind": kind, "nx": _log_int(rng, 40, 320), "ny": _log_int(rng, 40, 320), "nz": _log_int(rng, 40, 320),
                "lam": round(rng.uniform(0.01, 0.2), 3), "iters": rng.randint(5, 30), "x_max": rng.choice([None, 1.0])}
    edge = {"project": 512, "backproject": 512, "reconstruct": 384, "fdk": 384}[kind]
    n0 = _log_int(rng, 48, edge)
    n = tuple(max(24, int(n0 * rng.uniform(0.7, 1.0))) for _ in range(3)) if rng.random() < 0.6 else (n0, n0, n0)
    views = _log_int(rng, 24, 720)
    sel = views if kind == "fdk" else min(views, _log_int(rng, 4, 64))
    if kind in ("project", "backproject") and rng.random() < 0.2:
        sel = views
    if kind == "reconstruct":  # one epoch of at most 24 iterations
        sel = max(sel, 4, -(-views // 24))
    vox = n[0] * n[1] * n[2]
    budget = MAX_UNITS / (40 if kind == "reconstruct" else 4 if kind == "fdk" else 1) * 0.45
    if kind in ("reconstruct", "fdk"):
        while vox * views > budget:
            views = max(8, views // 2)
            sel = views if kind == "fdk" else max(4, min(sel, views))
    case = _op(kind, n, sel, views, dtype=rng.choice(["f32", "f32", "bf16", "f16"]), tuned=rng.random() < 0.3)
    case["voxel"] = rng.choice([1.0, 1.0, 0.5, 0.8])
    if kind == "fdk":
        case["tuned"] = False
    case["pixel"] = round(1.5 * case["voxel"] * rng.choice([1.0, 1.0, 0.9, 1.2]), 3)
    case["nu"] = max(32, int(case["nu"] * rng.uniform(0.8, 1.05)))
    case["nv"] = max(24, int(case["nv"] * rng.uniform(0.8, 1.05)))
    if kind == "backproject":
        case["accumulate"] = rng.random() < 0.3
    if kind == "reconstruct":
        case["graph"] = rng.random() < 0.5
        case["learned"] = rng.random() < 0.4
    return case


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _geom(case):
    return types.SimpleNamespace(nx=case["nx"], ny=case["ny"], nz=case["nz"], vx=case["voxel"], vy=case["voxel"], vz=case["voxel"],
                                 n_views=case["views"], sod=1000.0, sdd=1500.0, nu=case["nu"], nv=case["nv"], du=case["pixel"],
                                 dv=case["pixel"], angles=None)


def _batch_geoms(case):
    out, nv = [], case["volumes"]
    for i in range(nv):
        t = i / max(1, nv - 1)
        n = round(case["edge_lo"] + (case["edge_hi"] - case["edge_lo"]) * t)
        views = round(case["views_lo"] + (case["views_hi"] - case["views_lo"]) * t)
        det = math.ceil(1.5 * n)
        out.append(_geom({"nx": n, "ny": n, "nz": n, "voxel": 1.0, "views": views, "nu": det, "nv": det, "pixel": 1.5}))
    return out


def _ellipsoids(g, seed, count=12):
    """(centre, semi-axes, rotation, value): a background and `count` features, all of positive value."""
    rng = np.random.default_rng(seed)
    half = 0.5 * np.array([g.nx * g.vx, g.ny * g.vy, g.nz * g.vz])
    h = float(half.min())
    out = [(np.zeros(3), 0.85 * half, np.eye(3), 0.3)]
    for _ in range(count):
        c = rng.normal(size=3)
        c *= 0.5 * h * rng.uniform() ** (1 / 3) / np.linalg.norm(c)
        q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
        out.append((c, rng.uniform(0.05, 0.3, 3) * h, q, float(rng.uniform(0.02, 0.2))))
    return out


def _phantom(g, ells):
    z, y, x = (torch.arange(n, device=DEVICE, dtype=torch.float32) for n in (g.nz, g.ny, g.nx))
    x, y, z = ((x - 0.5 * (g.nx - 1)) * g.vx)[None, None], ((y - 0.5 * (g.ny - 1)) * g.vy)[None, :, None], ((z - 0.5 * (g.nz - 1)) * g.vz)[:, None, None]
    vol = torch.zeros((g.nz, g.ny, g.nx), device=DEVICE)
    for c, a, R, val in ells:
        r = 0.0
        for k in range(3):
            r = r + (((x - c[0]) * R[0, k] + (y - c[1]) * R[1, k] + (z - c[2]) * R[2, k]) / a[k]) ** 2
        vol += val * (r <= 1.0)
    return vol


def _angle(g, v):
    return 2.0 * math.pi * v / g.n_views


def _data(g, ells, views, seed, dtype):
    """Line integrals through the ellipsoids plus Gaussian noise of 1 % of the maximum, [view][nv][nu]."""
    u = (torch.arange(g.nu, device=DEVICE, dtype=torch.float32) - 0.5 * (g.nu - 1)) * g.du
    w = ((torch.arange(g.nv, device=DEVICE, dtype=torch.float32) - 0.5 * (g.nv - 1)) * g.dv)[:, None]
    out = torch.empty((len(views), g.nv, g.nu), device=DEVICE)
    for s, v in enumerate(views):
        c, sn = math.cos(_angle(g, v)), math.sin(_angle(g, v))
        src = np.array([g.sod * c, g.sod * sn, 0.0])
        d = [(-g.sdd * c - u * sn)[None, :].expand(g.nv, g.nu), (-g.sdd * sn + u * c)[None, :].expand(g.nv, g.nu), w.expand(g.nv, g.nu)]
        length = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
        acc = torch.zeros((g.nv, g.nu), device=DEVICE)
        for ctr, a, R, val in ells:
            o = (src - ctr) @ R / a
            e = [sum(d[i] * (float(R[i, k]) / float(a[k])) for i in range(3)) for k in range(3)]
            A = e[0] ** 2 + e[1] ** 2 + e[2] ** 2
            B = sum(float(o[k]) * e[k] for k in range(3))
            disc = B * B - A * (float(o @ o) - 1.0)
            acc += val * 2.0 * torch.sqrt(disc.clamp_min(0.0)) / A * length
        out[s] = acc
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    out += (0.01 * out.max()) * torch.randn(out.shape, device=DEVICE, generator=gen)
    return out.to(dtype)


def _selected(case, seed):
    """The views of the call: all in order, or a random sample without repetition."""
    if case["sel"] >= case["views"]:
        return list(range(case["views"]))
    return [int(v) for v in np.random.default_rng(seed + 7).permutation(case["views"])[:case["sel"]]]


def _params(g, n0, seed, case):
    code = DTYPES[case["dtype"]][1]
    return fbl.params_default(N0=n0, seed=seed, x_dtype=code, b_dtype=code, use_graph=int(case.get("graph", False)))


def _host_inputs(case, seed):
    """The input tensors of a case, from the seed alone."""
    kind = case["kind"]
    if kind == "prox_tv":
        g = _geom(dict(case, voxel=1.0, views=1, nu=1, nv=1, pixel=1.0))
        gen = torch.Generator(device=DEVICE).manual_seed(seed)
        v = _phantom(g, _ellipsoids(g, seed))
        return {"v": v + 0.05 * torch.randn(v.shape, device=DEVICE, generator=gen)}
    if kind == "batch":
        gs = _batch_geoms(case)
        return {"gs": gs, "bs": [_data(g, _ellipsoids(g, seed + 31 * i, 6), range(g.n_views), seed + i, DTYPES[case["dtype"]][0])
                                 for i, g in enumerate(gs)]}
    g, dt = _geom(case), DTYPES[case["dtype"]][0]
    ells = _ellipsoids(g, seed)
    if kind == "project":
        return {"g": g, "views": _selected(case, seed), "x": _phantom(g, ells).to(dt)}
    if kind == "reconstruct":
        return {"g": g, "b": _data(g, ells, range(g.n_views), seed, dt)}
    views = _selected(case, seed)
    out = {"g": g, "views": views, "y": _data(g, ells, views, seed, dt)}
    if case.get("accumulate"):
        out["x0"] = 100.0 * _phantom(g, ells)
    return out


def prepare(case, seed):
    s = dict(_host_inputs(case, seed), case=case, seed=seed)
    kind = case["kind"]
    if kind == "batch":
        s["G"] = [fbl.geometry_create(g) for g in s["gs"]]
        ps = [_params(g, -(-g.n_views // 12), seed + i, case) for i, g in enumerate(s["gs"])]
        s["batch"] = fbl.fblisa_batch_create(s["G"], ps)
        s["xs"] = [torch.zeros((g.nz, g.ny, g.nx), device=DEVICE, dtype=DTYPES[case["dtype"]][0]) for g in s["gs"]]
    elif kind != "prox_tv":
        s["G"] = fbl.geometry_create(s["g"])
        if case["tuned"]:
            fbl.geometry_autotune(s["G"], DTYPES[case["dtype"]][1] if kind != "backproject" else fbl.F32, min(case["sel"], 40))
        if case.get("learned"):
            from paper_2605_12085_gb300 import proposal
            s["net"], _ = proposal.load()
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "project":
        return fbl.project(s["G"], s["x"], s["views"], y_dtype=DTYPES[case["dtype"]][1])
    if kind == "backproject":
        if case.get("accumulate"):
            return fbl.backproject(s["G"], s["y"], s["views"], x=s["x0"].clone(), accumulate=True)
        return fbl.backproject(s["G"], s["y"], s["views"])
    if kind == "fdk":
        return fbl.fdk(s["G"], s["y"], s["views"])
    if kind == "prox_tv":
        return fbl.prox_tv(s["v"], case["lam"], case["iters"], x_max=math.inf if case["x_max"] is None else case["x_max"])
    if kind == "reconstruct":
        g = s["g"]
        S = fbl.fblisa_create(s["G"], _params(g, case["sel"], s["seed"], case))
        if case["learned"]:
            S.set_proposal(s["net"])
        x = torch.zeros((g.nz, g.ny, g.nx), device=DEVICE, dtype=DTYPES[case["dtype"]][0])
        steps = S.run(x, s["b"], 1, trace_cap=g.n_views)
        return {"x": x, "f": torch.tensor([[t["f_x"], t["f_xbar"]] for t in steps]), "alpha": torch.tensor([t["alpha"] for t in steps]),
                "backtracks": torch.tensor([t["backtracks"] for t in steps])}
    for x in s["xs"]:
        x.zero_()
    steps = s["batch"].run(s["xs"], s["bs"], 12)
    return {"xs": s["xs"], "alpha": torch.tensor([[t["alpha"] for t in it] for it in steps])}


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def _samples(g, n_sel):
    """In-volume samples of n_sel views: ray density at the axis times the volume, capped by the detector."""
    mag = g.sdd / g.sod
    cover = min(1.0, g.nu * g.du / mag / (max(g.nx, g.ny) * g.vx)) * min(1.0, g.nv * g.dv / mag / (g.nz * g.vz))
    return n_sel * g.nx * g.ny * g.nz * (mag * g.vx / g.du) * (mag * g.vz / g.dv) * cover


def work(case):
    kind = case["kind"]
    if kind == "prox_tv":
        n = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": 8 * n, "flops": 40 * n * case["iters"]}
    es = 4 if case["dtype"] == "f32" else 2
    if kind == "batch":
        flops, size = 0.0, 0.0
        for g in _batch_geoms(case):
            n0 = -(-g.n_views // 12)
            flops += 12 * _samples(g, n0) * (10 + 16 + 10)
            size += g.nx * g.ny * g.nz * es + g.n_views * g.nu * g.nv * es
        return {"bytes": size, "flops": flops}
    g = _geom(case)
    n, rays = g.nx * g.ny * g.nz, case["sel"] * g.nu * g.nv
    smp = _samples(g, case["sel"])
    if kind == "project":
        return {"bytes": es * (n + rays), "flops": 10 * smp}
    if kind == "backproject":
        return {"bytes": es * rays + 4 * n * (2 if case.get("accumulate") else 1), "flops": 16 * smp}
    if kind == "fdk":
        return {"bytes": es * rays + 4 * n, "flops": 12.0 * n * case["sel"] + 2.0 * rays * 30}
    # one residual projection, one backprojection and one trial objective per iteration
    its = -(-case["views"] // case["sel"])
    return {"bytes": es * (n + case["views"] * g.nu * g.nv), "flops": its * smp * (10 + 16 + 10)}


# ---------------------------------------------------------------------------
# The same results in 64 bits
# ---------------------------------------------------------------------------
class _Joseph:
    """A and A^T of a geometry in float64: per view and detector column the dominant axis, the in-plane
    crossing q_b(m) = qb0 + m qb1 and the vertical scale Zc(m) = zc0 + m zc1 (q_z = w Zc + cz)."""

    def __init__(self, g):
        self.g = g
        self.w = (torch.arange(g.nv, device=DEVICE, dtype=torch.float64) - 0.5 * (g.nv - 1)) * g.dv
        self.tables = {}

    def table(self, v):
        if v not in self.tables:
            g = self.g
            c, sn = math.cos(_angle(g, v)), math.sin(_angle(g, v))
            u = (np.arange(g.nu) - 0.5 * (g.nu - 1)) * g.du
            off = g.sdd - g.sod
            d = np.stack([(-off * c - u * sn) - g.sod * c, (-off * sn + u * c) - g.sod * sn])
            fam = (np.abs(d[1]) > np.abs(d[0])).astype(int)
            got = []
            for f in (0, 1):
                iu = np.nonzero(fam == f)[0]
                if not iu.size:
                    continue
                V, N, src = (g.vx, g.vy), (g.nx, g.ny), (g.sod * c, g.sod * sn)
                da, db = d[f][iu], d[1 - f][iu]
                p0 = -0.5 * (N[f] - 1) * V[f] - src[f]
                t = [torch.from_numpy(np.ascontiguousarray(a)).to(DEVICE) for a in (
                    (src[1 - f] + p0 * db / da) / V[1 - f] + 0.5 * (N[1 - f] - 1), V[f] * db / (da * V[1 - f]), p0 / (da * g.vz), V[f] / (da * g.vz),
                    V[f] / np.abs(da), da * da + db * db)]
                got.append((f, torch.from_numpy(iu).to(DEVICE), t))
            self.tables[v] = got
        return self.tables[v]

    def planes(self, f, t, ms):
        """In-plane rows and vertical rows (clamped into one zero on either side) with their fractions."""
        g = self.g
        nb = (g.ny, g.nx)[f]
        m = ms[:, None].double()
        qb = (t[0] + m * t[1]).clamp(-1.0, float(nb))
        b0 = torch.floor(qb).clamp_max_(nb - 1)
        qz = ((t[2] + m * t[3])[:, :, None] * self.w + 0.5 * (g.nz - 1)).clamp_(-1.0, float(g.nz))
        k0 = torch.floor(qz).clamp_max_(g.nz - 1)
        return b0.long() + 1, qb - b0, k0.long() + 1, qz - k0

    def weight(self, t):
        return (t[4] * torch.sqrt(t[5] + (self.w * self.w)[:, None])).t()  # [iu][iv]

    def chunks(self, f, iu):
        na = (self.g.nx, self.g.ny)[f]
        step = max(1, 40_000_000 // (iu.numel() * max(self.g.nv, self.g.nz)))
        for m0 in range(0, na, step):
            yield torch.arange(m0, min(na, m0 + step), device=DEVICE)

    def forward(self, x, views):
        g = self.g
        x = x.double()
        # [plane][in-plane][k] with a zero on either side in-plane and along k
        vol = [torch.nn.functional.pad(p, (1, 1, 1, 1)) for p in (x.permute(2, 1, 0), x.permute(1, 2, 0))]
        out = torch.zeros((len(views), g.nv, g.nu), device=DEVICE, dtype=torch.float64)
        for s, v in enumerate(views):
            for f, iu, t in self.table(v):
                acc = torch.zeros((iu.numel(), g.nv), device=DEVICE, dtype=torch.float64)
                for ms in self.chunks(f, iu):
                    b0, fb, k0, fz = self.planes(f, t, ms)
                    P, fb = vol[f], fb[:, :, None]
                    L = P[ms[:, None], b0] * (1 - fb) + P[ms[:, None], b0 + 1] * fb
                    lo = torch.gather(L, 2, k0)
                    lo += fz * (torch.gather(L, 2, k0 + 1) - lo)
                    acc += lo.sum(0)
                out[s, :, iu] = (acc * self.weight(t)).t()
        return out

    def back(self, y, views):
        g = self.g
        vol = [torch.zeros((na * (nb + 2), g.nz + 2), device=DEVICE, dtype=torch.float64) for na, nb in ((g.nx, g.ny), (g.ny, g.nx))]
        for s, v in enumerate(views):
            for f, iu, t in self.table(v):
                r = y[s].double()[:, iu].t() * self.weight(t)
                nb2 = (g.ny, g.nx)[f] + 2
                for ms in self.chunks(f, iu):
                    b0, fb, k0, fz = self.planes(f, t, ms)
                    T = torch.zeros((ms.numel(), iu.numel(), g.nz + 2), device=DEVICE, dtype=torch.float64)
                    rf = r * fz
                    T.scatter_add_(2, k0 + 1, rf)
                    T.scatter_add_(2, k0, r - rf)
                    rows, T, fb = (ms[:, None] * nb2 + b0).reshape(-1), T.reshape(-1, g.nz + 2), fb.reshape(-1, 1)
                    vol[f].index_add_(0, rows, T * (1 - fb))
                    vol[f].index_add_(0, rows + 1, T * fb)
        a = vol[0].view(g.nx, g.ny + 2, g.nz + 2)[:, 1:-1, 1:-1].permute(2, 1, 0)
        b = vol[1].view(g.ny, g.nx + 2, g.nz + 2)[:, 1:-1, 1:-1].permute(2, 0, 1)
        return a + b


def _permutation(seed, epoch, n):
    """Algorithm 1's mini-batch permutation: Fisher-Yates on a SplitMix64 stream."""
    mask = (1 << 64) - 1
    state, perm = (seed ^ (epoch * 0xD1B54A32D192ED03)) & mask, list(range(n))
    for i in range(n - 1):
        z = (state + (i + 1) * 0x9E3779B97F4A7C15) & mask
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & mask
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
        z ^= z >> 31
        j = min(n - 1, i + int(math.floor((z >> 11) * (1.0 / 9007199254740992.0) * (n - i))))
        perm[i], perm[j] = perm[j], perm[i]
    return perm


def _fb_lisa(g, b, n0, seed, iterations):
    """`iterations` iterations of Algorithm 1 from x = 0 with the library's default parameters, in float64."""
    A = _Joseph(g)
    x = torch.zeros((g.nz, g.ny, g.nx), device=DEVICE, dtype=torch.float64)
    per, steps = -(-g.n_views // n0), []
    for k in range(iterations):
        perm, it = _permutation(seed, 1 + k // per, g.n_views), k % per
        views = [perm[q % g.n_views] for q in range(it * n0, it * n0 + n0)]
        bn, scale = b[views].double(), g.n_views / n0
        r = A.forward(x, views) - bn
        f = 0.5 * scale * float((r * r).sum())
        grad = scale * A.back(r, views)
        alpha, bt = 1e-3, 0
        while True:
            xb = (x - alpha * grad - alpha).clamp_min(0.0)
            d = xb - x
            rhs = f + float((grad * d).sum()) + float((d * d).sum()) / (2.0 * alpha)
            fb = 0.5 * scale * float(((A.forward(xb, views) - bn) ** 2).sum())
            if fb <= rhs or bt == 60:
                break
            alpha, bt = 0.5 * alpha, bt + 1
        x = xb
        steps.append((f, fb, alpha, bt))
    return x, steps


def _exact_fdk(g, y, views):
    m, t = g.sod / g.sdd, g.du * g.sod / g.sdd
    f64 = dict(device=DEVICE, dtype=torch.float64)
    cu, cv = 0.5 * (g.nu - 1), 0.5 * (g.nv - 1)
    a, b = (torch.arange(g.nu, **f64) - cu) * t, ((torch.arange(g.nv, **f64) - cv) * g.dv * m)[:, None]
    k = torch.arange(g.nu, **f64)
    h = torch.where(k % 2 == 1, -1.0 / (math.pi ** 2 * k.clamp_min(1) ** 2 * t * t), torch.zeros_like(k))
    h[0] = 1.0 / (4.0 * t * t)
    idx = (torch.arange(g.nu, device=DEVICE)[:, None] - torch.arange(g.nu, device=DEVICE)[None]).abs()
    ramp, weight = t * h[idx], g.sod / torch.sqrt(g.sod ** 2 + a * a + b * b)
    xs, ys, zs = ((torch.arange(n, **f64) - 0.5 * (n - 1)) * v for n, v in ((g.nx, g.vx), (g.ny, g.vy), (g.nz, g.vz)))
    out = torch.zeros((g.nz, g.ny, g.nx), **f64)
    order = sorted(range(len(views)), key=lambda q: _angle(g, views[q]))
    ang = [_angle(g, views[q]) for q in order]
    for p, q in enumerate(order):
        gap = 2.0 * math.pi if len(ang) == 1 else 0.5 * ((ang[(p + 1) % len(ang)] + (2 * math.pi if p + 1 == len(ang) else 0.0)) - (
            ang[p - 1] - (2 * math.pi if p == 0 else 0.0)))
        filt = torch.nn.functional.pad((y[q].double() * weight) @ ramp, (1, 2, 1, 2))
        c, s = math.cos(ang[p]), math.sin(ang[p])
        U = (g.sod - (xs[None] * c + ys[:, None] * s)) / g.sod
        fu = ((-xs[None] * s + ys[:, None] * c) / U / t + cu).clamp(-1.0, float(g.nu))
        fv = (zs[:, None, None] / U / (g.dv * m) + cv).clamp(-1.0, float(g.nv))
        u0, v0 = torch.floor(fu), torch.floor(fv)
        tu, tv, at = fu - u0, fv - v0, (v0.long() + 1) * filt.shape[1] + (u0.long() + 1)
        flat = filt.reshape(-1)
        lo = flat[at] * (1 - tu) + flat[at + 1] * tu
        hi = flat[at + filt.shape[1]] * (1 - tu) + flat[at + filt.shape[1] + 1] * tu
        out += (lo + tv * (hi - lo)) * (0.5 * gap / (U * U))
    return out


def _exact_tv(v, lam, iters, x_max):
    v = v.double()
    axes = (2, 1, 0)

    def grad(x):
        return [torch.cat([torch.diff(x, dim=a), torch.zeros_like(x.narrow(a, 0, 1))], dim=a) for a in axes]

    def primal(q):
        kt = torch.zeros_like(v)
        for c, a in zip(q, axes):
            kt -= c
            kt.narrow(a, 1, v.shape[a] - 1).add_(c.narrow(a, 0, v.shape[a] - 1))
        return (v - lam * kt).clamp(0.0, x_max)

    q = [torch.zeros_like(v) for _ in axes]
    r, t = q, 1.0
    for _ in range(iters):
        p = [a + b / (12.0 * lam) for a, b in zip(r, grad(primal(r)))]
        norm = torch.sqrt(p[0] ** 2 + p[1] ** 2 + p[2] ** 2).clamp_min(1.0)
        p = [a / norm for a in p]
        tn = 0.5 * (1.0 + math.sqrt(1.0 + 4.0 * t * t))
        r = [a + ((t - 1.0) / tn) * (a - b) for a, b in zip(p, q)]
        q, t = p, tn
    return primal(q)


def exact(case, seed):
    kind = case["kind"]
    if kind == "prox_tv":
        s = _host_inputs(case, seed)
        return _exact_tv(s["v"], case["lam"], case["iters"], math.inf if case["x_max"] is None else case["x_max"])
    if kind == "batch":
        if case["dtype"] != "f32":  # every iterate is rounded to its storage type
            return None
        s, xs, alpha = _host_inputs(case, seed), [], []
        for i, (g, b) in enumerate(zip(s["gs"], s["bs"])):
            x, steps = _fb_lisa(g, b, -(-g.n_views // 12), seed + i, 12)
            xs.append(x)
            alpha.append([st[2] for st in steps])
        return {"xs": xs, "alpha": torch.tensor(alpha, dtype=torch.float64).t()}
    units = float(case["nx"]) * case["ny"] * case["nz"] * case["sel"]
    if kind == "project":
        if units > EXACT_FORWARD:
            return None
        s = _host_inputs(case, seed)
        return _Joseph(s["g"]).forward(s["x"], s["views"])
    if kind == "backproject":
        if units > EXACT_BACK:
            return None
        s = _host_inputs(case, seed)
        x = _Joseph(s["g"]).back(s["y"], s["views"])
        return x + s["x0"].double() if case.get("accumulate") else x
    if kind == "fdk":
        if units > EXACT_BACK:
            return None
        s = _host_inputs(case, seed)
        return _exact_fdk(s["g"], s["y"], s["views"])
    its = -(-case["views"] // case["sel"])
    if case["learned"] or case["dtype"] != "f32" or 12 * its * units > EXACT_FORWARD or its * units > EXACT_BACK:
        return None
    s = _host_inputs(case, seed)
    x, steps = _fb_lisa(s["g"], s["b"], case["sel"], seed, its)
    return {"x": x, "f": torch.tensor([st[:2] for st in steps], dtype=torch.float64), "alpha": torch.tensor([st[2] for st in steps], dtype=torch.float64),
            "backtracks": torch.tensor([st[3] for st in steps])}
