"""Workloads of the cone-beam reconstruction library, for timing and comparison.

Each case is one call (or one batch of calls) a program makes through
paper_2211_14212_gb300.cbct: a projection A x, a backprojection A^T y, a whole
solve, or a batch of requests to the server.  Sizes are those of the
repository's benchmark configurations and tests, or lie between them.

Inputs are analytic: a volume of random ellipsoids sampled at voxel centres,
and projections that are the exact chord lengths through such ellipsoids plus
photon noise, both computed on the GPU with torch alone, so that they depend
on nothing but the seed.  `exact` traces the rays in FP64 with torch.
"""
import math
import random

import numpy as np
import torch

from paper_2211_14212_gb300 import cbct

DTYPES = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


def _case(name, op, n, nz, vox, nu, nv, pix, angles, arc, dso, dsd, dtype="f32", **more):
    """n x n x nz voxels of vox (mm), nu x nv pixels of pix (mm), `angles` over `arc` degrees."""
    c = dict(op=op, nx=n, ny=n, nz=nz, dx=vox, dy=vox, dz=vox, nu=nu, nv=nv, du=pix, dv=pix, angles=angles, arc=arc,
             first=0.0, dso=dso, dsd=dsd, dtype=dtype)
    if name:
        c["name"] = name
    c.update(more)
    return c


def listed():
    return [
        # The smallest scan anybody reconstructs here (32^3, 60 views): a call of tens of
        # microseconds, where launches and allocations count; also a first look at a new scanner.
        _case("project_32", "project", 32, 32, 1.0, 64, 64, 1.2, 60, 360.0, 1000.0, 1500.0),
        # Ragged everything: 40 x 36 x 28 anisotropic voxels, odd detector, 23 views.
        dict(_case("backproject_ragged", "backproject", 40, 28, 1.0, 77, 45, 1.3, 23, 360.0, 300.0, 480.0),
             ny=36, dy=1.1, dz=0.9, dv=1.1),
        # The medical head scan (256^3, 512^2, 360 views): one product with A ...
        _case("project_256", "project", 256, 256, 1.0, 512, 512, 0.8, 360, 360.0, 1000.0, 1536.0),
        # ... and one with A^T.
        _case("backproject_256", "backproject", 256, 256, 1.0, 512, 512, 0.8, 360, 360.0, 1000.0, 1536.0),
        # The precision study's 512^3 scan with FP16 storage, every fourth view (an ordered subset).
        dict(_case("project_512_f16", "project", 512, 512, 0.5, 768, 512, 0.8, 180, 360.0, 1000.0, 1536.0, "f16")),
        # The micro-CT scan at magnification 6 (1024^3, 1536^2), one ordered subset of its 1600 views.
        _case("backproject_1024", "backproject", 1024, 1024, 0.1, 1536, 1536, 0.6, 40, 360.0, 200.0, 1200.0),
        # A request of the serving stream: coarse voxels under a fine detector (a voxel covers
        # several pixels), short scan, odd view count, BF16 storage.
        _case("backproject_128_bf16", "backproject", 128, 128, 2.0, 600, 600, 409.6 / 600, 243, 200.0, 1000.0, 1536.0,
              "bf16"),
        # The headline solve: LSQR on the head scan, a few iterations of the usual 30.
        _case("lsqr_256", "lsqr", 256, 256, 1.0, 512, 512, 0.8, 360, 360.0, 1000.0, 1536.0, iters=4, lam=0.0),
        # A small solve where the scalar steps and launches weigh most: CGLS, 20 iterations at 32^3.
        _case("cgls_32", "cgls", 32, 32, 1.0, 64, 64, 1.2, 60, 360.0, 1000.0, 1500.0, iters=20, lam=0.0),
        # Damped LSMR on a short scan with a ragged volume.
        dict(_case("lsmr_short_scan", "lsmr", 130, 97, 2.0, 257, 200, 1.6, 131, 200.0, 1000.0, 1536.0, iters=8, lam=30.0),
             ny=127, first=0.01),
        # BA-GMRES with the unmatched voxel-driven backprojector (forward projector, interpolating
        # backprojector and Arnoldi steps).
        _case("ba_gmres_voxel_128", "ba_gmres", 128, 128, 2.0, 256, 256, 1.6, 180, 360.0, 1000.0, 1536.0, iters=4),
        # Continuous batching: requests of different scans in flight at once, from and to host memory.
        dict(op="serve", name="serve_mix", pick=3, requests=5, n=96, iters=8),
    ]


# ------------------------------------------------------------------- drawing
def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case: any of the listed operations at sizes between the smallest and largest listed ones."""
    op = rng.choice(["project", "project", "backproject", "backproject", "lsqr", "cgls", "lsmr", "ba_gmres", "serve"])
    if op == "serve":
        return dict(op="serve", pick=rng.randrange(1 << 20), requests=rng.randint(2, 6), n=rng.randint(24, 128),
                    iters=rng.randint(4, 10))
    solver = op not in ("project", "backproject")
    n = int(_log(rng, 16, 160 if solver else 640))
    ny = max(8, int(n * rng.choice([1.0, 1.0, rng.uniform(0.8, 1.1)])))
    nz = max(8, int(n * rng.choice([1.0, 1.0, rng.uniform(0.4, 1.1)])))
    micro = rng.random() < 0.25
    fov, dso, dsd = (100.0, 200.0, 1200.0) if micro else (256.0, 1000.0, 1536.0)
    mag = dsd / dso
    vox = fov / max(n, ny)
    nu = max(16, int(n * rng.uniform(1.0, 2.5 if n < 300 else 1.6)))
    nv = max(16, int(max(nu * nz / n, 12) * rng.uniform(0.7, 1.1)))
    pix = fov * mag * rng.uniform(1.0, 1.15) / nu
    updates_per_view = n * ny * nz * 4 / math.pi * (vox * mag / pix) ** 2
    c = _case(None, op, n, nz, vox, nu, nv, pix, 1, rng.choice([360.0, 360.0, 200.0]), dso, dsd,
              "f32" if solver else rng.choice(["f32", "f32", "f16", "bf16"]))
    c["ny"] = ny
    c["first"] = rng.uniform(0.005, 0.02)
    products = 1
    if solver:
        c["iters"] = rng.randint(2, 12 if op != "ba_gmres" else 5)
        if op != "ba_gmres":
            c["lam"] = rng.choice([0.0, 0.0, 30.0])
        products = 2 * c["iters"] + 1
    # no more work than half the largest listed case, nor more rays than it has pixels
    most = min(720.0, 4e10 / (updates_per_view * products), 4e7 * (1.0 if not solver else 0.25) / (nu * nv))
    c["angles"] = max(3, int(_log(rng, min(12, most * 0.5), most)))
    return c


# -------------------------------------------------------------------- inputs
def _angles(c):
    return c["first"] + np.arange(c["angles"], dtype=np.float64) * (math.radians(c["arc"]) / c["angles"])


def _spec(c):
    return {k: c[k] for k in ("nx", "ny", "nz", "dx", "dy", "dz", "nu", "nv", "du", "dv", "dso", "dsd")}


def _ellipsoids(c, seed):
    """Ten ellipsoids (centre, semi-axes, rotation about z, attenuation in 1/mm) inside the volume."""
    rng = np.random.Generator(np.random.PCG64(seed))
    ext = np.array([c["nx"] * c["dx"], c["ny"] * c["dy"], c["nz"] * c["dz"]])
    return [(rng.uniform(-0.25, 0.25, 3) * ext, rng.uniform(0.05, 0.25, 3) * ext, rng.uniform(0.0, math.pi),
             0.02 * rng.uniform(0.05, 1.0) * 256.0 / ext[0]) for _ in range(10)]


def _volume(c, seed):
    """The ellipsoids' summed attenuation at voxel centres, x[k][j][i], FP32."""
    def centres(n, d):
        return (torch.arange(n, device="cuda", dtype=torch.float32) + 0.5) * d - 0.5 * n * d
    x, y, z = centres(c["nx"], c["dx"]), centres(c["ny"], c["dy"]), centres(c["nz"], c["dz"])
    vol = torch.zeros((c["nz"], c["ny"], c["nx"]), device="cuda")
    for o, s, phi, rho in _ellipsoids(c, seed):
        cp, sp = math.cos(phi), math.sin(phi)
        ox, oy = (x - o[0])[None, :], (y - o[1])[:, None]
        plane = ((cp * ox + sp * oy) / s[0]) ** 2 + ((cp * oy - sp * ox) / s[1]) ** 2
        ez = ((z - o[2]) / s[2]) ** 2
        for k0 in range(0, c["nz"], 64):
            vol[k0:k0 + 64] += rho * ((ez[k0:k0 + 64, None, None] + plane) <= 1.0)
    return vol


def _projections(c, seed):
    """Chord lengths through the ellipsoids times attenuation plus log-transformed photon noise
    (I0 = 1e5, Gaussian limit of the counts), y[a][iv][iu], FP32."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = torch.empty((c["angles"], c["nv"], c["nu"]), device="cuda")
    u = ((torch.arange(c["nu"], device="cuda") - 0.5 * (c["nu"] - 1)) * c["du"])[None, :]
    v = ((torch.arange(c["nv"], device="cuda") - 0.5 * (c["nv"] - 1)) * c["dv"])[:, None]
    shapes = _ellipsoids(c, seed)
    length = torch.sqrt(c["dsd"] ** 2 + u * u + v * v)
    for a, t in enumerate(_angles(c)):
        ct, st = math.cos(t), math.sin(t)
        acc = torch.zeros((c["nv"], c["nu"]), device="cuda")
        for o, s, phi, rho in shapes:
            cp, sp = math.cos(phi), math.sin(phi)
            # source and ray direction in the ellipsoid's frame, scaled to the unit sphere
            sx, sy = c["dso"] * ct - o[0], c["dso"] * st - o[1]
            px, py, pz = (cp * sx + sp * sy) / s[0], (cp * sy - sp * sx) / s[1], -o[2] / s[2]
            dx, dy = -c["dsd"] * ct - u * st, -c["dsd"] * st + u * ct
            qx, qy, qz = (cp * dx + sp * dy) / s[0], (cp * dy - sp * dx) / s[1], v / s[2]
            qq = qx * qx + qy * qy + qz * qz
            m = -(px * qx + py * qy + pz * qz) / qq                     # closest approach
            d2 = (px + m * qx) ** 2 + (py + m * qy) ** 2 + (pz + m * qz) ** 2
            acc += rho * 2.0 * torch.sqrt(torch.clamp((1.0 - d2) / qq, min=0.0))
        acc *= length
        noise = torch.randn(acc.shape, device="cuda", generator=gen)
        out[a] = acc + noise * torch.exp(0.5 * acc.clamp(max=8.0)) * 1e5 ** -0.5
    return out


def _requests(c):
    """The scans of a batch: 0.5 .. 1.4 of n^3 voxels over 256 mm, various detectors, full or short scans."""
    rng = random.Random(c["pick"])
    out = []
    for i in range(c["requests"]):
        n = max(16, int(c["n"] * rng.uniform(0.5, 1.4)))
        nu = int(n * rng.uniform(1.2, 2.4))
        short = rng.random() < 0.5
        r = _case(None, "lsqr" if rng.random() < 0.5 else "lsmr", n, n, 256.0 / n, nu, nu, 409.6 / nu,
                  rng.randint(45, 160), 200.0 if short else 360.0, 1000.0, 1536.0, lam=0.0, iters=c["iters"])
        out.append(r)
    return out


class _Scan:
    """A scan description with attributes, as Server.submit takes it."""

    def __init__(self, c):
        for k, v in _spec(c).items():
            setattr(self, k, v)
        self.angles = _angles(c)


# ---------------------------------------------------------------- the library
def prepare(case, seed):
    if case["op"] == "serve":
        server = cbct.Server(64 << 30, max_slots=8)
        jobs = [(_Scan(r), _projections(r, seed + 101 * i).cpu().numpy(), r["op"], r["iters"])
                for i, r in enumerate(_requests(case))]
        return {"case": case, "server": server, "jobs": jobs}
    geom = cbct.Geometry(angles=_angles(case), **_spec(case))
    data = _volume(case, seed) if case["op"] == "project" else _projections(case, seed)
    return {"case": case, "geom": geom, "data": data.to(DTYPES[case["dtype"]]), "stream": torch.cuda.Stream()}


def _history(h):
    # histories are norms of FP32 vectors, kept in FP64
    return np.asarray(h, dtype=np.float32)


def run(state):
    c = state["case"]
    if c["op"] == "serve":
        server = state["server"]
        ids = [server.submit(scan, b, solver=solver, iters=iters) for scan, b, solver, iters in state["jobs"]]
        done = [server.wait(i, timeout=60.0) for i in ids]
        return [{"x": d.x, "resid": _history(d.report.resid), "iters": d.report.iters_done} for d in done]
    geom, data = state["geom"], state["data"]
    if c["op"] == "project":
        return cbct.project(geom, data)
    if c["op"] == "backproject":
        return cbct.backproject(geom, data)
    # solvers replay a captured iteration, which needs a stream other than the legacy default one
    state["stream"].wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(state["stream"]):
        if c["op"] == "ba_gmres":
            x, rep = cbct.ba_gmres(geom, data, c["iters"], backprojector="voxel")
            hist = {"normal_resid": _history(rep.normal_resid)}
        else:
            x, rep = getattr(cbct, c["op"])(geom, data, c["iters"], lam=c["lam"])
            hist = {"resid": _history(rep.resid), "normal_resid": _history(rep.normal_resid)}
    torch.cuda.current_stream().wait_stream(state["stream"])
    return dict(hist, x=x, iters=rep.iters_done)


# ----------------------------------------------------------------------- work
def _updates(c):
    """Ray-voxel pairs of one product: voxels x views x (area of a voxel's shadow / area of a pixel)."""
    mag = c["dsd"] / c["dso"]
    return c["nx"] * c["ny"] * c["nz"] * c["angles"] * (4 / math.pi) * 0.5 * (c["dx"] + c["dy"]) * c["dz"] * mag ** 2 / (
        c["du"] * c["dv"])


def work(case):
    if case["op"] == "serve":
        parts = [work(r) for r in _requests(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    m, n = case["nx"] * case["ny"] * case["nz"], case["angles"] * case["nv"] * case["nu"]
    size = 4 if case["dtype"] == "f32" else 2
    products = 1 if case["op"] in ("project", "backproject") else 2 * case["iters"] + 1
    # every product reads one vector and writes the other
    return {"bytes": products * size * (m + n), "flops": products * 2 * _updates(case)}


# ---------------------------------------------------------- FP64 ray tracing
def _segments(c, a0, a1):
    """Yields (flat voxel index, alpha length) of every ray of views a0..a1, piece by piece, as
    [view, iv, iu] FP64 tensors: alpha runs from 0 at the source to 1 at the pixel.  The x/y plane
    crossings of a detector column are the same for all its rows; they are sorted once per column,
    and inside each x/y cell a row's z crossings are walked one by one."""
    f8 = dict(device="cuda", dtype=torch.float64)
    t = torch.tensor(_angles(c)[a0:a1], **f8)
    u = (torch.arange(c["nu"], **f8) - 0.5 * (c["nu"] - 1)) * c["du"]
    v = (torch.arange(c["nv"], **f8) - 0.5 * (c["nv"] - 1)) * c["dv"]
    ct, st = torch.cos(t)[:, None], torch.sin(t)[:, None]
    edges, lo, hi = [], None, None
    src = {"x": c["dso"] * ct, "y": c["dso"] * st}
    step = {"x": -c["dsd"] * ct - u * st, "y": -c["dsd"] * st + u * ct}
    for ax in "xy":
        n, d = c["n" + ax], c["d" + ax]
        planes = (torch.arange(n + 1, **f8) - 0.5 * n) * d
        flat = step[ax] == 0
        al = (planes - src[ax][..., None]) / torch.where(flat, torch.ones_like(step[ax]), step[ax])[..., None]
        inside = (src[ax] >= planes[0]) & (src[ax] < planes[-1])
        near = torch.where(flat, torch.where(inside, 0.0, 2.0), al.amin(-1))
        far = torch.where(flat, torch.where(inside, 1.0, -1.0), al.amax(-1))
        edges.append(torch.where(flat[..., None], torch.full_like(al, 2.0), al))
        lo = near if lo is None else torch.maximum(lo, near)
        hi = far if hi is None else torch.minimum(hi, far)
    hi = torch.maximum(hi, lo)
    e = torch.cat(edges, -1)
    e = torch.minimum(torch.maximum(e, lo[..., None]), hi[..., None]).sort(-1).values        # [view, iu, crossing]
    bz = -0.5 * c["nz"] * c["dz"]
    rise = v[None, :, None]                                        # z = rise * alpha (the source is at z = 0)
    up = torch.sign(rise)
    safe = torch.where(rise == 0, torch.ones_like(rise), rise)
    for s in range(e.shape[-1] - 1):
        b0, b1 = e[:, :, s], e[:, :, s + 1]
        if not bool((b1 > b0).any()):
            continue
        mid = 0.5 * (b0 + b1)
        i = torch.floor((src["x"] + mid * step["x"]) / c["dx"] + 0.5 * c["nx"]).long().clamp_(0, c["nx"] - 1)
        j = torch.floor((src["y"] + mid * step["y"]) / c["dy"] + 0.5 * c["ny"]).long().clamp_(0, c["ny"] - 1)
        cell = (j * c["nx"] + i)[:, None, :]
        a, b = b0[:, None, :], b1[:, None, :]
        k = torch.floor((rise * a - bz) / c["dz"])
        last = torch.floor((rise * b - bz) / c["dz"])
        pieces = int((last - k).abs().max()) + 1
        start = a.expand_as(k)
        for _ in range(pieces):
            leave = (bz + (k + (up > 0)) * c["dz"]) / safe         # alpha at which the row leaves slab k
            end = torch.where(up == 0, b, torch.minimum(leave, b)).maximum(start)
            ok = (k >= 0) & (k < c["nz"])
            yield (k.clamp(0, c["nz"] - 1).long() * (c["ny"] * c["nx"]) + cell,
                   torch.where(ok, end - start, torch.zeros((), **f8)))
            start, k = end, k + up


def _chunks(c):
    per = max(1, int(2.5e7 / (c["nu"] * c["nv"])))
    return [(a, min(c["angles"], a + per)) for a in range(0, c["angles"], per)]


def _lengths(c):
    f8 = dict(device="cuda", dtype=torch.float64)
    u = (torch.arange(c["nu"], **f8) - 0.5 * (c["nu"] - 1)) * c["du"]
    v = (torch.arange(c["nv"], **f8) - 0.5 * (c["nv"] - 1)) * c["dv"]
    return torch.sqrt(c["dsd"] ** 2 + u[None, :] ** 2 + v[:, None] ** 2)


def _forward64(c, x):
    x = x.double().reshape(-1)
    out = torch.zeros((c["angles"], c["nv"], c["nu"]), device="cuda", dtype=torch.float64)
    for a0, a1 in _chunks(c):
        for idx, length in _segments(c, a0, a1):
            out[a0:a1] += length * x[idx]
    return out * _lengths(c)


def _transpose64(c, y):
    out = torch.zeros(c["nz"] * c["ny"] * c["nx"], device="cuda", dtype=torch.float64)
    for a0, a1 in _chunks(c):
        w = y[a0:a1].double() * _lengths(c)
        for idx, length in _segments(c, a0, a1):
            out.index_add_(0, idx.reshape(-1), (length * w).reshape(-1))
    return out.reshape(c["nz"], c["ny"], c["nx"])


def _voxel_driven64(c, y):
    """Bilinear sample of every view at each voxel centre's projection, weighted by the ray density."""
    f8 = dict(device="cuda", dtype=torch.float64)

    def centres(n, d):
        return (torch.arange(n, **f8) + 0.5) * d - 0.5 * n * d
    x, yy, z = centres(c["nx"], c["dx"])[None, :], centres(c["ny"], c["dy"])[:, None], centres(c["nz"], c["dz"])
    out = torch.zeros((c["nz"], c["ny"], c["nx"]), **f8)
    for a, t in enumerate(_angles(c)):
        view = torch.nn.functional.pad(y[a].double(), (2, 2, 2, 2))       # [iv][iu], a zero border
        mag = c["dsd"] / (c["dso"] - (x * math.cos(t) + yy * math.sin(t)))
        u = (yy * math.cos(t) - x * math.sin(t)) * mag
        v = z[:, None, None] * mag
        fu, fv = u / c["du"] + 0.5 * (c["nu"] - 1), v / c["dv"] + 0.5 * (c["nv"] - 1)
        iu, iv = torch.floor(fu), torch.floor(fv)
        tu, tv = fu - iu, fv - iv
        iu, iv = (iu + 2).clamp(0, c["nu"] + 2).long(), (iv + 2).clamp(0, c["nv"] + 2).long()
        val = ((1 - tv) * ((1 - tu) * view[iv, iu] + tu * view[iv, iu + 1])
               + tv * ((1 - tu) * view[iv + 1, iu] + tu * view[iv + 1, iu + 1]))
        out += val * mag ** 2 * torch.sqrt(c["dsd"] ** 2 + u ** 2 + v ** 2)
    return out * (c["dx"] * c["dy"] * c["dz"] / (c["du"] * c["dv"] * c["dsd"]))


def _krylov64(c, b, method):
    """CGLS / LSQR / LSMR iterate after c["iters"] steps from its definition: FP64 Golub-Kahan
    vectors, then the projected least-squares problem solved densely.  Returns x and the residual
    norm per iteration."""
    lam = c["lam"]
    b = b.double()
    beta = [float(b.norm())]
    u = b / beta[0]
    v = _transpose64(c, u)
    alpha = [float(v.norm())]
    v /= alpha[0]
    basis, resid, y = [v], [], None
    for k in range(1, c["iters"] + 1):
        u = _forward64(c, v) - alpha[-1] * u
        beta.append(float(u.norm()))
        u /= beta[-1]
        v = _transpose64(c, u) - beta[-1] * v
        alpha.append(float(v.norm()))
        v /= alpha[-1]
        h = np.zeros((k + 1, k))
        h[np.arange(k), np.arange(k)] = alpha[:k]
        h[np.arange(1, k + 1), np.arange(k)] = beta[1:k + 1]
        e = np.zeros(k + 1)
        e[0] = beta[0]
        if method == "lsmr":
            m = np.vstack([h.T @ h + lam ** 2 * np.eye(k), np.eye(1, k, k - 1) * alpha[k] * beta[k]])
            y = np.linalg.lstsq(m, np.concatenate([h.T @ e, [0.0]]), rcond=None)[0]
        else:
            y = np.linalg.lstsq(np.vstack([h, lam * np.eye(k)]), np.concatenate([e, np.zeros(k)]), rcond=None)[0]
        damped = 0.0 if method == "cgls" else lam ** 2 * float(y @ y)      # CGLS reports ||b - A x|| itself
        resid.append(math.sqrt(float(np.sum((e - h @ y) ** 2)) + damped))
        if k < c["iters"]:
            basis.append(v)
    return sum(float(w) * q for w, q in zip(y, basis)), resid


def _ba_gmres64(c, b):
    """x minimising ||B (b - A x)|| over the Krylov space of B A and B b, and that norm per iteration."""
    r = _voxel_driven64(c, b)
    beta = float(r.norm())
    q, h, hist, y = [r / beta], np.zeros((c["iters"] + 1, c["iters"])), [], None
    for k in range(c["iters"]):
        w = _voxel_driven64(c, _forward64(c, q[-1]))
        for _ in range(2):
            for i, qi in enumerate(q):
                d = float((w * qi).sum())
                h[i, k] += d
                w = w - d * qi
        h[k + 1, k] = float(w.norm())
        e = np.zeros(k + 2)
        e[0] = beta
        y = np.linalg.lstsq(h[:k + 2, :k + 1], e, rcond=None)[0]
        hist.append(float(np.linalg.norm(e - h[:k + 2, :k + 1] @ y)))
        q.append(w / h[k + 1, k])
    return sum(float(wi) * qi for wi, qi in zip(y, q)), hist


def exact(case, seed):
    if case["op"] == "serve":
        return None
    c = case
    # rays x x/y cells x products, the cost of the tracing below (the transpose scatters)
    steps = c["angles"] * c["nu"] * c["nv"] * (c["nx"] + c["ny"] + 2.0)
    cost = {"project": 1.0, "backproject": 2.0, "ba_gmres": 1.0 * c.get("iters", 0)}.get(c["op"], 3.0 * c.get("iters", 0) + 2.0)
    if steps * cost > 1.0e11 or (c["op"] == "ba_gmres" and c["angles"] * c["nx"] * c["ny"] * c["nz"] * c["iters"] > 1e10):
        return None
    data = (_volume(c, seed) if c["op"] == "project" else _projections(c, seed)).to(DTYPES[c["dtype"]])
    if c["op"] == "project":
        return _forward64(c, data)
    if c["op"] == "backproject":
        return _transpose64(c, data)
    if c["op"] == "ba_gmres":
        x, hist = _ba_gmres64(c, data.double())
        return {"normal_resid": np.asarray(hist), "x": x, "iters": None}
    x, resid = _krylov64(c, data, c["op"])
    return {"resid": np.asarray(resid), "normal_resid": None, "x": x, "iters": None}
