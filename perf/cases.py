"""The work this library is used for, as measurable cases.

Every case runs the public API (Geometry, the solvers, autograd, ROF) on the
circular cone-beam geometry of the repository's workloads: DSO 1000 mm, DSD
1536 mm, a 256 mm field of view, a detector that the volume's shadow fills,
rays sampled every half voxel, uniform angles over 360 degrees.  Sizes are
those of the named workloads (synth.workload), of the serving protocols
(serving_bench) and of the operator benchmark, and ragged ones in between.
Phantoms are seeded random ellipsoids; projections are their analytic line
integrals with 0.5 % noise on the rays that cross the object, so the inputs
depend on no projector.

A case: "kind" (which entry point), volume "nx, ny, nz", detector "nu, nv",
"angles", "dtype" (storage), "offset" (detector and volume off centre), and
what the kind takes ("iters", "batch", "block", ...).
"""
import math

import numpy as np
import torch

from paper_1905_03748_gb300 import autograd, synth, tigre

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}
BYTES = {"f32": 4, "bf16": 2, "f16": 2}


def _case(kind, n, det, angles, dtype="f32", offset=False, **more):
    nx, ny, nz = (n, n, n) if isinstance(n, int) else n
    nu, nv = (det, det) if isinstance(det, int) else det
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, nu=nu, nv=nv, angles=angles, dtype=dtype,
                offset=offset, **more)


def listed():
    out = {
        # one subset of an OS-SART sweep written by the user: the smallest call
        # there is (20 of the 100 angles of the 64^3 workload)
        "forward_block_64": _case("forward", 64, 128, 100, block=20),
        # the 64^3 x 100 workload as bench.py runs it: ten SIRT iterations
        "sirt_64": _case("sirt", 64, 128, 100, iters=10),
        # a group of four equal requests on the reconstruction server
        # (128^3 / 256^2 / 90 angles / BF16 protocol), graph replay on a stream
        "serve_128_bf16_x4": _case("cgls_batch", 128, 256, 90, "bf16", iters=6, batch=4),
        # iterative reconstruction with the regulariser (OS-SART with subsets
        # of 20 angles and 20 TV steps after each iteration), 192^3 protocol
        "sart_tv_192": _case("sart", 192, 320, 180, iters=2, subset=20, tv_steps=20),
        # a gradient step on a differentiable projector: A x and the exact
        # transpose of the residual, ragged sizes
        "autograd_135": _case("autograd", (135, 121, 109), (203, 171), 91, offset=True),
        # the 256^3 / 384^2 / 360 BF16 protocol reconstructed alone
        "cgls_256_bf16": _case("cgls", 256, 384, 360, "bf16", iters=2),
        # the ray-voxel intersection projector on ragged sizes, off centre
        "siddon_257": _case("siddon", (257, 243, 201), (333, 273), 180, offset=True),
        # analytic reconstruction of detector data kept in FP16, ragged sizes
        "fdk_389_f16": _case("fdk", (389, 405, 301), (509, 397), 361, "f16", offset=True),
        # image denoising (ROF), 30 iterations
        "rof_320": _case("rof", (320, 300, 288), 1, 1, iters=30),
        # the operators of the benchmark workload (one CGLS iteration is one
        # of each)
        "forward_512": _case("forward", 512, 512, 360),
        "backward_512": _case("backward", 512, 512, 360, weight="matched"),
        # the projection at the large in-core size, sparse angles
        "forward_1024": _case("forward", 1024, 1024, 90),
    }
    return [dict(c, name=name) for name, c in out.items()]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(c):
    """Ray samples (two per voxel) of one pass, up to a constant."""
    reps = {"sirt": 4, "sart": 4, "cgls": 3, "cgls_batch": 3, "autograd": 3}.get(c["kind"], 1)
    return (reps * c.get("iters", 1) * c.get("batch", 1) * c["nu"] * c["nv"]
            * c.get("block", c["angles"]) * max(c["nx"], c["ny"]))


def draw(rng):
    """One more case: a kind, its sizes over the range of the listed ones
    (log-uniform, mostly ragged), its storage type and options."""
    ranges = {  # volume edge, angles
        "forward": (64, 800, 20, 400), "backward": (64, 640, 20, 400), "sirt": (48, 160, 60, 200),
        "sart": (64, 224, 60, 200), "cgls": (96, 320, 90, 360), "cgls_batch": (64, 192, 60, 180),
        "autograd": (48, 192, 30, 120), "siddon": (64, 400, 45, 360), "fdk": (96, 480, 90, 500),
        "rof": (64, 400, 1, 1)}
    while True:
        kind = rng.choice(sorted(ranges))
        lo, hi, alo, ahi = ranges[kind]
        n = _log(rng, lo, hi)
        cube = rng.random() < 0.3
        nx, ny, nz = (n if cube else max(16, int(n * rng.uniform(0.7, 1.0))) for _ in range(3))
        up = rng.choice((1.0, 1.25, 1.5, 2.0))
        nu, nv = int(max(nx, ny) * up), int(nz * up)
        dtype = rng.choice({"forward": ("f32", "f32", "bf16", "f16"), "cgls": ("f32", "bf16"),
                            "backward": ("f32", "f32", "bf16", "f16"),
                            "cgls_batch": ("f32", "bf16"), "fdk": ("f32", "f16")}.get(kind, ("f32",)))
        c = _case(kind, (nx, ny, nz), (nu, nv), _log(rng, alo, ahi), dtype, rng.random() < 0.5)
        if kind == "forward" and rng.random() < 0.3:
            c["block"] = max(1, c["angles"] // rng.randint(2, 8))
        if kind == "backward":
            c["weight"] = rng.choice(("matched", "fdk"))
        if kind in ("sirt", "sart", "cgls", "cgls_batch"):
            c["iters"] = rng.randint(1, 6 if kind != "cgls" else 2)
        if kind == "cgls_batch":
            c["batch"] = rng.randint(2, 4)
        if kind == "sart":
            c["subset"], c["tv_steps"] = rng.choice((10, 20, 30)), rng.choice((0, 10, 20))
        if kind == "rof":
            c["nu"] = c["nv"] = 1
            c["iters"] = rng.randint(10, 40)
        if _cost(c) <= 9.0e10:
            return c


# ------------------------------------------------------------------ inputs

def _geometry(c):
    d = 256.0 / max(c["nx"], c["ny"])
    half = 0.5 * max(c["nx"], c["ny"]) * d
    du = 2.0 * 1536.0 * half / ((1000.0 - half) * c["nu"])
    dv = 2.0 * 1536.0 * 0.5 * c["nz"] * d / ((1000.0 - half) * c["nv"])
    off = bool(c["offset"])
    return dict(DSO=1000.0, DSD=1536.0, n_voxel=(c["nx"], c["ny"], c["nz"]), d_voxel=(d, d, d),
                off_origin=(0.5, -0.3, 0.2) if off else (0.0, 0.0, 0.0), n_det=(c["nu"], c["nv"]),
                d_det=(du, dv), off_det=(1.3 * du, -0.7 * dv) if off else (0.0, 0.0), accuracy=0.5)


def _angles(c):
    return 2.0 * math.pi * np.arange(c["angles"], dtype=np.float64) / c["angles"]


def _ellipsoids(c, seed):
    geo = _geometry(c)
    n, d = min(geo["n_voxel"]), geo["d_voxel"][0]
    return synth.random_ellipsoids(n, d, 16, seed, r_vox=(12.0, 150.0))


def _phantom(c, seed):
    geo = _geometry(c)
    return synth.voxelize_torch(_ellipsoids(c, seed), geo["n_voxel"], geo["d_voxel"],
                                (0, c["nz"]), "cuda", geo["off_origin"])


def _frame(geo, t):
    """Source, pixel (0, 0)'s offset from it, and the pixel steps of one angle."""
    cs, sn = math.cos(t), math.sin(t)
    nu, nv = geo["n_det"]
    du, dv = geo["d_det"]
    u0 = -0.5 * (nu - 1) * du + geo["off_det"][0]
    v0 = -0.5 * (nv - 1) * dv + geo["off_det"][1]
    src = np.array([geo["DSO"] * cs, geo["DSO"] * sn, 0.0])
    base = np.array([-geo["DSD"] * cs - u0 * sn, -geo["DSD"] * sn + u0 * cs, v0])
    return src, base, np.array([-sn * du, cs * du, 0.0]), np.array([0.0, 0.0, dv])


def _projections(c, seed, noise=0.005):
    """Line integrals of the phantom's ellipsoids (analytic, FP64), plus noise."""
    geo = _geometry(c)
    nu, nv = geo["n_det"]
    f64 = dict(dtype=torch.float64, device="cuda")
    p, q = torch.arange(nu, **f64)[None, :], torch.arange(nv, **f64)[:, None]
    u = p * geo["d_det"][0] - 0.5 * (nu - 1) * geo["d_det"][0] + geo["off_det"][0]
    v = q * geo["d_det"][1] - 0.5 * (nv - 1) * geo["d_det"][1] + geo["off_det"][1]
    length = torch.sqrt(geo["DSD"] ** 2 + u * u + v * v)
    ells = _ellipsoids(c, seed)
    out = torch.empty((c["angles"], nv, nu), dtype=torch.float32, device="cuda")
    for a, t in enumerate(_angles(c)):
        src, base, eu, ev = _frame(geo, t)
        acc = torch.zeros((nv, nu), **f64)
        for e in ells:
            m = e.rot / np.array(e.axes)[:, None]
            o, b, x, y = m @ (src - np.array(e.centre)), m @ base, m @ eu, m @ ev
            A = (b @ b + 2 * (b @ x) * p + (x @ x) * p * p) + \
                (2 * (b @ y) * q + (y @ y) * q * q) + (2 * (x @ y)) * (p * q)
            B = (o @ b + (o @ x) * p) + (o @ y) * q
            acc += (2.0 * e.density) * torch.sqrt(torch.clamp(B * B - A * (o @ o - 1.0), min=0.0)) / A
        out[a] = acc * length
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    sigma = noise * float(out.max())
    for a in range(c["angles"]):
        out[a] += (out[a] > 0) * torch.randn((nv, nu), generator=gen, device="cuda") * sigma
    return out


def prepare(case, seed):
    c, dt = case, DTYPES[case["dtype"]]
    s = {"case": c}
    if c["kind"] == "rof":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        f = _phantom(c, seed)
        s["f"] = f + 0.1 * torch.randn(f.shape, generator=gen, device="cuda")
        s["out"] = torch.empty_like(f)
        return s
    s["G"] = G = tigre.Geometry(_geometry(c), _angles(c))
    kind = c["kind"]
    if kind == "siddon":
        tigre.tigre_geometry_set_projector(G.handle, "siddon")
    if kind in ("forward", "siddon"):
        s["vol"] = _phantom(c, seed).to(dt)
        s["out"] = torch.empty((c.get("block", c["angles"]),) + G.proj_shape[1:], dtype=dt,
                               device="cuda")
    elif kind == "autograd":
        s["vol"] = _phantom(c, seed).requires_grad_()
        s["b"] = _projections(c, seed + 1)
    elif kind == "cgls_batch":
        s["b"] = [_projections(c, 1000 * seed + i).to(dt) for i in range(c["batch"])]
        s["x"] = [torch.empty(G.vol_shape, dtype=dt, device="cuda") for _ in range(c["batch"])]
        s["stream"] = torch.cuda.Stream()
    else:
        s["b"] = _projections(c, seed).to(dt)
        out = torch.float32 if kind == "fdk" else dt
        s["x"] = torch.empty(G.vol_shape, dtype=out, device="cuda")
    return s


def run(state):
    s, c = state, state["case"]
    kind, G = c["kind"], s.get("G")
    if kind == "forward":
        block = c.get("block", c["angles"])
        return G.forward(s["vol"], out=s["out"], angle_begin=(c["angles"] - block) // 2,
                         angle_count=block)
    if kind == "siddon":
        return G.forward(s["vol"], out=s["out"])
    if kind == "backward":
        return G.backward(s["b"], out=s["x"], weight=c["weight"])
    if kind == "fdk":
        return G.fdk(s["b"], out=s["x"])
    if kind == "autograd":
        y = autograd.forward_project(s["vol"], G)
        g, = torch.autograd.grad(y, s["vol"], y.detach() - s["b"])
        return {"proj": y.detach(), "grad": g}
    if kind == "rof":
        return tigre.tigre_rof_denoise(s["f"], 12.0, c["iters"], out=s["out"])
    if kind == "cgls":
        h = tigre.tigre_cgls(G.handle, s["b"], s["x"], c["iters"], x0_zero=True)
        return {"x": s["x"], "residuals": h.tolist()}
    if kind == "cgls_batch":
        s["stream"].wait_stream(torch.cuda.current_stream())
        b = tigre.tigre_cgls_batch_begin(G.handle, s["b"], s["x"], n_iter_hint=c["iters"],
                                         stream=s["stream"], graph=True, x0_zero=True)
        for done in range(0, c["iters"], 2):  # two iterations a tick, as the server does
            tigre.tigre_cgls_batch_iterate(b, min(2, c["iters"] - done))
        h = [tigre.tigre_cgls_batch_history(b, i, c["iters"]).tolist() for i in range(c["batch"])]
        tigre.tigre_cgls_batch_end(b)
        torch.cuda.current_stream().wait_stream(s["stream"])
        return {"x": s["x"], "residuals": h}
    s["x"].zero_()
    if kind == "sirt":
        h = tigre.tigre_sirt(G.handle, s["b"], s["x"], c["iters"])
    else:
        h = tigre.tigre_sart(G.handle, s["b"], s["x"], c["iters"], subset_size=c["subset"],
                             nonneg=True, tv_steps=c["tv_steps"])
    return {"x": s["x"], "residuals": h.tolist()}


# -------------------------------------------------------------------- work

def _samples(c, angles):
    """Ray samples (interpolated) or voxels crossed (Siddon) of `angles`
    projections, from a coarse grid of rays."""
    geo = _geometry(c)
    n, d = np.array(geo["n_voxel"], float), np.array(geo["d_voxel"])
    lo = (-0.5 * (n + 1)) * d + np.array(geo["off_origin"])
    hi = -lo + 2 * np.array(geo["off_origin"])
    total = 0.0
    for t in np.arange(16) * (2 * math.pi / 16) + 0.1:
        src, base, eu, ev = _frame(geo, t)
        p = (np.arange(24) + 0.5) / 24 * c["nu"] - 0.5
        q = (np.arange(24) + 0.5) / 24 * c["nv"] - 0.5
        r = base + p[None, :, None] * eu + q[:, None, None] * ev
        with np.errstate(divide="ignore", invalid="ignore"):
            ta, tb = (lo - src) / r, (hi - src) / r
        t0 = np.maximum(np.minimum(ta, tb).max(-1), 0.0)
        t1 = np.minimum(np.maximum(ta, tb).min(-1), 1.0)
        span = np.clip(t1 - t0, 0.0, None)
        if c["kind"] == "siddon":
            total += (span * (np.abs(r) / d).sum(-1)).mean()
        else:
            total += (span * np.linalg.norm(r, axis=-1)).mean() / (0.5 * d[0])
    return total / 16 * c["nu"] * c["nv"] * angles


def work(case):
    c, e = case, BYTES[case["dtype"]]
    vol = c["nx"] * c["ny"] * c["nz"]
    na = c.get("block", c["angles"])
    proj = c["nu"] * c["nv"] * na
    kind, it = c["kind"], c.get("iters", 1)
    # 22 per trilinear sample, 12 per voxel and angle, 3 per voxel crossed,
    # 30 per voxel of a TV gradient, 40 per voxel of a ROF iteration
    if kind == "rof":
        return {"bytes": 8.0 * vol, "flops": it * 40.0 * vol}
    fwd = 3.0 * _samples(c, na) if kind == "siddon" else 22.0 * _samples(c, na)
    bwd = 12.0 * vol * na
    if kind in ("forward", "siddon"):
        return {"bytes": float(e * (vol + proj)), "flops": fwd}
    if kind == "backward":
        return {"bytes": float(e * (vol + proj)), "flops": bwd}
    if kind == "fdk":
        return {"bytes": float(4 * vol + e * proj), "flops": bwd + 2.0 * proj * c["nu"] / 2}
    if kind == "autograd":
        return {"bytes": 4.0 * (2 * vol + 3 * proj), "flops": 2 * fwd}
    if kind in ("sirt", "sart"):  # also A 1; x starts from zero
        tv = it * c.get("tv_steps", 0)
        return {"bytes": 4.0 * (vol + proj),
                "flops": (it + 1) * fwd + it * bwd + 30.0 * tv * vol}
    batch = c.get("batch", 1)
    return {"bytes": float(batch * e * (vol + proj)),
            "flops": batch * (it * fwd + (it + 1) * bwd)}


# ------------------------------------------------------- the same in 64 bits

def _unit(i, n):
    """A coordinate in voxel units as grid_sample takes it (align_corners)."""
    return i * (2.0 / (n - 1)) - 1.0


class _Exact:
    """The operators in FP64 with torch alone."""

    def __init__(self, c):
        self.c, self.geo, self.angles = c, _geometry(c), _angles(c)
        self.f64 = dict(dtype=torch.float64, device="cuda")

    def _rays(self, t):
        """Per ray of an angle: first sample and step (index units, x y z), weight, count."""
        geo = self.geo
        nu, nv = geo["n_det"]
        src, base, eu, ev = _frame(geo, t)
        q, p = torch.arange(nv, **self.f64)[:, None], torch.arange(nu, **self.f64)[None, :]
        t0, t1 = torch.zeros((nv, nu), **self.f64), torch.ones((nv, nu), **self.f64)
        s, r = [], []
        for k in range(3):
            n, d = geo["n_voxel"][k], geo["d_voxel"][k]
            s.append((src[k] - geo["off_origin"][k]) / d + 0.5 * (n - 1))
            r.append((base[k] + p * eu[k] + q * ev[k]) / d)
            ta, tb = (-1.0 - s[k]) / r[k], (n - s[k]) / r[k]
            level = r[k] == 0
            t0 = torch.maximum(t0, torch.where(level, t0, torch.minimum(ta, tb)))
            t1 = torch.minimum(t1, torch.where(level, t1, torch.maximum(ta, tb)))
            if not -1.0 < s[k] < n:
                t1 = torch.where(level, -1.0, t1)
        full = torch.sqrt(sum((r[k] * geo["d_voxel"][k]) ** 2 for k in range(3)))
        length = torch.clamp(t1 - t0, min=0.0) * full
        step = geo["accuracy"] * min(geo["d_voxel"])
        K = torch.where(t1 > t0, torch.clamp(torch.ceil(length / step - 1e-9), min=1.0), 0.0)
        inv = 1.0 / torch.clamp(K, min=1.0)
        dt = (t1 - t0) * inv
        first = [s[k] + (t0 + 0.5 * dt) * r[k] for k in range(3)]
        return first, [dt * r[k] for k in range(3)], length * inv, K

    def _grids(self, t):
        """(grid, weight) chunks over the samples of an angle's rays."""
        first, step, h, K = self._rays(t)
        n = self.geo["n_voxel"]
        per = max(1, int(3.0e7 / K.numel()))
        for k0 in range(0, int(K.max()), per):
            k = torch.arange(k0, min(k0 + per, int(K.max())), **self.f64)[:, None, None]
            grid = torch.stack([_unit(first[i] + k * step[i], n[i]) for i in range(3)], dim=-1)
            yield grid[None], torch.where(k < K, h, 0.0)

    def forward(self, vol, angles=None):
        v = vol.double()[None, None]
        out = []
        for t in self.angles if angles is None else angles:
            acc = 0.0
            for grid, w in self._grids(t):
                f = torch.nn.functional.grid_sample(v, grid, "bilinear", "zeros", True)[0, 0]
                acc = acc + (f * w).sum(0)
            out.append(acc)
        return torch.stack(out)

    def adjoint(self, proj):
        c = self.c
        vol = torch.zeros((1, 1, c["nz"], c["ny"], c["nx"]), **self.f64)
        like = torch.empty_like(vol)
        for a, t in enumerate(self.angles):
            for grid, w in self._grids(t):
                vol += torch.ops.aten.grid_sampler_3d_backward(
                    (w * proj[a].double())[None, None], like, grid, 0, 0, True, [True, False])[0]
        return vol[0, 0]

    def siddon(self, vol):
        geo, v = self.geo, vol.double().reshape(-1)
        nu, nv = geo["n_det"]
        nx, ny, nz = geo["n_voxel"]
        q, p = torch.arange(nv, **self.f64)[:, None], torch.arange(nu, **self.f64)[None, :]
        out = []
        for t in self.angles:
            src, base, eu, ev = _frame(geo, t)
            t0, t1 = torch.zeros((nv, nu), **self.f64), torch.ones((nv, nu), **self.f64)
            s, r, cross = [], [], []
            for k in range(3):
                n, d = geo["n_voxel"][k], geo["d_voxel"][k]
                s.append((src[k] - geo["off_origin"][k]) / d + 0.5 * (n - 1))
                r.append(((base[k] + p * eu[k] + q * ev[k]) / d).expand(nv, nu))
                cr = (torch.arange(n + 1, **self.f64) - 0.5 - s[k]) / r[k][..., None]
                t0 = torch.maximum(t0, torch.minimum(cr[..., 0], cr[..., -1]))
                t1 = torch.minimum(t1, torch.maximum(cr[..., 0], cr[..., -1]))
                cross.append(cr)
            t1 = torch.maximum(t0, t1)
            cut = torch.cat(cross, -1).clamp(t0[..., None], t1[..., None]).sort(-1).values
            mid = 0.5 * (cut[..., 1:] + cut[..., :-1])
            i = [torch.floor(s[k] + mid * r[k][..., None] + 0.5).long().clamp(0, geo["n_voxel"][k] - 1)
                 for k in range(3)]
            f = v[(i[2] * ny + i[1]) * nx + i[0]]
            full = torch.sqrt(sum((r[k] * geo["d_voxel"][k]) ** 2 for k in range(3)))
            out.append((f * (cut[..., 1:] - cut[..., :-1])).sum(-1) * full)
        return torch.stack(out)

    def backward(self, proj, weight="matched", angles=None, ones=None):
        """sum over angles of w * bilinear(proj); with `ones`, also of w * bilinear(1)."""
        geo = self.geo
        (nx, ny, nz), (dx, dy, dz) = geo["n_voxel"], geo["d_voxel"]
        (nu, nv), (du, dv) = geo["n_det"], geo["d_det"]
        X, Y, Z = ((torch.arange(n, **self.f64) - 0.5 * (n - 1)) * d + o
                   for n, d, o in zip(geo["n_voxel"], geo["d_voxel"], geo["off_origin"]))
        X, Y = X[None, :], Y[:, None]
        out = torch.zeros((nz, ny, nx), **self.f64)
        den = torch.zeros((nz, ny, nx), **self.f64) if ones is not None else None
        per = max(1, int(3.0e7 / (nx * ny)))
        for a, t in enumerate(self.angles if angles is None else angles):
            cs, sn = math.cos(t), math.sin(t)
            depth = geo["DSO"] - (X * cs + Y * sn)
            mag = geo["DSD"] / depth
            pu = (Y * cs - X * sn) * mag / du + 0.5 * (nu - 1) - geo["off_det"][0] / du
            l2 = (X - geo["DSO"] * cs) ** 2 + (Y - geo["DSO"] * sn) ** 2
            img = proj[a].double()[None, None]
            for z0 in range(0, nz, per):
                z = Z[z0:z0 + per, None, None]
                pv = z * mag / dv + 0.5 * (nv - 1) - geo["off_det"][1] / dv
                grid = torch.stack([_unit(pu, nu).expand_as(pv), _unit(pv, nv)], -1)
                grid = grid.reshape(1, -1, nx, 2)
                if weight == "fdk":
                    w = (geo["DSO"] / depth) ** 2
                else:
                    w = dx * dy * dz / (du * dv) * geo["DSD"] ** 2 / depth ** 3 * torch.sqrt(l2 + z * z)
                f = torch.nn.functional.grid_sample(img, grid, "bilinear", "zeros", True)
                out[z0:z0 + per] += w * f.reshape(pv.shape)
                if ones is not None:
                    f = torch.nn.functional.grid_sample(ones, grid, "bilinear", "zeros", True)
                    den[z0:z0 + per] += w * f.reshape(pv.shape)
        return out if ones is None else (out, den)

    def fdk(self, proj):
        geo, na = self.geo, len(self.angles)
        (nu, nv), (du, dv) = geo["n_det"], geo["d_det"]
        u = (torch.arange(nu, **self.f64) - 0.5 * (nu - 1)) * du + geo["off_det"][0]
        v = (torch.arange(nv, **self.f64) - 0.5 * (nv - 1)) * dv + geo["off_det"][1]
        cosw = geo["DSD"] / torch.sqrt(geo["DSD"] ** 2 + u[None, :] ** 2 + v[:, None] ** 2)
        tau = du * geo["DSO"] / geo["DSD"]
        k = torch.arange(nu, **self.f64)[:, None] - torch.arange(nu, **self.f64)[None, :]
        ramp = torch.where(k == 0, 0.25, torch.where(k % 2 == 0, 0.0, -1.0 / (math.pi * k) ** 2)) / tau
        filt = torch.stack([(proj[a].double() * cosw) @ ramp for a in range(na)]) * (math.pi / na)
        return self.backward(filt, "fdk")

    def tv_step(self, x, alpha, eps):
        D = []
        for axis in (2, 1, 0):
            d = torch.zeros_like(x)
            n = x.shape[axis]
            d.narrow(axis, 1, n - 1).copy_(x.narrow(axis, 1, n - 1) - x.narrow(axis, 0, n - 1))
            D.append(d)
        inv = 1.0 / torch.sqrt(D[0] ** 2 + D[1] ** 2 + D[2] ** 2 + eps)
        g = (D[0] + D[1] + D[2]) * inv
        for axis, d in zip((2, 1, 0), D):
            n = x.shape[axis]
            g.narrow(axis, 0, n - 1).sub_((d * inv).narrow(axis, 1, n - 1))
        norm = torch.linalg.vector_norm(g)
        return x - alpha / norm * g if float(norm) > 0 else x

    def sart(self, b, iters, subset, tv_steps=0, nonneg=False):
        c = self.c
        x = torch.zeros((c["nz"], c["ny"], c["nx"]), **self.f64)
        W = self.forward(torch.ones_like(x))
        W = torch.where(W > 1e-12, 1.0 / W, 0.0)
        ones = torch.ones((1, 1, c["nv"], c["nu"]), **self.f64)
        hist = []
        for _ in range(iters):
            before, sq = x.clone(), 0.0
            for a0 in range(0, c["angles"], subset):
                ang = self.angles[a0:a0 + subset]
                r = b[a0:a0 + subset].double() - self.forward(x, ang)
                sq += float((r * r).sum())
                num, den = self.backward(r * W[a0:a0 + subset], angles=ang, ones=ones)
                x = x + torch.where(den > 1e-12, num / den, 0.0)
                x = x.clamp(min=0.0) if nonneg else x
            hist.append(math.sqrt(sq))
            alpha = 0.002 * float(torch.linalg.vector_norm(x - before))
            for _ in range(tv_steps):
                x = self.tv_step(x, alpha, 1e-8)
        return {"x": x, "residuals": hist}

    def cgls(self, b, iters):
        r = b.double()
        p = self.backward(r)
        gamma, x, hist = (p * p).sum(), torch.zeros_like(p), []
        for _ in range(iters):
            q = self.forward(p)
            alpha = gamma / (q * q).sum()
            x = x + alpha * p
            r = r - alpha * q
            hist.append(float(torch.linalg.vector_norm(r)))
            s = self.backward(r)
            new = (s * s).sum()
            p = s + new / gamma * p
            gamma = new
        return {"x": x, "residuals": hist}


def _rof(f, lam, iters):
    f = f.double()
    tau = 1.0 / math.sqrt(12.0)
    u, bar = f.clone(), f.clone()
    p = [torch.zeros_like(f) for _ in range(3)]
    for _ in range(iters):
        for i, axis in enumerate((2, 1, 0)):
            n = f.shape[axis]
            p[i].narrow(axis, 0, n - 1).add_(tau * (bar.narrow(axis, 1, n - 1) - bar.narrow(axis, 0, n - 1)))
        inv = 1.0 / torch.clamp(torch.sqrt(p[0] ** 2 + p[1] ** 2 + p[2] ** 2), min=1.0)
        div = torch.zeros_like(f)
        for i, axis in enumerate((2, 1, 0)):
            p[i] *= inv
            n = f.shape[axis]
            div.narrow(axis, 0, n - 1).add_(p[i].narrow(axis, 0, n - 1))
            div.narrow(axis, 1, n - 1).sub_(p[i].narrow(axis, 0, n - 1))
        new = (u + tau * div + tau * lam * f) / (1.0 + tau * lam)
        bar, u = 2.0 * new - u, new
    return u


def exact(case, seed):
    c, kind = case, case["kind"]
    passes = c.get("batch", 1) * (c.get("iters", 1) + (kind in ("sirt", "sart")))
    rays = c["nu"] * c["nv"] * c.get("block", c["angles"]) * passes
    if kind not in ("rof", "backward", "fdk") and rays * max(c["nx"], c["ny"]) > 3.0e10:
        return None  # more than about 20 seconds of FP64 samples
    dt = DTYPES[c["dtype"]]
    E = _Exact(c)
    if kind == "forward":
        block = c.get("block", c["angles"])
        a0 = (c["angles"] - block) // 2
        return E.forward(_phantom(c, seed).to(dt), E.angles[a0:a0 + block])
    if kind == "siddon":
        return E.siddon(_phantom(c, seed))
    if kind == "autograd":
        y = E.forward(_phantom(c, seed))
        return {"proj": y, "grad": E.adjoint(y - _projections(c, seed + 1))}
    if kind == "rof":
        return _rof(prepare(c, seed)["f"], 12.0, c["iters"])
    if kind == "cgls_batch":
        got = [E.cgls(_projections(c, 1000 * seed + i).to(dt), c["iters"]) for i in range(c["batch"])]
        return {"x": [g["x"] for g in got], "residuals": [g["residuals"] for g in got]}
    b = _projections(c, seed).to(dt)
    if kind == "backward":
        return E.backward(b, c["weight"])
    if kind == "fdk":
        return E.fdk(b)
    if kind == "cgls":
        return E.cgls(b, c["iters"])
    if kind == "sirt":
        return E.sart(b, c["iters"], c["angles"])
    return E.sart(b, c["iters"], c["subset"], c["tv_steps"], True)
