"""The measured work of this framework: what a user has it do, through its Python entry points.

Eleven kinds of call cover the path: novel views of an MPI (a viewer's single view, a light
field's grid, a display's arc), single HSGD iterations (coarse and fine levels, odd sizes, both
storage types, both selection rules), a whole refinement, the batched step of the server, the
differentiable render with its backward pass, the gradient volume and the learned iteration.
Sizes come from the repository's workloads (128x96 to 1920x1080, 8 to 64 planes, 1 to 8 source
views, 1 to 45 novel views); ``draw`` spreads over the same ranges.

Every refinement starts from a coarse MPI that the caller holds and copies into the working MPI,
as a server does with each request, so every pass does the same work on the same values.

``exact`` evaluates the same results in 64-bit torch from the ray/plane geometry, without this
repository's code.  Which planes a pixel keeps is decided on 32-bit keys (products of the stored
alphas, a documented part of the interface), so the selection alone is formed in 32 bits there.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2307_03017_gb300 as rl
from paper_2307_03017_gb300.autograd import warp_composite

DEV = "cuda"
NEAR, FAR = 1.0, 100.0


# ------------------------------------------------------------------------------ cases

def listed():
    return [
        # a viewer's single head-tracked view of a small MPI: latency and launches
        dict(name="view_256x192", kind="render", H=192, W=256, D=16, T=1, poses="rotated", dtype="bf16"),
        # the 3x3 grid of novel views of one refined 512x384 scene
        dict(name="views_grid_512x384", kind="render", H=384, W=512, D=32, T=9, poses="grid", dtype="f32"),
        # one frame of a 45-view light-field display
        dict(name="views_arc_1920x1080", kind="render", H=1080, W=1920, D=64, T=45, poses="arc", dtype="bf16"),
        # the three iterations' ends of a 512x384 refinement: the coarsest (latency) and the finest
        dict(name="step_l2_512x384", kind="step", H=384, W=512, D=32, N=4, k=5, level=2, poses="rotated",
             select="topk", prior=0.0, dtype="f32"),
        dict(name="step_l0_512x384", kind="step", H=384, W=512, D=32, N=4, k=5, level=0, poses="rotated",
             select="topk", prior=0.0, dtype="f32"),
        # forward-facing captures at 378x512: three views, 40 planes, odd level height, the window
        # selection and the sparsity prior
        dict(name="step_l1_378x512", kind="step", H=378, W=512, D=40, N=3, k=5, level=1, poses="rotated",
             select="mvs", prior=0.1, dtype="bf16"),
        # one fine iteration of the display workload: eight views on a grid
        dict(name="step_l0_1920x1080", kind="step", H=1080, W=1920, D=64, N=8, k=5, level=0, poses="grid",
             select="topk", prior=0.0, dtype="bf16"),
        # a whole coarse-to-fine refinement
        dict(name="refine_512x384", kind="refine", H=384, W=512, D=32, N=4, k=5, iters=3, poses="rotated", dtype="f32"),
        # one step of the server's batched engine: requests of mixed sizes and levels
        dict(name="batch_8_requests", kind="batch", n=8, Hmax=768, Wmax=1024, Dmax=64, Nmax=6, k=5, mix=1),
        # training through the render: views and the MPI's gradient, at a size no tile divides
        dict(name="backward_375x500", kind="backward", H=375, W=500, D=32, T=4, poses="rotated", dtype="f32"),
        # the learned update's input, and one learned iteration
        dict(name="volume_l0_512x384", kind="volume", H=384, W=512, D=32, N=4, k=5, level=0, dtype="f32"),
        dict(name="learned_l0_512x384", kind="learned", H=384, W=512, D=32, N=4, k=5, level=0, dtype="f32"),
    ]


# The largest listed work, in bilinear samples (views x planes x pixels): 45 x 64 x 1080 x 1920.
_MOST_SAMPLES = 2.0e9


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["render", "render", "step", "step", "step", "refine", "batch", "backward", "volume", "learned"])
    dtype = rng.choice(["f32", "bf16"])
    if kind == "batch":
        return dict(kind=kind, n=rng.randint(1, 12), Hmax=_log(rng, 192, 768), Wmax=_log(rng, 256, 1024),
                    Dmax=rng.randint(16, 64), Nmax=rng.randint(2, 6), k=rng.randint(1, 8), mix=rng.randint(0, 1 << 20))
    most_h, most_w = (1080, 1920) if kind in ("render", "step") else (540, 960)
    level = rng.choice([0, 1, 2]) if kind in ("step", "volume", "learned") else 0
    iters = rng.choice([2, 3])
    unit = (1 << level) if kind != "refine" else 4
    H = max(1, _log(rng, 96, most_h) // unit) * unit
    W = max(1, _log(rng, 128, most_w) // unit) * unit
    D = rng.randint(8, 64)
    views = _log(rng, 1, 45) if kind == "render" else rng.randint(1 if kind == "backward" else 2, 7)
    while views > 1 and views * D * H * W > _MOST_SAMPLES:
        views -= 1
    poses = rng.choice(["rotated", "grid"] + (["arc"] if kind == "render" else []))
    if kind in ("render", "backward"):
        return dict(kind=kind, H=H, W=W, D=D, T=views, poses=poses, dtype=dtype)
    k = rng.randint(1, min(8, D))
    c = dict(kind=kind, H=H, W=W, D=D, N=views, k=k, dtype=dtype)
    if kind == "step":
        c.update(level=level, poses=poses, select=rng.choice(["topk", "topk", "mvs"]), prior=rng.choice([0.0, 0.0, 0.1]))
    elif kind == "refine":
        c.update(iters=iters, poses=poses)
    else:
        c.update(level=level)
    return c


# ----------------------------------------------------------------------------- scenes

class Camera:
    """World -> camera pinhole (x = R X + t, pixel = K x / z)."""

    def __init__(self, K, R, t):
        self.K, self.R, self.t = (np.asarray(a, dtype=np.float64) for a in (K, R, t))


def _intrinsics(H, W):
    return np.array([[W, 0.0, (W - 1) / 2.0], [0.0, W, (H - 1) / 2.0], [0.0, 0.0, 1.0]])


def _cameras(rng, n, H, W, poses, what):
    """n views about the reference camera: small random rotations and translations, a planar grid
    (pure translations), or an arc looking at the harmonic mean depth."""
    K = _intrinsics(H, W)
    cams = []
    if poses == "rotated":
        for _ in range(n):
            axis = rng.normal(size=3)
            axis /= np.linalg.norm(axis)
            ang = math.radians(rng.uniform(0.0, 2.0))
            S = np.array([[0, -axis[2], axis[1]], [axis[2], 0, -axis[0]], [-axis[1], axis[0], 0]])
            R = np.eye(3) + math.sin(ang) * S + (1 - math.cos(ang)) * (S @ S)
            cams.append(Camera(K, R, rng.uniform(-0.1, 0.1, size=3)))
    elif poses == "grid":
        rows = max(1, int(round(math.sqrt(n / 2.0)))) if what == "source" else max(1, int(math.sqrt(n)))
        cols = -(-n // rows)
        span = 0.3 if what == "source" else 0.1
        jx, jy = rng.uniform(-0.02, 0.02, size=2)
        for i in range(n):
            x = 0.0 if cols == 1 else -span + 2 * span * (i % cols) / (cols - 1)
            y = 0.0 if rows == 1 else (-span + 2 * span * (i // cols) / (rows - 1)) / (3.0 if what == "source" else 1.0)
            cams.append(Camera(K, np.eye(3), -np.array([x + jx, y + jy, 0.0])))
    else:  # arc
        zf = 2.0 / (1.0 / NEAR + 1.0 / FAR)
        jy = rng.uniform(-0.02, 0.02)
        for i in range(n):
            x = 0.0 if n == 1 else -0.2 + 0.4 * i / (n - 1)
            phi = math.asin(x / zf)
            C = np.array([zf * math.sin(phi), jy, zf - zf * math.cos(phi)])
            z = np.array([0.0, 0.0, zf]) - C
            z /= np.linalg.norm(z)
            ex = np.cross(np.array([0.0, 1.0, 0.0]), z)
            ex /= np.linalg.norm(ex)
            R = np.stack([ex, np.cross(z, ex), z])
            cams.append(Camera(K, R, -R @ C))
    return cams


def _rho(D):
    if D == 1:
        return np.array([1.0 / FAR])
    return 1.0 / FAR + np.arange(D) / (D - 1) * (1.0 / NEAR - 1.0 / FAR)


def _meet(ref, cam, rho, H, W):
    """Where the ray of every pixel of `cam` meets the plane of inverse depth rho (a number or a
    tensor [H, W]) in the reference image: (x, y, in front), float64."""
    f64 = dict(dtype=torch.float64, device=DEV)
    v, u = torch.meshgrid(torch.arange(H, **f64), torch.arange(W, **f64), indexing="ij")
    Rr = cam.R @ ref.R.T
    C = ref.t - Rr.T @ cam.t
    mx, my = (u - cam.K[0, 2]) / cam.K[0, 0], (v - cam.K[1, 2]) / cam.K[1, 1]
    A = Rr.T
    dx, dy, dz = (float(A[i, 0]) * mx + float(A[i, 1]) * my + float(A[i, 2]) for i in range(3))
    # C + s dir on the plane z = 1 / rho: X / Z = rho C_x + (1 - rho C_z) dir_x / dir_z
    near = 1.0 - rho * float(C[2])
    x = ref.K[0, 0] * (rho * float(C[0]) + near * dx / dz) + ref.K[0, 2]
    y = ref.K[1, 1] * (rho * float(C[1]) + near * dy / dz) + ref.K[1, 2]
    return x, y, (dz > 0) & (torch.as_tensor(near, device=DEV) > 0)


def _waves(rng, u, v, W, n, lo, hi):
    """A smooth colour field [H, W, 3]: a base and n cosines a channel."""
    out = []
    for _ in range(3):
        acc = torch.full_like(u, float(rng.uniform(0.25, 0.75)))
        for _ in range(n):
            p, ang, a, ph = rng.uniform(W / 4.0, 1.5 * W), rng.uniform(0, 2 * math.pi), rng.uniform(lo, hi), rng.uniform(0, 6.3)
            acc = acc + float(a) * torch.cos(float(2 * math.pi / p * math.cos(ang)) * u + float(2 * math.pi / p * math.sin(ang)) * v + float(ph))
        out.append(acc)
    return torch.stack(out, -1).clamp_(0.0, 1.0)


def _scene(seed, H, W, D, dtype, src=()):
    """A layered scene on D planes as an upstream network gives it: on every pixel the surface's
    plane is opaque and the next one partly so, other planes hold smooth colours, and everything
    carries noise of 0.05, clamped to [0, 1].  Returns the coarse MPI, the images of the `src`
    cameras (noise 0.01) and the reference camera."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed) + 1)
    ref = Camera(_intrinsics(H, W), np.eye(3), np.zeros(3))
    f32 = dict(dtype=torch.float32, device=DEV)
    v, u = torch.meshgrid(torch.arange(H, **f32), torch.arange(W, **f32), indexing="ij")
    inv = torch.full((H, W), float(rng.uniform(0.02, 0.08)), **f32)  # inverse depth of the surface
    colour = _waves(rng, u, v, W, 4, 0.03, 0.12)
    for _ in range(int(rng.integers(3, 9))):
        uc, vc = rng.uniform(0, W), rng.uniform(0, H)
        ru, rv, th = rng.uniform(0.08, 0.35) * W, rng.uniform(0.08, 0.35) * H, rng.uniform(0, math.pi)
        r = float(rng.uniform(0.1, 0.95))
        a = ((u - uc) * math.cos(th) + (v - vc) * math.sin(th)) / ru
        b = (-(u - uc) * math.sin(th) + (v - vc) * math.cos(th)) / rv
        hit = ((a * a + b * b) <= 1.0) & (inv < r)
        inv = torch.where(hit, r + 0.02 * a, inv)
        colour = torch.where(hit[..., None], _waves(rng, u, v, W, 3, 0.03, 0.12), colour)
    rho = _rho(D)
    inv = inv.clamp(float(rho[0]), float(rho[-1]))
    step = float(rho[1] - rho[0]) if D > 1 else 1.0
    at = ((inv - float(rho[0])) / step).clamp(0.0, max(D - 1, 1) - 1e-3)
    lo, frac = at.floor(), at - at.floor()
    M = torch.empty((D, H, W, 4), dtype=dtype, device=DEV)
    for d in range(D):
        here, above = lo == d, lo == d - 1
        on = (here | above)[..., None]
        c = torch.where(on, colour, _waves(rng, u, v, W, 2, 0.05, 0.2))
        alpha = torch.where(here, torch.ones_like(u), torch.where(above, frac, torch.zeros_like(u)))
        p = torch.cat([c, alpha[..., None]], -1)
        p += 0.05 * torch.randn(p.shape, generator=gen, **f32)
        M[d] = p.clamp_(0.0, 1.0).to(dtype)
    images = torch.empty((len(src), H, W, 3), **f32)
    for i, cam in enumerate(src):
        x, y, _ = _meet(ref, cam, inv.double(), H, W)
        grid = torch.stack([2 * x / max(W - 1, 1) - 1, 2 * y / max(H - 1, 1) - 1], -1).float()[None]
        im = torch.nn.functional.grid_sample(colour.permute(2, 0, 1)[None], grid, padding_mode="border", align_corners=True)
        images[i] = (im[0].permute(1, 2, 0) + 0.01 * torch.randn((H, W, 3), generator=gen, **f32)).clamp_(0.0, 1.0)
    return M, images, ref


def _dtype(case):
    return torch.float32 if case["dtype"] == "f32" else torch.bfloat16


def _schedule(iters):
    return (2, 1, 0) if iters == 3 else (2, 0)


def _requests(case):
    """The batched step's requests: the server's sizes, plane and view counts, at mixed levels."""
    rng = np.random.default_rng(case["mix"])
    out = []
    for i in range(case["n"]):
        f = float(rng.choice([0.25, 0.5, 0.75, 1.0]))
        H, W = max(16, int(case["Hmax"] * f) // 4 * 4), max(16, int(case["Wmax"] * f) // 4 * 4)
        out.append(dict(H=H, W=W, D=max(8, case["Dmax"] * int(rng.integers(1, 5)) // 4), N=int(rng.integers(2, case["Nmax"] + 1)),
                        k=case["k"], level=(2, 1, 0)[i % 3], poses="rotated", select="topk", prior=0.0, dtype="bf16"))
    return out


# ------------------------------------------------------------------------ prepare, run

class _NetParams:
    """Random parameters of the learned network (five 3x3x3 blocks of 32 channels)."""

    def __init__(self, seed, c_in):
        rng = np.random.default_rng(seed)
        self.eps = 1e-5
        names = ("conv_w", "conv_b", "bn_gamma", "bn_beta", "bn_mean", "bn_var")
        for n in names:
            setattr(self, n, [])
        for i in range(5):
            c = c_in if i == 0 else 32
            self.conv_w.append((rng.standard_normal((32, c, 3, 3, 3)) * math.sqrt(2.0 / (27 * c))).astype(np.float32))
            self.conv_b.append((rng.standard_normal(32) * 0.05).astype(np.float32))
            self.bn_gamma.append(rng.uniform(0.5, 1.5, 32).astype(np.float32))
            self.bn_beta.append((rng.standard_normal(32) * 0.1).astype(np.float32))
            self.bn_mean.append((rng.standard_normal(32) * 0.1).astype(np.float32))
            self.bn_var.append(rng.uniform(0.5, 2.0, 32).astype(np.float32))
        self.out_w = (rng.standard_normal((4, 32)) * math.sqrt(1.0 / 32) * 0.1).astype(np.float32)
        self.out_b = np.zeros(4, dtype=np.float32)


def _selection(case):
    return rl.SELECT_MVS if case.get("select") == "mvs" else rl.SELECT_TOPK


def _step_state(case, seed):
    H, W, D, N, k = case["H"], case["W"], case["D"], case["N"], case["k"]
    src = _cameras(np.random.default_rng(seed + 7), N, H, W, case.get("poses", "rotated"), "source")
    coarse, images, ref = _scene(seed, H, W, D, _dtype(case), src)
    level = case.get("level", 0)
    s = dict(case=case, src=src, images=images, coarse=coarse, m=rl.make_mpi(torch.empty_like(coarse), NEAR, FAR, ref))
    if case["kind"] != "volume":
        s["S"] = torch.empty((k, H >> level, W >> level), dtype=torch.uint8, device=DEV)
    if case["kind"] in ("step", "batch", "refine"):
        s["loss"] = torch.empty(case.get("iters", 1), dtype=torch.float32, device=DEV)
        s["ws"] = rl.workspace(N, D, H, W, k, coarse.dtype, DEV)
    elif case["kind"] == "learned":
        s["net"] = rl.LgdNet(_NetParams(seed + 9, 4 * N + 4), device=DEV)
        s["ws"] = torch.empty(rl.reallife_lgd_step_workspace_bytes(N, D, H, W, k, coarse.dtype), dtype=torch.uint8, device=DEV)
    else:
        s["ws"] = torch.empty(rl.reallife_gradient_volume_workspace_bytes(N, D, H, W, k, coarse.dtype), dtype=torch.uint8, device=DEV)
        s["m"] = rl.make_mpi(coarse, NEAR, FAR, ref)
        s["V"] = torch.empty((4 * N + 4, k, H >> level, W >> level), dtype=torch.float32, device=DEV)
        s["S"] = torch.empty((k, H >> level, W >> level), dtype=torch.uint8, device=DEV)
    return s


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("render", "backward"):
        H, W, D, T = case["H"], case["W"], case["D"], case["T"]
        cams = _cameras(np.random.default_rng(seed + 7), T, H, W, case["poses"], "novel")
        M, _, ref = _scene(seed, H, W, D, _dtype(case))
        s = dict(case=case, cams=cams, m=rl.make_mpi(M, NEAR, FAR, ref), ref=ref)
        if kind == "render":
            s["out"] = torch.empty((T, H, W, 3), dtype=torch.float32, device=DEV)
        else:
            gen = torch.Generator(device=DEV)
            gen.manual_seed(int(seed) + 3)
            s["M"] = M.requires_grad_(True)
            s["g"] = 0.1 * torch.randn((T, H, W, 3), generator=gen, device=DEV)
        return s
    if kind == "batch":
        items = [_step_state(dict(r, kind="batch"), seed + 101 * i) for i, r in enumerate(_requests(case))]
        table = rl.BatchTable(len(items), device=DEV)
        rl.reallife_batch_prepare([rl.BatchItem(s["m"], s["images"], s["src"], s["case"]["k"], s["ws"], s["case"]["level"],
                                                s["loss"]) for s in items], table)
        return dict(case=case, items=items, table=table)
    return _step_state(case, seed)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "render":
        return rl.reallife_render(s["m"], s["cams"], out=s["out"])
    if kind == "backward":
        views = warp_composite(s["M"], NEAR, FAR, s["ref"], s["cams"])
        (grad,) = torch.autograd.grad(views, s["M"], s["g"])
        return views.detach(), grad
    if kind == "batch":
        for it in s["items"]:
            it["m"].data.copy_(it["coarse"])
        rl.reallife_hsgd_step_batch(s["table"])
        return [(it["m"].data, it["loss"]) for it in s["items"]]
    if kind == "volume":
        return rl.reallife_gradient_volume(s["m"], s["images"], s["src"], case["k"], case["level"], V=s["V"], S_out=s["S"], ws=s["ws"])
    s["m"].data.copy_(s["coarse"])
    if kind == "step":
        rl.reallife_hsgd_step(s["m"], s["images"], s["src"], case["k"], level=case["level"], loss_out=s["loss"],
                              S_out=s["S"], ws=s["ws"], selection=_selection(case), lambda_s=case["prior"])
        return s["m"].data, s["loss"], s["S"]
    if kind == "refine":
        rl.reallife_refine(s["m"], s["images"], s["src"], case["k"], _schedule(case["iters"]), loss_per_iter=s["loss"], ws=s["ws"])
        return s["m"].data, s["loss"]
    rl.reallife_lgd_step(s["m"], s["images"], s["src"], case["k"], s["net"], case["level"], S_out=s["S"], ws=s["ws"])
    return s["m"].data, s["S"]


# -------------------------------------------------------------------------------- work

# Operations of one bilinear RGBA sample with its coordinates and weights, of its step of the over
# operator, and of its adjoint (both per view, plane and pixel).
_SAMPLE, _OVER, _ADJOINT = 46, 8, 30


def work(case):
    kind = case["kind"]
    if kind == "batch":
        both = [work(dict(r, kind="step")) for r in _requests(case)]
        return {"bytes": sum(w["bytes"] for w in both), "flops": sum(w["flops"] for w in both)}
    H, W, D = case["H"], case["W"], case["D"]
    mpi = D * H * W * 4 * (4 if case["dtype"] == "f32" else 2)
    if kind == "render":
        return {"bytes": mpi + 12 * case["T"] * H * W, "flops": case["T"] * D * H * W * (_SAMPLE + _OVER)}
    if kind == "backward":
        return {"bytes": 2 * mpi + 24 * case["T"] * H * W, "flops": case["T"] * D * H * W * (_SAMPLE + 2 * _OVER + _ADJOINT + 32)}
    N, k = case["N"], case["k"]
    images = 12 * N * H * W
    if kind == "refine":
        samples = sum(N * D * (H >> l) * (W >> l) for l in _schedule(case["iters"]))
        return {"bytes": 2 * mpi + images, "flops": samples * (_SAMPLE + 2 * _OVER + _ADJOINT)}
    level = case["level"]
    h, w = H >> level, W >> level
    if kind == "step":
        return {"bytes": 2 * mpi + images + k * h * w, "flops": N * D * h * w * (_SAMPLE + 2 * _OVER + _ADJOINT)}
    voxel = N * (4 * 12 + (4 ** level) * 30)  # one alpha weight and the children's colours a view
    flops = N * D * h * w * 24 + k * h * w * voxel
    if kind == "volume":
        return {"bytes": mpi + images + (4 * N + 4) * k * h * w * 4 + k * h * w, "flops": flops}
    net = 2 * k * h * w * (27 * 32 * (4 * N + 4 + 4 * 32) + 32 * 4)
    return {"bytes": 2 * mpi + images + k * h * w, "flops": flops + net}


# ------------------------------------------------------------------------------- exact

def _taps(x, y, ok, H, W):
    """The four taps of a bilinear sample (zero padding): (pixel index, weight) pairs."""
    x0, y0 = x.floor(), y.floor()
    fx, fy = x - x0, y - y0
    out = []
    for oy, ox, wt in ((0, 0, (1 - fx) * (1 - fy)), (0, 1, fx * (1 - fy)), (1, 0, (1 - fx) * fy), (1, 1, fx * fy)):
        xi, yi = x0 + ox, y0 + oy
        inside = ok & (xi >= 0) & (xi < W) & (yi >= 0) & (yi < H)
        idx = (yi.clamp(0, H - 1) * W + xi.clamp(0, W - 1)).long()
        out.append((idx.reshape(-1), torch.where(inside, wt, torch.zeros_like(wt)).reshape(-1, 1)))
    return out


def _gather(plane, taps):
    """Bilinear sample [pixels, C] of plane [H * W, C]."""
    return sum(wt * plane[idx] for idx, wt in taps)


def _over(M, ref, cam, rho, h, w, keep=False):
    """The composite [h * w, 3] of the MPI M (float64 [D, H, W, 4]) in view `cam`; with keep, every
    plane's sample too."""
    D, H, W = M.shape[:3]
    C = torch.zeros((h * w, 3), dtype=torch.float64, device=DEV)
    T = torch.ones((h * w, 1), dtype=torch.float64, device=DEV)
    kept = [None] * D
    for d in range(D - 1, -1, -1):
        m = _gather(M[d].reshape(H * W, 4), _taps(*_meet(ref, cam, float(rho[d]), h, w), H, W))
        C += T * m[:, 3:] * m[:, :3]
        if keep:
            kept[d] = (m, T)
        T = T * (1 - m[:, 3:])
    return C, kept


def _adjoint(M, ref, cam, rho, h, w, kept, r, G):
    """Adds the adjoint of _over for dL/dC = r [h * w, 3] to G [D, H * W, 4]."""
    D, H, W = M.shape[:3]
    B = torch.zeros((h * w, 3), dtype=torch.float64, device=DEV)
    for d in range(D):
        m, T = kept[d]
        g = torch.cat([T * m[:, 3:] * r, T * ((m[:, :3] - B) * r).sum(1, keepdim=True)], 1)
        for idx, wt in _taps(*_meet(ref, cam, float(rho[d]), h, w), H, W):
            G[d].index_add_(0, idx, wt * g)
        B = m[:, :3] * m[:, 3:] + (1 - m[:, 3:]) * B


def _at_level(cam, level):
    s = 2.0 ** -level
    K = np.array(cam.K)
    K[0, 0], K[1, 1], K[0, 2], K[1, 2] = K[0, 0] * s, K[1, 1] * s, (K[0, 2] + 0.5) * s - 0.5, (K[1, 2] + 0.5) * s - 0.5
    return Camera(K, cam.R, cam.t)


def _down(x, level):
    """Means of 2^l x 2^l blocks of x [P, H, W, C], summed row by row in x's own type."""
    if level == 0:
        return x
    s = 1 << level
    parts = [x[:, i::s, j::s] for i in range(s) for j in range(s)]
    acc = parts[0]
    for p in parts[1:]:
        acc = acc + p
    return acc * (1.0 / (s * s))


def _select(M, level, k, rule):
    """The kept planes [k, h, w] (ascending) of the stored MPI, decided on 32-bit keys."""
    a = _down(M[..., 3:].float(), level)[..., 0].to(M.dtype).float()
    D, h, w = a.shape
    keys = torch.empty_like(a)
    T = torch.ones((h, w), dtype=torch.float32, device=DEV)
    for d in range(D - 1, -1, -1):
        keys[d] = a[d] * T
        T = T * (1.0 - a[d])
    if rule == "mvs":
        best = torch.argsort(keys, dim=0, descending=True, stable=True)[0]
        start = (best - (k - 1) // 2).clamp(0, D - k)
        return start[None] + torch.arange(k, device=DEV).view(k, 1, 1)
    return torch.argsort(keys, dim=0, descending=True, stable=True)[:k].sort(0).values


def _restore(M, S, step, level):
    """M (float64 copy) with step [k, h, w, 4] added on the kept voxels, clamped to [0, 1]."""
    out = M.double()
    up = lambda t: t.repeat_interleave(1 << level, 1).repeat_interleave(1 << level, 2)  # noqa: E731
    S, step = up(S), up(step)
    for j in range(S.shape[0]):
        idx = S[j][None, ..., None].expand(1, *S.shape[1:], 4)
        out.scatter_(0, idx, (out.gather(0, idx) + step[j][None]).clamp(0.0, 1.0))
    return out


def _exact_step(s, case):
    M, level, k, N = s["coarse"], case["level"], case["k"], case["N"]
    D, h, w = case["D"], case["H"] >> level, case["W"] >> level
    rho = _rho(D)
    Ml, Il = _down(M.double(), level), _down(s["images"].double(), level)
    ref = _at_level(s["m"].ref, level)
    G = torch.zeros((D, h * w, 4), dtype=torch.float64, device=DEV)
    loss = torch.zeros((), dtype=torch.float64, device=DEV)
    for i, cam in enumerate(s["src"]):
        cam = _at_level(cam, level)
        C, kept = _over(Ml, ref, cam, rho, h, w, keep=True)
        e = C - Il[i].reshape(h * w, 3)
        loss += (e * e).sum() / (2 * N)
        _adjoint(Ml, ref, cam, rho, h, w, kept, e / N, G)
    if case["prior"]:
        a = Ml[..., 3].reshape(D, h * w)
        G[..., 3] += case["prior"] / (D * h * w) * torch.sign(0.5 - a) / (1.5 - (0.5 - a).abs())
    S = _select(M, level, k, case["select"])
    idx = S[..., None].expand(*S.shape, 4)
    step = -G.view(D, h, w, 4).gather(0, idx)
    return _restore(M, S, step, level), loss.reshape(1), S.to(torch.uint8)


def _exact_volume(s, case):
    """V [4N + 4, k, h, w] and the kept planes."""
    M, level, k, N = s["coarse"], case["level"], case["k"], case["N"]
    H, W, D, h, w = case["H"], case["W"], case["D"], case["H"] >> level, case["W"] >> level
    rho = torch.as_tensor(_rho(D), device=DEV)
    Ml = _down(M.double(), level)
    S = _select(M, level, k, "topk")
    ref, refl = s["m"].ref, _at_level(s["m"].ref, level)
    V = torch.zeros((4 * N + 4, k, h, w), dtype=torch.float64, device=DEV)

    def into(a, b, r, hh, ww):
        # pixels of camera a on the planes of inverse depth r [hh, ww], seen by camera b
        f64 = dict(dtype=torch.float64, device=DEV)
        y, x = torch.meshgrid(torch.arange(hh, **f64), torch.arange(ww, **f64), indexing="ij")
        Rr = b.R @ a.R.T
        t = b.t - Rr @ a.t
        m = [(x - a.K[0, 2]) / a.K[0, 0], (y - a.K[1, 2]) / a.K[1, 1]]
        X, Y, Z = (float(Rr[i, 0]) * m[0] + float(Rr[i, 1]) * m[1] + float(Rr[i, 2]) + r * float(t[i]) for i in range(3))
        return b.K[0, 0] * X / Z + b.K[0, 2], b.K[1, 1] * Y / Z + b.K[1, 2], Z > 0

    for i, cam in enumerate(s["src"]):
        caml = _at_level(cam, level)
        A = torch.empty((D, h * w, 1), dtype=torch.float64, device=DEV)
        T = torch.ones((h * w, 1), dtype=torch.float64, device=DEV)
        for d in range(D - 1, -1, -1):
            a = _gather(Ml[d, ..., 3].reshape(h * w, 1), _taps(*_meet(refl, caml, float(rho[d]), h, w), h, w))
            A[d] = a * T
            T = T * (1 - a)
        for j in range(k):
            r = rho[S[j]]
            base = S[j].reshape(-1) * (h * w)
            V[3 * N + i, j] = sum(wt * A.view(-1, 1)[base + idx] for idx, wt in _taps(*into(refl, caml, r, h, w), h, w)).view(h, w)
            up = r.repeat_interleave(1 << level, 0).repeat_interleave(1 << level, 1)
            img = s["images"][i].double().reshape(H * W, 3)
            V[3 * i:3 * i + 3, j] = _down(_gather(img, _taps(*into(ref, cam, up, H, W), H, W)).view(1, H, W, 3), level)[0].permute(2, 0, 1)
    V[4 * N:] = Ml.gather(0, S[..., None].expand(*S.shape, 4)).permute(3, 0, 1, 2)
    return V, S


def _exact_learned(s, case, seed):
    V, S = _exact_volume(s, case)
    p = _NetParams(seed + 9, V.shape[0])
    f = lambda a: torch.from_numpy(a).to(DEV).double()  # noqa: E731
    k, h, w = V.shape[1:]
    x = V.permute(1, 2, 3, 0)
    for i in range(5):
        g = f(p.bn_gamma[i]) / torch.sqrt(f(p.bn_var[i]) + p.eps)
        wt = f(p.conv_w[i])
        pad = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
        acc = f(p.conv_b[i]).expand(k, h, w, 32).clone()
        for a in range(3):
            for b in range(3):
                for c in range(3):
                    acc += pad[a:a + k, b:b + h, c:c + w] @ wt[:, :, a, b, c].T
        x = torch.relu((acc - f(p.bn_mean[i])) * g + f(p.bn_beta[i]))
    res = x @ f(p.out_w).T + f(p.out_b)
    return _restore(s["coarse"], S, res, case["level"]), S.to(torch.uint8)


def exact(case, seed):
    kind = case["kind"]
    if kind == "refine":
        # Every iteration selects on what the iteration before left: where two keys lie within 32-bit
        # rounding the planes kept, and with them the MPI, have no value of their own in 64 bits.
        return None
    s = prepare(case, seed)
    with torch.no_grad():
        if kind in ("render", "backward"):
            H, W, T = case["H"], case["W"], case["T"]
            rho = _rho(case["D"])
            M = s["m"].data.detach().double()
            views = torch.empty((T, H, W, 3), dtype=torch.float64, device=DEV)
            G = torch.zeros((case["D"], H * W, 4), dtype=torch.float64, device=DEV) if kind == "backward" else None
            for i, cam in enumerate(s["cams"]):
                C, kept = _over(M, s["ref"], cam, rho, H, W, keep=G is not None)
                views[i] = C.view(H, W, 3)
                if G is not None:
                    _adjoint(M, s["ref"], cam, rho, H, W, kept, s["g"][i].double().reshape(H * W, 3), G)
            return views if G is None else (views, G.view(case["D"], H, W, 4))
        if kind == "batch":
            return [_exact_step(it, it["case"])[:2] for it in s["items"]]
        if kind == "step":
            return _exact_step(s, case)
        if kind == "volume":
            V, S = _exact_volume(s, case)
            return V, S.to(torch.uint8)
        return _exact_learned(s, case, seed)
