"""Performance cases: what users of this package have it do, over the sizes,
data types and options they do it with.

``listed()`` gives the fixed cases, ``draw(rng)`` further ones of the same
ranges; ``prepare`` makes a case's inputs and the handle a program keeps,
``run`` is one pass through the public entry points, ``work`` the bytes and
operations a pass cannot do without, ``exact`` its results in 64 bits from
plain torch.

Scenes are synthetic depth maps of the kind the estimator is for: a floor, a
back wall and spheres and tilted patches in front of them (so smooth surfaces
and depth steps), sensor noise of 0.0012 z^2 m, a range of 0.4-6 m, 2 % of the
pixels without a reading, intrinsics fx = fy = 0.82 W.
"""
import math
import random

import torch

import paper_2209_08241_gb300 as nrm

# The frame sizes (W, H) of the uneven batch and their shares.
SIZES = ((320, 240), (640, 480), (1280, 720), (1920, 1080), (4096, 3072))
SHARES = (0.3, 0.3, 0.2, 0.15, 0.05)

MAX_FRAME_PX = 4096 * 3072
MAX_BATCH_PX = 64 * 1920 * 1080


def listed():
    return [
        # One camera frame as it arrives (a VGA sensor in a control loop): the
        # smallest call, where the launch and the call path count.
        dict(name="frame_vga_f32", kind="frame", w=640, h=480, dtype="f32", out="f32", alpha=2, mask="secant"),
        # One 720p frame of a 16-bit depth sensor with its organised point
        # cloud: what a mapping or registration program takes per frame.
        dict(name="points_720p_u16", kind="points", w=1280, h=720, dtype="u16", out="f32", alpha=2, mask="secant"),
        # Recorded full-HD sequences, 16-bit millimetres, in batches of 64, with
        # each of the three normal formats: float4 for geometry code,
        # half4 for networks, the octahedral code for storage.
        dict(name="batch_1080p_u16_f32", kind="batch", n=64, w=1920, h=1080, dtype="u16", out="f32", alpha=2,
             mask="secant"),
        dict(name="batch_1080p_u16_f16", kind="batch", n=64, w=1920, h=1080, dtype="u16", out="f16", alpha=2,
             mask="secant"),
        dict(name="batch_1080p_u16_oct16", kind="batch", n=64, w=1920, h=1080, dtype="u16", out="oct16", alpha=2,
             mask="secant"),
        # Frames of many cameras in one launch: 256 float32 frames of five
        # sizes, each with its own intrinsics (the largest case).
        dict(name="mix_256_f32", kind="mix", n=256, pick=3, dtype="f32", out="f32", alpha=2, mask="secant"),
        # Regions of interest cut from frames: 48 pieces of odd widths and
        # heights, whose rows are not aligned to anything; distance 1.
        dict(name="crops_48_u16", kind="crops", n=48, pick=5, dtype="u16", out="f32", alpha=1, mask="secant"),
        # A training step of a depth network with this as its loss layer:
        # forward, then the gradient of the cosine loss against target normals.
        dict(name="loss_32_vga", kind="loss", n=32, w=640, h=480, alpha=2, mask="secant"),
        # The averaged multi-scale variant, batched, single-pair form.
        dict(name="scales_pair_16_1080p_u16", kind="scales", n=16, w=1920, h=1080, dtype="u16", out="f32",
             form="pair", scales=4, mask="secant"),
        # The same in the four-direction form on one large float32 frame.
        dict(name="scales_quad_12mp_f32", kind="scales", n=1, w=4096, h=3072, dtype="f32", out="f32", form="quad",
             scales=4, mask="secant"),
        # Plane-fitting ground truth of a full-HD depth map, 25 points a pixel.
        dict(name="planefit_1080p_f32", kind="planefit", w=1920, h=1080, dtype="f32", radius=2),
        # The evaluation of a normal map against a reference: its angle images
        # and their mean squared errors.
        dict(name="evaluate_12mp", kind="evaluate", w=4096, h=3072),
    ]


def draw(rng):
    kind = rng.choice(["frame", "points", "batch", "batch", "mix", "crops", "loss", "scales", "planefit", "evaluate"])
    c = dict(kind=kind)
    if kind in ("frame", "points", "planefit", "evaluate"):
        c["w"], c["h"] = _size(rng, MAX_FRAME_PX)
    elif kind in ("batch", "loss", "scales"):
        top = MAX_BATCH_PX // (4 if kind == "scales" else 3 if kind == "loss" else 1)
        c["w"], c["h"] = _size(rng, min(MAX_FRAME_PX, top))
        c["n"] = max(1, min(round(math.exp(rng.uniform(0.0, math.log(128)))), top // (c["w"] * c["h"])))
    else:
        c["n"] = round(math.exp(rng.uniform(math.log(4), math.log(128))))
        c["pick"] = rng.randrange(1 << 20)
    if kind == "evaluate":
        return c
    if kind == "planefit":
        return c | dict(dtype=rng.choice(["f32", "u16"]), radius=rng.choice([1, 2, 2, 3, 4]))
    c["mask"] = rng.choice(["secant", "secant", "raw"])
    if kind == "loss":
        return c | dict(alpha=rng.choice([1, 2, 2, 3, 4]))
    c |= dict(dtype=rng.choice(["f32", "u16"]), out=rng.choice(["f32", "f16", "oct16"]))
    if kind == "scales":
        return c | dict(form=rng.choice(["pair", "quad"]), scales=rng.randint(2, 6))
    return c | dict(alpha=rng.choice([1, 1, 2, 2, 2, 3, 4, 8]))


def _size(rng, top):
    """A frame size from 320 x 240 up to ``top`` pixels, half of the time odd."""
    px = math.exp(rng.uniform(math.log(320 * 240), math.log(top)))
    aspect = rng.choice([4 / 3, 4 / 3, 16 / 9, 1.0, 10 / 9])
    w, h = math.sqrt(px * aspect), math.sqrt(px / aspect)
    if rng.random() < 0.5:
        return int(w) | 1, int(h) | 1
    return max(16, int(w) // 16 * 16), max(8, int(h) // 8 * 8)


def _sizes(case):
    """(W, H) of each frame of a batch."""
    if case["kind"] == "mix":
        return random.Random(case["pick"]).choices(SIZES, SHARES, k=case["n"])
    if case["kind"] == "crops":
        rng = random.Random(case["pick"])
        return [(round(math.exp(rng.uniform(math.log(64), math.log(900)))) | 1,
                 round(math.exp(rng.uniform(math.log(48), math.log(700)))) | 1) for _ in range(case["n"])]
    return [(case["w"], case["h"])] * case.get("n", 1)


def _starts(sizes):
    """Where each frame's pixels begin in a buffer that holds a whole batch
    (frames start on multiples of 512 pixels), and the buffer's pixels."""
    starts, total = [], 0
    for w, h in sizes:
        starts.append(total)
        total += (w * h + 511) // 512 * 512
    return starts, total


def _views(buffer, sizes):
    """The (H, W, ...) view of each frame in a batch's buffer."""
    return [buffer[at:at + w * h].view(h, w, *buffer.shape[1:]) for (w, h), at in zip(sizes, _starts(sizes)[0])]


def _pool(sizes, channels, dtype):
    """One zeroed buffer for a batch and its frames' views."""
    shape = (_starts(sizes)[1],) + ((channels,) if channels else ())
    buffer = torch.zeros(shape, dtype=dtype, device="cuda")
    return buffer, _views(buffer, sizes)


# ------------------------------------------------------------------ inputs


def _intrinsics(w, h):
    return (0.82 * w, 0.82 * w, (w - 1) / 2.0, (h - 1) / 2.0)


def _rays(w, h, K, dtype):
    fx, fy, cx, cy = K
    u = (torch.arange(w, device="cuda", dtype=dtype) - cx) / fx
    v = (torch.arange(h, device="cuda", dtype=dtype) - cy) / fy
    return u[None, :], v[:, None]


def _depth(w, h, seed, dtype, holes=True, noise=True):
    """One depth map (H, W) on the GPU: float32 metres or uint16 millimetres, 0 = no reading."""
    rng = random.Random(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    K = _intrinsics(w, h)
    fx, fy, cx, cy = K
    u, v = _rays(w, h, K, torch.float32)
    yaw = rng.uniform(-0.35, 0.35)
    z = rng.uniform(4.5, 6.5) / (math.cos(yaw) + math.sin(yaw) * u).expand(h, w)
    z = torch.minimum(z, torch.where(v > 0.02, 1.2 / v.clamp(min=0.02), torch.full_like(v, 1e3)))
    for i in range(rng.randint(20, 30)):
        zc, r = rng.uniform(1.2, 5.5), rng.uniform(0.1, 0.6)
        uc, vc = (rng.uniform(0, w) - cx) / fx, (rng.uniform(0, h) - cy) / fy
        reach = 1.6 * r / (zc - r)
        x0, x1 = max(0, int((uc - reach) * fx + cx)), min(w, int((uc + reach) * fx + cx) + 1)
        y0, y1 = max(0, int((vc - reach) * fy + cy)), min(h, int((vc + reach) * fy + cy) + 1)
        if x0 >= x1 or y0 >= y1:
            continue
        us, vs, part = u[:, x0:x1], v[y0:y1], z[y0:y1, x0:x1]
        if i % 2:  # a sphere around zc (uc, vc, 1)
            a = us * us + vs * vs + 1.0
            b = zc * (us * uc + vs * vc + 1.0)
            disc = b * b - a * (zc * zc * (uc * uc + vc * vc + 1.0) - r * r)
            t = torch.where(disc > 0, (b - disc.clamp(min=0).sqrt()) / a, torch.full_like(b, 1e3))
        else:      # a tilted rectangle through zc (uc, vc, 1)
            p, q = rng.uniform(-1.0, 1.0), rng.uniform(-1.0, 1.0)
            t = zc * (1.0 + p * uc + q * vc) / (1.0 + p * us + q * vs)
            away = ((us * t - uc * zc).abs() > r) | ((vs * t - vc * zc).abs() > 0.7 * r) | (t <= 0.3)
            t = torch.where(away, torch.full_like(t, 1e3), t)
        torch.minimum(part, t, out=part)
    if noise:
        z = z + 0.0012 * z * z * torch.randn((h, w), generator=gen, device="cuda")
    bad = (z < 0.4) | (z > (6.0 if holes else 100.0))
    if holes:
        bad |= torch.rand((h, w), generator=gen, device="cuda") < 0.02
    if dtype == "u16":
        return torch.where(bad, 0.0, (z * 1000.0).round().clamp(1, 65535)).to(torch.int32).to(torch.uint16)
    return torch.where(bad, 0.0, z)


def _directions(w, h, gen):
    """(H, W, 4) float32 unit vectors (fourth component 0), uniform on the sphere."""
    t = torch.randn((h, w, 4), generator=gen, device="cuda")
    t[..., 3] = 0.0
    return t / t.norm(dim=-1, keepdim=True).clamp(min=1e-6)


def _maps(w, h, seed):
    """A normal map and a reference a few degrees off it, each with its mask (masked normals are 0)."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n = _surface(_depth(w, h, seed, "f32", noise=False, holes=False).double(), _intrinsics(w, h)).float()
    ref = n + 0.05 * _directions(w, h, gen)
    ref = ref / ref.norm(dim=-1, keepdim=True)
    va = (torch.rand((h, w), generator=gen, device="cuda") > 0.05).to(torch.uint8)
    vb = (torch.rand((h, w), generator=gen, device="cuda") > 0.03).to(torch.uint8)
    return n * va[..., None], va, ref * vb[..., None], vb


def _surface(z, K):
    """(H, W, 4) unit surface normals of a depth map from central differences (borders wrap)."""
    u, v = _rays(z.shape[1], z.shape[0], K, z.dtype)
    dx = (torch.roll(z, -1, 1) - torch.roll(z, 1, 1)) * K[0]
    dy = (torch.roll(z, -1, 0) - torch.roll(z, 1, 0)) * K[1]
    n = torch.stack([-dx, -dy, 2 * z + u * dx + v * dy, torch.zeros_like(z)], -1)
    return n / n.norm(dim=-1, keepdim=True)


def _tau(case, sizes):
    """The mask threshold: the default angle statistic, or for the raw length
    (which grows with distance squared) three times that of a frontal plane at 6 m."""
    if case.get("mask") != "raw":
        return 12.0
    a = case.get("alpha") or case.get("scales", 1)
    return 3.0 * (6.0 * a / (0.82 * min(w for w, h in sizes))) ** 2


def _params(case, **kw):
    return nrm.NormalParams(alpha=case.get("alpha", 2), mask_mode=case.get("mask", "secant"),
                            tau=_tau(case, _sizes(case)), out_dtype=case.get("out", "f32"), **kw)


def prepare(case, seed):
    kind, sizes = case["kind"], _sizes(case)
    if kind == "evaluate":
        w, h = sizes[0]
        return dict(kind=kind, maps=_maps(w, h, seed), est=nrm.BatchedEstimator())
    if kind in ("frame", "points", "planefit"):
        w, h = sizes[0]
        est = nrm.NormalEstimator(_intrinsics(w, h), h, w, _params(case), in_dtype=case["dtype"])
        d = _depth(w, h, seed, case["dtype"])
        n, m = est.new_outputs()
        p = torch.empty((h, w, 4), device="cuda") if kind == "points" else None
        return dict(kind=kind, est=est, depth=d, normals=n, valid=m, points=p, radius=case.get("radius"))
    est = nrm.BatchedEstimator(_params(case))
    items = [(_depth(w, h, (seed << 10) + i, case.get("dtype", "f32"), holes=kind != "loss"), _intrinsics(w, h))
             for i, (w, h) in enumerate(sizes)]
    channels = est.params.out_channels
    normals, normal_views = _pool(sizes, channels, est.params.torch_out_dtype)
    valid, valid_views = _pool(sizes, 0, torch.uint8)
    frames, _ = est.make_frames(items, list(zip(normal_views, valid_views)))
    state = dict(kind=kind, est=est, n=len(items), frames=frames, outputs=(normals, valid), keep=[items],
                 alphas=tuple(range(1, case.get("scales", 0) + 1)), form=case.get("form"))
    if kind == "loss":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        targets = [_directions(w, h, gen) for w, h in sizes]
        grads, grad_views = _pool(sizes, 0, torch.float32)
        grad_frames, _ = est.make_grad_frames(items, targets, valid_views, grad_views)
        state |= dict(grad_frames=grad_frames, grads=grads, scale=torch.empty(len(items), device="cuda"),
                      keep=[items, targets])
    return state


def run(state):
    kind, est = state["kind"], state["est"]
    if kind == "frame":
        return est.estimate(state["depth"], state["normals"], state["valid"])
    if kind == "points":
        return (*est.estimate(state["depth"], state["normals"], state["valid"], points=state["points"]),
                state["points"])
    if kind == "planefit":
        return est.plane_fit(state["depth"], state["radius"], state["normals"], state["valid"])
    if kind == "evaluate":
        n, va, ref, vb = state["maps"]
        phi, theta = nrm.spherical_images(n, va)
        return phi, theta, nrm.angle_mse(est, n, va, ref, vb)
    if kind == "scales":
        est.run_multiscale(state["frames"], state["n"], state["alphas"], state["form"])
        return state["outputs"]
    est.run(state["frames"], state["n"])
    if kind != "loss":
        return state["outputs"]
    est.cosine_loss_scale(state["grad_frames"], state["n"], state["scale"])
    est.run_backward_scaled(state["grad_frames"], state["n"], state["scale"])
    return *state["outputs"], state["scale"], state["grads"]


def work(case):
    """Each input read once, each output written once; operations of the closed
    form, the mask and the normalisation (multi-scale: the stencil per scale;
    plane fit: the window sums and the eigenvector)."""
    kind = case["kind"]
    px = sum(w * h for w, h in _sizes(case))
    if kind == "evaluate":
        # Both maps and masks in, two angle images and three numbers out.
        return {"bytes": px * (16 + 1 + 16 + 1 + 8) + 24, "flops": px * 100}
    depth = 4 if case.get("dtype", "f32") == "f32" else 2
    if kind == "planefit":
        return {"bytes": px * (depth + 17), "flops": px * (12 * (2 * case["radius"] + 1) ** 2 + 200)}
    out = {"f32": 16, "f16": 8, "oct16": 4}[case.get("out", "f32")] + 1
    if kind == "points":
        out += 16
    if kind == "loss":
        # Depth and targets in; normals, mask, gradient and the factors out.
        return {"bytes": px * (4 + 16 + 17 + 4) + 4 * case["n"], "flops": px * 130}
    per = 40
    if kind == "scales":
        per = 26 + (17 if case["form"] == "quad" else 13) * case["scales"]
    return {"bytes": px * (depth + out), "flops": px * per}


# ------------------------------------------------------------- in 64 bits


def _shift(z, dx, dy):
    """z at (x + dx, y + dy), NaN outside the frame."""
    h, w = z.shape
    if abs(dx) >= w or abs(dy) >= h:
        return torch.full_like(z, math.nan)
    return torch.nn.functional.pad(z, (max(0, -dx), max(0, dx), max(0, -dy), max(0, dy)), value=math.nan)[
        max(0, dy):max(0, dy) + h, max(0, dx):max(0, dx) + w]


def _metres(depth):
    z = depth.to(torch.int32).double() * 0.001 if depth.dtype == torch.uint16 else depth.double()
    return torch.where((z > 0) & torch.isfinite(z), z, math.nan)


def _normals(z, K, alphas, form, mask, tau):
    """Unit normals (H, W, 3; 0 where masked) and the mask (bool)."""
    fx, fy, _, _ = K
    u, v = _rays(z.shape[1], z.shape[0], K, torch.float64)
    nx = ny = P = 0.0
    for a in alphas:
        d2, d3 = _shift(z, a, 0), _shift(z, 0, a)
        if form == "pair":
            nx = nx - a / fy * d3 * (d2 - z)
            ny = ny - a / fx * d2 * (d3 - z)
            P = P + a * a / (fx * fy) * d2 * d3
        else:
            d4, d5 = _shift(z, -a, 0), _shift(z, 0, -a)
            nx = nx - a / (4 * fy) * (d3 + d5) * (d2 - d4)
            ny = ny - a / (4 * fx) * (d2 + d4) * (d3 - d5)
            P = P + a * a / (4 * fx * fy) * (d2 + d4) * (d3 + d5)
    nx, ny, P = nx / len(alphas), ny / len(alphas), P / len(alphas)
    nz = P - u * nx - v * ny
    q = nx * nx + ny * ny + nz * nz
    keep = (q * (1 + u * u + v * v) <= tau * tau * P * P) if mask == "secant" else (q <= tau * tau)
    keep = keep & (q > 0) & (z == z)
    n = torch.stack([nx, ny, nz], -1) / q.sqrt()[..., None]
    return torch.where(keep[..., None], n, 0.0), keep


def _four(n):
    return torch.nn.functional.pad(n, (0, 1))


def _smallest(S):
    """Eigenvector of the smallest eigenvalue of symmetric 3 x 3 matrices given
    as {(i, j): tensor}, by cyclic Jacobi rotations."""
    a = dict(S)
    vec = {(i, j): torch.full_like(a[0, 0], float(i == j)) for i in range(3) for j in range(3)}
    for p, q in ((0, 1), (0, 2), (1, 2)) * 8:
        apq = a[p, q]
        theta = (a[q, q] - a[p, p]) / (2 * torch.where(apq == 0, 1.0, apq))
        t = torch.where(theta >= 0, 1.0, -1.0) / (theta.abs() + (theta * theta + 1).sqrt())
        t = torch.where(apq == 0, 0.0, t)
        c = 1 / (t * t + 1).sqrt()
        s = t * c
        a[p, p], a[q, q], a[p, q] = a[p, p] - t * apq, a[q, q] + t * apq, torch.zeros_like(apq)
        r = 3 - p - q
        rp, rq = (min(r, p), max(r, p)), (min(r, q), max(r, q))
        a[rp], a[rq] = c * a[rp] - s * a[rq], s * a[rp] + c * a[rq]
        for k in range(3):
            vec[k, p], vec[k, q] = c * vec[k, p] - s * vec[k, q], s * vec[k, p] + c * vec[k, q]
    low = torch.stack([a[0, 0], a[1, 1], a[2, 2]], -1).argmin(-1, keepdim=True)
    return torch.stack([torch.stack([vec[k, j] for j in range(3)], -1).gather(-1, low)[..., 0] for k in range(3)], -1)


def _planes(z, K, R):
    u, v = _rays(z.shape[1], z.shape[0], K, torch.float64)
    # Relative to the centre point, which keeps the sums free of cancellation.
    pts = []
    for dy in range(-R, R + 1):
        for dx in range(-R, R + 1):
            zz = _shift(z, dx, dy)
            pts.append((zz * (u + dx / K[0]) - z * u, zz * (v + dy / K[1]) - z * v, zz - z))
    n = len(pts)
    mean = [sum(p[i] for p in pts) / n for i in range(3)]
    S = {(i, j): sum((p[i] - mean[i]) * (p[j] - mean[j]) for p in pts) for i in range(3) for j in range(i, 3)}
    keep = torch.isfinite(S[0, 0] + S[1, 1] + S[2, 2])
    vec = _smallest({k: torch.where(keep, s, float(k[0] == k[1])) for k, s in S.items()})
    away = vec[..., 0] * u + vec[..., 1] * v + vec[..., 2]
    return torch.where(keep[..., None], vec * torch.where(away < 0, -1.0, 1.0)[..., None], 0.0)


def _loss_gradient(depth, K, alpha, mask, tau, target):
    """(normals, mask, scale, dL/d depth) of L = mean over valid pixels of 1 - n . t."""
    z = _metres(depth)
    _, keep = _normals(z, K, (alpha,), "quad", mask, tau)
    fill = torch.where(z == z, z, 1.0).requires_grad_()
    h, w = z.shape
    with torch.enable_grad():
        wide = torch.nn.functional.pad(fill[None, None], (alpha,) * 4, value=1.0)[0, 0]
        d2, d4 = wide[alpha:alpha + h, 2 * alpha:], wide[alpha:alpha + h, :w]
        d3, d5 = wide[2 * alpha:, alpha:alpha + w], wide[:h, alpha:alpha + w]
        u, v = _rays(w, h, K, torch.float64)
        nx = -alpha / (4 * K[1]) * (d3 + d5) * (d2 - d4)
        ny = -alpha / (4 * K[0]) * (d2 + d4) * (d3 - d5)
        nz = alpha * alpha / (4 * K[0] * K[1]) * (d2 + d4) * (d3 + d5) - u * nx - v * ny
        n = torch.stack([nx, ny, nz], -1)
        n = n / n.norm(dim=-1, keepdim=True)
        scale = -1.0 / max(int(keep.sum()), 1)
        loss = (torch.where(keep, (n * target[..., :3].double()).sum(-1), 0.0)).sum() * scale
        grad, = torch.autograd.grad(loss, fill)
    return torch.where(keep[..., None], n.detach(), 0.0), scale, grad


def _angles(n, valid):
    phi = torch.atan2(n[..., 1], n[..., 0])
    phi = torch.where(phi < 0, phi + 2 * math.pi, phi)
    theta = torch.atan2((n[..., 0] ** 2 + n[..., 1] ** 2).sqrt(), n[..., 2])
    on = valid != 0
    return torch.where(on, phi, 0.0), torch.where(on, theta, 0.0)


@torch.no_grad()
def exact(case, seed):
    kind, sizes = case["kind"], _sizes(case)
    if kind == "evaluate":
        n, va, ref, vb = _maps(*sizes[0], seed)
        (pa, ta), (pb, tb) = _angles(n.double(), va), _angles(ref.double(), vb)
        both = ((va != 0) & (vb != 0)).double()
        count = both.sum().clamp(min=1)
        mse = torch.stack([((ta - tb) ** 2 * both).sum() / count, ((pa - pb) ** 2 * both).sum() / count, both.sum()])
        return pa, ta, mse
    tau = _tau(case, sizes)
    if kind in ("frame", "points", "planefit"):
        w, h = sizes[0]
        K = _intrinsics(w, h)
        z = _metres(_depth(w, h, seed, case["dtype"]))
        if kind == "planefit":
            return _four(_planes(z, K, case["radius"])), None
        # (The octahedral codes are whole numbers: no value in 64 bits.)
        n = None if case["out"] == "oct16" else _four(_normals(z, K, (case["alpha"],), "quad", case["mask"], tau)[0])
        if kind == "frame":
            return None if n is None else (n, None)
        u, v = _rays(w, h, K, torch.float64)
        zz = torch.where(z == z, z, 0.0)
        return n, None, torch.stack([zz * u, zz * v, zz, torch.zeros_like(zz)], -1)
    if kind != "loss" and case["out"] == "oct16":
        return None
    normals, normal_views = _pool(sizes, 4, torch.float64)
    if kind == "loss":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        grads, grad_views = _pool(sizes, 0, torch.float64)
        scale = torch.zeros(case["n"], dtype=torch.float64, device="cuda")
        for i, (w, h) in enumerate(sizes):
            n, scale[i], grad_views[i][:] = _loss_gradient(
                _depth(w, h, (seed << 10) + i, "f32", holes=False), _intrinsics(w, h), case["alpha"], case["mask"],
                tau, _directions(w, h, gen))
            normal_views[i][..., :3] = n
        return normals, None, scale, grads
    alphas = tuple(range(1, case["scales"] + 1)) if kind == "scales" else (case["alpha"],)
    for i, (w, h) in enumerate(sizes):
        z = _metres(_depth(w, h, (seed << 10) + i, case["dtype"]))
        normal_views[i][..., :3], _ = _normals(z, _intrinsics(w, h), alphas, case.get("form", "quad"), case["mask"], tau)
    return normals, None
