"""The work that a user of this library has it do, as cases that can be timed and compared.

Each case is one call (or the pair of calls that belong together) of the Python API on a synthetic
scene: Gaussians in anisotropic clusters seen by a calibrated rig, with the sizes of the
repository's workloads (paper_2604_17155_gb300/workloads.py), of its tests, or in between. Inputs
are drawn on the GPU from the seed alone and never with the library: the targets are views of one
smooth 3D field, so that they agree between cameras as photographs of one scene do.

exact() restates the method (projection, depth order, blending, normal equations, solve, adjoint) in
64-bit torch for the cases small enough for it.
"""
from __future__ import annotations

import math

import numpy as np
import torch

_DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}


def _case(name, kind, n, cams, width, height, degree, channels, dtype, fov=50.0, content="rgb", precision="mixed", sets=1,
          scale=-4.5, radius=None):
    """One case. radius: of the scene; by default the density of the repository's cluster scenes."""
    c = dict(kind=kind, n=n, cams=cams, width=width, height=height, degree=degree, channels=channels, dtype=dtype, fov=fov,
             content=content, precision=precision, sets=sets, scale=scale,
             radius=float(radius if radius is not None else 4.0 * (n / 2e5) ** (1.0 / 3.0)))
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # A thousand Gaussians, eight thumbnails, one FP32 colour each: the interactive or unit-sized
        # call, where launches and the host count.
        _case("tiny_plain", "colorize", 1000, 8, 128, 128, 0, 3, "f32", precision="plain", scale=-3.5, radius=1.0),
        # One novel view of a captured object: what a viewer draws after colorizing.
        _case("render_view", "render", 200_000, 1, 800, 800, 3, 3, "f32", fov=45.0, radius=4.0),
        # The repository's relighting workload: photographs of an object under one light, degree-3 colour.
        _case("relight", "colorize", 200_000, 100, 800, 800, 3, 3, "f32", fov=45.0, radius=4.0),
        # Several lightings of one geometry with a shared factorisation (RGB each, degree 3).
        _case("relight_sets", "sets", 100_000, 48, 640, 480, 3, 3, "f32", sets=3),
        # One refinement step on the relighting workload (render, residuals, update).
        _case("refine_step", "refine", 200_000, 100, 800, 800, 3, 3, "f32", fov=45.0, radius=4.0),
        # A training step through the colorization: coefficients, then the gradients of a loss on them
        # with respect to targets and opacities.
        _case("train_step", "train", 100_000, 40, 800, 800, 3, 3, "f32", fov=45.0),
        # Views of the whole rig from given coefficients (evaluation of a colorized scene).
        _case("render_rig", "render", 200_000, 100, 800, 800, 3, 3, "f32", fov=45.0, radius=4.0),
        # Feature enrichment: 64 BF16 feature channels on a million Gaussians.
        _case("features", "colorize", 1_000_000, 150, 1000, 750, 0, 64, "bf16", fov=60.0, content="features", radius=6.0),
        # Large segmentation: one-hot masks of 16 classes on three million Gaussians.
        _case("masks", "colorize", 3_000_000, 200, 1600, 1060, 0, 16, "f16", fov=55.0, content="masks", radius=10.0),
        # The colour pass of the same large scene: degree-3 RGB in two camera passes.
        _case("large_rgb", "colorize", 3_000_000, 200, 1600, 1060, 3, 3, "f32", fov=55.0, radius=10.0),
        # One rank's share of a camera-sharded job, packed sums and solve, at odd sizes and 5 channels
        # (RGB with two material maps), degree 2.
        _case("shard_odd", "shard", 30_011, 37, 333, 217, 2, 5, "f32"),
        # Masks held in page-locked host memory (21 classes, odd width), results back on the host.
        _case("masks_host", "host", 120_000, 48, 641, 427, 0, 21, "f16", content="masks"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same kinds, between the listed extremes in every size."""
    kind = rng.choice(["colorize", "colorize", "colorize", "colorize", "sets", "refine", "train", "render", "shard", "host"])
    fov = round(rng.uniform(40.0, 65.0), 1)
    content = rng.choice(["rgb", "rgb", "masks", "features"]) if kind in ("colorize", "host") else "rgb"
    if content == "rgb":
        degree = rng.choice([0, 1, 2, 3, 3, 3])
        channels = rng.choice([3, 3, 3, 1, 2, 4, 5, 7])
        dtype = rng.choice(["f32", "f32", "f16", "bf16"])
    else:
        degree = 0
        channels = rng.choice([16, 21, 33, 64]) if content == "features" else rng.choice([16, 16, 19, 30])
        dtype = "bf16" if content == "features" else "f16"
    n = _log(rng, 1000, 2_000_000)
    # a fit of degree L takes at least a few more views than its (L+1)^2 coefficients
    cams = _log(rng, 1 if kind == "render" else (2, 8, 16, 24)[degree], 200)
    width = rng.randint(100, 1600)
    height = max(64, int(width * rng.uniform(0.55, 1.0)))
    sets = rng.choice([2, 3, 4]) if kind == "sets" else 1
    # below the largest listed cases in pairs, walked pixels, target bytes and per-camera sums
    walks = {"train": 3, "refine": 2}.get(kind, sets)
    channels_all = channels * sets
    while (n * cams * walks > 4e8 or width * height * cams * walks > 3e8 or width * height * cams * channels_all > 3e9
           or (degree and n * cams * (1 + channels_all) > 1.2e9)):
        if cams > 36:
            cams = cams * 2 // 3
        elif width * height * cams * max(walks, 0.1 * channels_all) > 3e8:
            width, height = width * 4 // 5, height * 4 // 5
        else:
            n = max(1000, n // 2)
    precision = "plain" if rng.random() < 0.15 else "mixed"
    return _case(None, kind, n, cams, width, height, degree, channels, dtype, fov, content, precision, sets)


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
def _gen(seed, stream):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1_000_003 + stream) % (1 << 62))
    return g


def _scene(case, seed):
    """means, scales, quaternions, opacities [float32, CUDA]: a mixture of anisotropic clusters inside
    a ball, as workloads.cluster_scene draws it."""
    n, radius = case["n"], case["radius"]
    s = radius / 4.0
    g = _gen(seed, 1)
    k = 40
    d = torch.randn((k, 3), generator=g, device="cuda", dtype=torch.float64)
    u = torch.rand((k, 1), generator=g, device="cuda", dtype=torch.float64)
    centres = d / d.norm(dim=1, keepdim=True) * (3.0 * s) * u ** (1.0 / 3.0)
    stds = (0.1 + 0.7 * torch.rand((k, 3), generator=g, device="cuda", dtype=torch.float64)) * s
    q = torch.randn((k, 4), generator=g, device="cuda", dtype=torch.float64)
    axes = _rotations(q)
    means = torch.empty((n, 3), device="cuda", dtype=torch.float32)
    filled = 0
    while filled < n:
        m = 2 * (n - filled) + 64
        cid = torch.randint(0, k, (m,), generator=g, device="cuda")
        local = torch.randn((m, 3), generator=g, device="cuda", dtype=torch.float64) * stds[cid]
        p = centres[cid] + (axes[cid] @ local[:, :, None])[:, :, 0]
        p = p[p.norm(dim=1) <= radius][: n - filled].float()
        means[filled:filled + len(p)] = p
        filled += len(p)
    scales = torch.exp(case["scale"] + 0.5 * torch.randn((n, 3), generator=g, device="cuda"))
    quats = torch.randn((n, 4), generator=g, device="cuda")
    opacity = torch.sigmoid(0.5 + 2.0 * torch.randn(n, generator=g, device="cuda"))
    return means, scales, quats, opacity


def _rotations(q):
    w, x, y, z = (q / q.norm(dim=-1, keepdim=True)).unbind(-1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], -1).reshape(q.shape[:-1] + (3, 3))


def _rig(case):
    """Cameras at Fibonacci points of the upper hemisphere, looking at the origin: intrinsics [C,4] and
    world-to-camera [C,3,4] (float32)."""
    c, r = case["cams"], 1.5 * case["radius"]
    golden = math.pi * (3.0 - math.sqrt(5.0))
    f = case["width"] / 2.0 / math.tan(math.radians(case["fov"]) / 2.0)
    poses = np.empty((c, 3, 4))
    for k in range(c):
        z = 1.0 - (k + 0.5) / c
        rho = math.sqrt(1.0 - z * z)
        p = r * np.array([rho * math.cos(k * golden), rho * math.sin(k * golden), z])
        fwd = -p / np.linalg.norm(p)
        up = np.array([0.0, 0.0, 1.0]) if abs(fwd[2]) < 0.999 else np.array([0.0, 1.0, 0.0])
        right = np.cross(fwd, up)
        right /= np.linalg.norm(right)
        rot = np.stack([right, np.cross(fwd, right), fwd])
        poses[k, :, :3] = rot
        poses[k, :, 3] = -rot @ p
    intr = np.tile(np.array([f, f, case["width"] / 2.0, case["height"] / 2.0]), (c, 1))
    return intr.astype(np.float32), poses.astype(np.float32)


def _targets(case, seed, stream, intr, poses):
    """[C,H,W,K] on the GPU: each pixel shows a smooth 3D field at the point of its ray nearest to the
    scene's centre. rgb: values in [0,1] with some dependence on the view; masks: one-hot of the
    nearest of K seeds (Voronoi cells); features: unit-variance random Fourier features."""
    cams, w, h, k = case["cams"], case["width"], case["height"], case["channels"]
    g = _gen(seed, stream)
    radius = case["radius"]
    out = torch.empty((cams, h, w, k), dtype=_DTYPES[case["dtype"]], device="cuda")
    freq = torch.randn((3, k), generator=g, device="cuda") * (3.0 / radius)
    freq2 = torch.randn((3, k), generator=g, device="cuda") * (8.0 / radius)
    phase = torch.rand(k, generator=g, device="cuda") * (2.0 * math.pi)
    view = torch.randn((3, k), generator=g, device="cuda") * 0.1
    seeds = torch.randn((k, 3), generator=g, device="cuda")
    seeds = seeds / seeds.norm(dim=1, keepdim=True) * (0.8 * radius * torch.rand((k, 1), generator=g, device="cuda") ** (1.0 / 3.0))
    fx, fy, cx, cy = (float(v) for v in intr[0])
    x = (torch.arange(w, device="cuda") + 0.5 - cx) / fx
    y = (torch.arange(h, device="cuda") + 0.5 - cy) / fy
    rays = torch.stack([x[None, :].expand(h, w), y[:, None].expand(h, w), torch.ones((h, w), device="cuda")], -1)
    rays = (rays / rays.norm(dim=-1, keepdim=True)).reshape(-1, 3)
    pose = torch.from_numpy(poses).cuda()
    for j in range(cams):
        rot, t = pose[j, :, :3], pose[j, :, 3]
        eye = -(rot.T @ t)
        d = rays @ rot
        p = eye - (d @ eye)[:, None] * d
        if case["content"] == "rgb":
            v = 0.5 + 0.22 * torch.cos(p @ freq + phase) + 0.12 * torch.cos(p @ freq2 - phase) + d @ view
            out[j] = v.clamp_(0.0, 1.0).reshape(h, w, k)
        elif case["content"] == "masks":
            label = ((seeds * seeds).sum(1) - 2.0 * (p @ seeds.T)).argmin(1)
            out[j] = torch.zeros((h * w, k), dtype=out.dtype, device="cuda").scatter_(1, label[:, None], 1.0).reshape(h, w, k)
        else:
            out[j] = (math.sqrt(2.0) * torch.cos(p @ freq + phase)).reshape(h, w, k)
    return out


def _coefficients(case, seed):
    """Degree-L coefficients of plausible colours: DC in [0, 1] / Y_0 and small higher bands."""
    g = _gen(seed, 7)
    b = (case["degree"] + 1) ** 2
    c = 0.1 * torch.randn((case["n"], b, case["channels"]), generator=g, device="cuda")
    c[:, 0] = torch.rand((case["n"], case["channels"]), generator=g, device="cuda") * math.sqrt(4.0 * math.pi)
    return c


def _loss_weights(case, seed):
    return torch.randn((case["n"], (case["degree"] + 1) ** 2, case["channels"]), generator=_gen(seed, 8), device="cuda")


def prepare(case, seed):
    from paper_2604_17155_gb300 import icgs

    means, scales, quats, opacity = _scene(case, seed)
    intr, poses = _rig(case)
    s = dict(case=case, icgs=icgs, scene=icgs.Scene(means, scales, quats, opacity),
             cams=icgs.Cameras(case["width"], case["height"], intr, poses.reshape(-1, 12)))
    kind = case["kind"]
    if kind == "render":
        s["coeffs"] = _coefficients(case, seed)
        return s
    s["targets"] = [_targets(case, seed, 20 + k, intr, poses) for k in range(case["sets"])]
    if kind == "host":
        s["targets"] = [t.cpu().pin_memory() for t in s["targets"]]
        # the caller's page-locked result buffers, reused from call to call
        b = (case["degree"] + 1) ** 2
        s["out"] = (torch.empty((case["n"], b, case["channels"]), pin_memory=True),
                    torch.empty((case["n"],), dtype=torch.uint8, pin_memory=True))
    elif kind == "train":
        s["targets"][0].requires_grad_(True)
        s["opacity"] = opacity.clone().requires_grad_(True)
        s["loss_weights"] = _loss_weights(case, seed)
    elif kind == "refine":
        # the coefficients and solve records of the single shot, which a refinement starts from
        coeffs, _, record = icgs.colorize(s["scene"], s["cams"], s["targets"][0], case["degree"], precision=case["precision"])
        s["coeffs"], s["record"] = coeffs, record
    return s


def run(s):
    case, icgs, scene, cams = s["case"], s["icgs"], s["scene"], s["cams"]
    degree, precision, kind = case["degree"], case["precision"], case["kind"]
    if kind == "render":
        return icgs.render(scene, cams, s["coeffs"], degree)
    targets = s["targets"]
    if kind == "colorize":
        return icgs.colorize(scene, cams, targets[0], degree, precision=precision)
    if kind == "sets":
        return icgs.colorize_sets(scene, cams, targets, degree, precision=precision)[:3]
    if kind == "host":
        return icgs.colorize_host(scene, cams, targets[0], degree, precision=precision, coeffs_out=s["out"][0],
                                  status_out=s["out"][1])
    if kind == "refine":
        return icgs.colorize_refine(scene, cams, targets[0], degree, s["coeffs"].clone(), s["record"], 1, precision=precision)
    if kind == "train":
        c = icgs.colorize_differentiable(scene, cams, targets[0], s["opacity"], degree, precision=precision)
        loss = (s["loss_weights"] * c * c).sum()
        grad_targets, grad_opacity = torch.autograd.grad(loss, (targets[0], s["opacity"]))
        return c, grad_targets, grad_opacity
    sums = icgs.accumulate(scene, cams, targets[0], degree, precision=precision)
    return (sums,) + icgs.solve(sums, degree, precision=precision)


def work(case):
    """Bytes: scene, targets and results once. Operations: the contributing (pixel, Gaussian) pairs --
    each Gaussian's footprint, at most the about 48 a pixel blends before it is opaque -- times the
    weight and its sums, and the normal equations and solves."""
    n, cams, k, b = case["n"], case["cams"], case["channels"] * case["sets"], (case["degree"] + 1) ** 2
    pixels = case["width"] * case["height"] * cams
    item = 4 if case["dtype"] == "f32" else 2
    f = case["width"] / 2.0 / math.tan(math.radians(case["fov"]) / 2.0)
    sigma2 = (f * math.exp(case["scale"]) / (1.5 * case["radius"])) ** 2 * 1.1 + 0.3
    pairs = min(10.0 * math.pi * sigma2 * n * cams, 48.0 * pixels)
    tri = b * (b + 1) // 2
    scene, targets, coeffs, record = 44 * n, pixels * k * item, 4 * n * b * k, 12 * n * tri
    blend = pairs * (15 + 2 * (1 + k))
    fold = 2.0 * n * cams * (tri + b * k) if b > 1 else 0.0
    solve = n * (b ** 3 / 3.0 + 2.0 * b * b * k)
    kind = case["kind"]
    if kind == "render":
        return {"bytes": scene + coeffs + pixels * k * 4, "flops": pairs * (15 + 2 * k) + 2.0 * n * cams * b * k}
    if kind == "refine":
        return {"bytes": scene + targets + 2 * coeffs + record, "flops": 2 * blend + fold + solve}
    if kind == "train":
        return {"bytes": scene + 2 * targets + pixels * k * 4 + 2 * coeffs + record, "flops": 3 * blend + fold + 3 * solve}
    if kind == "shard":
        return {"bytes": scene + targets + 16 * n * (tri + b * k + 1) + coeffs + record + n, "flops": blend + fold + solve}
    return {"bytes": scene + targets + coeffs + n + (0 if kind == "host" else record), "flops": blend + fold + solve}


# ------------------------------------------------------------------------------------------
# the method in 64 bits
# ------------------------------------------------------------------------------------------
_TILE, _NEAR, _ALPHA_MIN, _ALPHA_MAX, _T_MIN, _LAMBDA = 16, 0.2, 1.0 / 255.0, 0.99, 1e-4, (1e-5, 1e-4, 1e-3, 1e-2)


def _sh(d, degree):
    """Real orthonormal harmonics of unit directions [n,3], index l*l + l + m."""
    x, y, z = d.unbind(1)
    out = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    if degree > 0:
        c = math.sqrt(3 / (4 * math.pi))
        out += [c * y, c * z, c * x]
    if degree > 1:
        c = math.sqrt(15 / math.pi)
        out += [c / 2 * x * y, c / 2 * y * z, math.sqrt(5 / math.pi) / 4 * (3 * z * z - 1), c / 2 * x * z, c / 4 * (x * x - y * y)]
    if degree > 2:
        a, b, c = math.sqrt(35 / (2 * math.pi)) / 4, math.sqrt(105 / math.pi), math.sqrt(21 / (2 * math.pi)) / 4
        out += [a * y * (3 * x * x - y * y), b / 2 * x * y * z, c * y * (5 * z * z - 1), math.sqrt(7 / math.pi) / 4 * z * (5 * z * z - 3),
                c * x * (5 * z * z - 1), b / 4 * z * (x * x - y * y), a * x * (x * x - 3 * y * y)]
    return torch.stack(out, 1)


def _project(case, scene, intr, pose):
    """Visible Gaussians of one camera: index, mean, conic, opacity, depth key, tile rectangle."""
    means, scales, quats, opacity = (t.double() for t in scene)
    w, h = case["width"], case["height"]
    fx, fy, cx, cy = (float(v) for v in intr)
    pose32 = torch.from_numpy(np.ascontiguousarray(pose)).cuda()
    rot, tr = pose32[:, :3].double(), pose32[:, 3].double()
    key = tr[2].expand(len(means))  # the depth key: three float32 fused multiply-adds
    for a in range(3):
        key = (rot[2, a] * means[:, a] + key).float().double()
    cam = means @ rot.T + tr
    zx, zy = cam[:, 0] / cam[:, 2], cam[:, 1] / cam[:, 2]
    limx, limy = 1.3 * w / 2 / fx, 1.3 * h / 2 / fy
    ux, uy, iz = zx.clamp(-limx, limx), zy.clamp(-limy, limy), 1 / cam[:, 2]
    zero = torch.zeros_like(iz)
    jac = torch.stack([fx * iz, zero, -fx * ux * iz, zero, fy * iz, -fy * uy * iz], 1).reshape(-1, 2, 3)
    p = (jac @ rot) @ (_rotations(quats) * scales[:, None, :])
    cov = p @ p.transpose(1, 2)
    a, b, c = cov[:, 0, 0] + 0.3, cov[:, 0, 1], cov[:, 1, 1] + 0.3
    det = a * c - b * b
    mx, my = fx * zx + cx, fy * zy + cy
    reach = 2 * torch.log(255 * opacity)
    hx, hy = torch.sqrt(reach.clamp_min(0) * a) + 1e-6, torch.sqrt(reach.clamp_min(0) * c) + 1e-6
    x0, x1 = torch.ceil(mx - hx - 0.5).clamp_min(0), torch.floor(mx + hx - 0.5).clamp_max(w - 1)
    y0, y1 = torch.ceil(my - hy - 0.5).clamp_min(0), torch.floor(my + hy - 0.5).clamp_max(h - 1)
    ok = (key > _NEAR) & (255 * opacity >= 1) & (x0 <= x1) & (y0 <= y1)
    idx = ok.nonzero()[:, 0]
    conic = torch.stack([c / det, -b / det, a / det], 1)
    rect = torch.stack([x0, y0, x1, y1], 1)[idx].long() // _TILE
    return idx, torch.stack([mx, my], 1)[idx], conic[idx], opacity[idx], key[idx], rect


def _tiles(case, scene, intr, pose):
    """Blend weights of one camera, tile chunk by tile chunk: yields (Gaussian index [t,m], pixel index
    [t,256] (-1 outside), w, T before, alpha, exp(-q/2), all [t,m,256])."""
    w, h = case["width"], case["height"]
    idx, mean, conic, opacity, key, rect = _project(case, scene, intr, pose)
    if not len(idx):
        return
    tx = -(-w // _TILE)
    nx, ny = rect[:, 2] - rect[:, 0] + 1, rect[:, 3] - rect[:, 1] + 1
    order = torch.sort(key, stable=True).indices
    who = torch.repeat_interleave(order, (nx * ny)[order])
    first = torch.cumsum((nx * ny)[order], 0) - (nx * ny)[order]
    k = torch.arange(len(who), device="cuda") - torch.repeat_interleave(first, (nx * ny)[order])
    tile = (rect[who, 1] + k // nx[who]) * tx + rect[who, 0] + k % nx[who]
    by_tile = torch.sort(tile, stable=True)
    who, tile = who[by_tile.indices], by_tile.values
    ids, counts = torch.unique_consecutive(tile, return_counts=True)
    starts = torch.cumsum(counts, 0) - counts
    size = torch.sort(counts)
    ids, counts, starts = ids[size.indices], size.values, starts[size.indices]
    lens = counts.tolist()
    px = torch.arange(_TILE * _TILE, device="cuda")
    at = 0
    while at < len(lens):
        end = at + 1
        while end < len(lens) and (end + 1 - at) * lens[end] * 256 <= 24_000_000:
            end += 1
        m = lens[end - 1]
        slot = torch.arange(m, device="cuda")
        valid = slot[None] < counts[at:end, None]
        g = who[(starts[at:end, None] + slot[None]).clamp_max(len(who) - 1)]
        x = (ids[at:end] % tx * _TILE)[:, None] + px % _TILE
        y = (ids[at:end] // tx * _TILE)[:, None] + px // _TILE
        inside = (x < w) & (y < h)
        dx = x[:, None, :] + 0.5 - mean[g, 0][:, :, None]
        dy = y[:, None, :] + 0.5 - mean[g, 1][:, :, None]
        q = conic[g, 0][:, :, None] * dx * dx + 2 * conic[g, 1][:, :, None] * dx * dy + conic[g, 2][:, :, None] * dy * dy
        e = torch.exp(-0.5 * q)
        alpha = (opacity[g][:, :, None] * e).clamp_max(_ALPHA_MAX)
        ok = (alpha >= _ALPHA_MIN) & valid[:, :, None] & inside[:, None, :]
        after = torch.cumprod(torch.where(ok, 1 - alpha, 1.0), 1)
        before = torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
        weight = torch.where(ok & (after >= _T_MIN), alpha * before, 0.0)
        yield idx[g], torch.where(inside, y * w + x, -1), weight, before, alpha, e
        at = end


def _directions(means, pose, degree):
    rot, t = torch.from_numpy(np.ascontiguousarray(pose)).cuda().double().split([3, 1], 1)
    d = means.double() + (rot.T @ t)[:, 0]
    return _sh(d / d.norm(dim=1, keepdim=True), degree)


def _pixels(img, at):
    """Pixels [t,256] of one image [H,W,K] as float64; zero outside."""
    flat = img.reshape(-1, img.shape[-1])
    return torch.where((at >= 0)[:, :, None], flat[at.clamp_min(0)].double(), 0.0)


def _cholesky(a):
    b = a.shape[1]
    low = torch.zeros_like(a)
    for j in range(b):
        v = a[:, j:, j] - (low[:, j:, :j] @ low[:, j, :j, None])[:, :, 0]
        low[:, j:, j] = v / torch.sqrt(v[:, :1])
    return low


def _solve(low, rhs):
    b = low.shape[1]
    y = rhs.clone()
    for i in range(b):
        y[:, i] = (y[:, i] - (low[:, i, None, :i] @ y[:, :i])[:, 0]) / low[:, i, i, None]
    for i in reversed(range(b)):
        y[:, i] = (y[:, i] - (low[:, None, i + 1:, i] @ y[:, i + 1:])[:, 0]) / low[:, i, i, None]
    return y


def _normal(case, scene, intr, poses, images, gram=True):
    """G [n,B,B], b [n,B,K], w [n] over the rig; images(j) gives camera j's target image."""
    n, degree = case["n"], case["degree"]
    b = (degree + 1) ** 2
    big = torch.zeros((n, b, b) if gram else (0, b, b), dtype=torch.float64, device="cuda")
    rhs, wsum = None, torch.zeros(n, dtype=torch.float64, device="cuda")
    for j in range(case["cams"]):
        img = images(j)
        k = img.shape[-1]
        sums = torch.zeros((n, 1 + k), dtype=torch.float64, device="cuda")
        for g, at, weight, _, _, _ in _tiles(case, scene, intr[j], poses[j]):
            t = _pixels(img, at)
            t = torch.cat([torch.ones_like(t[:, :, :1]), t], 2)
            sums.index_add_(0, g.reshape(-1), (weight @ t).reshape(-1, 1 + k))
        y = _directions(scene[0], poses[j], degree)
        if gram:
            big += (sums[:, 0, None] * y)[:, :, None] * y[:, None, :]
        more = y[:, :, None] * sums[:, None, 1:]
        rhs = more if rhs is None else rhs.add_(more)
        wsum += sums[:, 0]
    return big, rhs, wsum


def _factor(case, big, wsum):
    lam = torch.tensor([_LAMBDA[l] for l in range(case["degree"] + 1) for _ in range(2 * l + 1)], dtype=torch.float64, device="cuda")
    a = big + wsum[:, None, None] * torch.diag(lam)
    seen = wsum > 0
    a = torch.where(seen[:, None, None], a, torch.eye(a.shape[1], dtype=torch.float64, device="cuda"))
    return _cholesky(a), lam, seen


def _render(case, scene, intr, pose, coeffs):
    colour = (_directions(scene[0], pose, case["degree"])[:, :, None] * coeffs.double()).sum(1)
    img = torch.zeros((case["height"] * case["width"], coeffs.shape[2]), dtype=torch.float64, device="cuda")
    for g, at, weight, _, _, _ in _tiles(case, scene, intr, pose):
        v = (weight.transpose(1, 2) @ colour[g]).reshape(-1, coeffs.shape[2])
        at = at.reshape(-1)
        img[at[at >= 0]] = v[at >= 0]
    return img.reshape(case["height"], case["width"], -1)


def _evaluations(case):
    """Roughly, the (pixel, listed Gaussian) evaluations that exact() takes."""
    f = case["width"] / 2.0 / math.tan(math.radians(case["fov"]) / 2.0)
    side = 2 * math.sqrt(10.0 * ((f * math.exp(case["scale"]) / (1.5 * case["radius"])) ** 2 * 1.1 + 0.3)) / _TILE + 1
    passes = {"refine": 3, "train": 2.5, "sets": case["sets"]}.get(case["kind"], 1)
    return 256.0 * case["n"] * case["cams"] * side * side * passes * (1 + case["channels"] / 16.0)


def exact(case, seed):
    kind, degree = case["kind"], case["degree"]
    if _evaluations(case) > 6e10 or case["n"] * case["cams"] * (degree + 1) ** 4 > 2e10:
        return None
    scene = _scene(case, seed)
    intr, poses = _rig(case)
    if kind == "render":
        coeffs = _coefficients(case, seed)
        return torch.stack([_render(case, scene, intr[j], poses[j], coeffs) for j in range(case["cams"])])
    sets = [_targets(case, seed, 20 + k, intr, poses) for k in range(case["sets"])]
    big, rhs, wsum = _normal(case, scene, intr, poses, lambda j: torch.cat([t[j] for t in sets], -1))
    low, lam, seen = _factor(case, big, wsum)
    c = torch.where(seen[:, None, None], _solve(low, rhs), 0.0)
    if kind == "host":
        return c, None
    if kind in ("colorize", "sets"):
        return c, None, None
    if kind == "shard":
        i = torch.triu_indices(big.shape[1], big.shape[1])
        return torch.cat([big[:, i[0], i[1]], rhs.reshape(len(c), -1), wsum[:, None]], 1), c, None, None
    if kind == "refine":
        def residual(j):
            return sets[0][j].double() - _render(case, scene, intr[j], poses[j], c)
        _, res, _ = _normal(case, scene, intr, poses, residual, gram=False)
        step = _solve(low, res - wsum[:, None, None] * lam[None, :, None] * c)
        return torch.where(seen[:, None, None], c + step, 0.0)
    # train: L = sum r c^2; u = A^-1 dL/dc, dL/dS_j = Y_j^T u, dL/dV_j = -u (Y_j Y_j^T + Lambda) c
    u = torch.where(seen[:, None, None], _solve(low, 2.0 * _loss_weights(case, seed).double() * c), 0.0)
    reg = (u * lam[None, :, None] * c).sum((1, 2))
    grad_o = torch.zeros(case["n"], dtype=torch.float64, device="cuda")
    grad_t = torch.zeros(tuple(sets[0].shape), dtype=torch.float64, device="cuda")
    for j in range(case["cams"]):
        y = _directions(scene[0], poses[j], degree)
        a = (y[:, :, None] * u).sum(1)
        beta = -(a * (y[:, :, None] * c).sum(1)).sum(1) - reg
        flat = grad_t[j].reshape(-1, grad_t.shape[-1])
        for g, at, weight, before, alpha, e in _tiles(case, scene, intr[j], poses[j]):
            v = (weight.transpose(1, 2) @ a[g]).reshape(-1, a.shape[1])
            pix = at.reshape(-1)
            flat[pix[pix >= 0]] = v[pix >= 0]
            gain = a[g] @ _pixels(sets[0][j], at).transpose(1, 2) + beta[g][:, :, None]
            part = torch.cumsum(gain * weight, 1)
            d = gain * before - (part[:, -1:] - part) / (1 - alpha)
            d = torch.where((weight > 0) & (alpha < _ALPHA_MAX), d * e, 0.0)
            grad_o.index_add_(0, g.reshape(-1), d.sum(2).reshape(-1))
    return c, grad_t, grad_o
