"""The work this framework is used for, as timed cases.

A light-field program segments its views (SLIC), estimates planes and depth
maps frame by frame (cold, warm-started, batched, from host memory), or drives
the stages itself (sweep, iteration, rasterisation, fusion, superpixel
statistics).  Each case is one such call through the Python binding of the C
ABI; the sizes are those of the repository's workload configurations, or
smaller and odd ones between them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1812_06856_gb300 import lfd, synth

DTYPES = {"rgba8": torch.uint8, "f16": torch.float16, "bf16": torch.bfloat16, "f32": torch.float32}
TEXEL_BYTES = {"rgba8": 4, "f16": 8, "bf16": 8, "f32": 16}
D_MIN, D_MAX = 2.0, 8.0
TRUNCATION, ALPHA, ETA = 0.04, 0.1, 0.5


def _case(kind, rig, views, width, height, pitch, perturb, fmt, labels=0, iterations=0, name=None):
    case = dict(kind=kind, rig=rig, views=views, width=width, height=height, pitch=pitch, perturb=perturb, fmt=fmt,
                labels=labels, iterations=iterations)
    return case if name is None else dict(name=name, **case)


def listed():
    return [
        # a cold frame of a small stereo-like line rig: the smallest frame, where launches and latency count
        _case("frame", "line", 3, 320, 240, 16, False, "rgba8", 64, 4, "frame_3x320x240_rgba8"),
        # a cold frame of an 8-camera arc at Middlebury-like size (converging cameras, irregular superpixels)
        _case("frame", "arc", 8, 1024, 768, 14, True, "rgba8", 256, 6, "frame_8x1024x768_rgba8"),
        # a cold frame of a 4x4 full-HD array with half-float views: the largest frame
        _case("frame", "grid", 16, 1920, 1080, 16, False, "f16", 256, 8, "frame_16x1920x1080_f16"),
        # a frame whose images, label maps and results live in pinned host memory (copies included)
        _case("host", "line", 4, 640, 480, 12, True, "rgba8", 128, 5, "host_4x640x480_rgba8"),
        # the server's steady state: the queued frames of two rigs (an arc, and a grid of 1280x720 views) in one
        # warm-started call of three iterations
        _case("warm", "arc", 8, 1024, 768, 14, True, "rgba8", 256, 3, "warm_two_rigs_rgba8"),
        # many light fields of uneven shapes in one cold batched call
        _case("batch", "mix", 4, 640, 480, 0, True, "rgba8", 192, 6, "batch_cold_mixed_rgba8"),
        # the plane sweep alone with every label's cost (inspection, training targets), float views, odd sizes
        _case("sweep", "arc", 5, 801, 603, 11, True, "f32", 97, 0, "sweep_costs_5x801x603_f32"),
        # one refinement iteration alone with choices and energies, bfloat16 views
        _case("iterate", "grid", 9, 1280, 720, 16, False, "bf16", 256, 2, "iterate_9x1280x720_bf16"),
        # dense depth maps from planes, full HD
        _case("rasterize", "grid", 16, 1920, 1080, 16, False, "f16", 64, 0, "rasterize_16x1920x1080"),
        # stability-based fusion of the depth maps of a 3x3 array
        _case("fuse", "grid", 9, 1280, 720, 16, False, "rgba8", 64, 0, "fuse_9x1280x720"),
        # SLIC segmentation of a frame's views (the step before every frame that brings no label maps)
        _case("slic", "arc", 8, 1024, 768, 14, False, "rgba8", 0, 10, "slic_8x1024x768_rgba8"),
        # superpixel statistics of one view without allocation (fixed-memory programs, capture)
        _case("stats", "line", 2, 1280, 720, 16, True, "f16", 0, 0, "stats_1280x720_f16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "host", "warm", "batch", "sweep", "iterate", "rasterize", "fuse", "slic",
                       "stats"])
    width = _log_int(rng, 200, 1920)
    height = max(120, min(1080, int(width * rng.uniform(0.5, 0.8))))
    views = rng.randint(2, 12)
    rig = rng.choice(["line", "arc", "grid"])
    fmt = rng.choice(["rgba8", "rgba8", "f16", "bf16", "f32"])
    pitch = rng.randint(8, 32)
    labels = _log_int(rng, 30, 256)
    iterations = rng.randint(2, 8)
    perturb = rng.random() < 0.5
    if kind in ("warm", "batch"):
        width, height, views, fmt = min(width, 1024), min(height, 768), min(views, 8), "rgba8"
        iterations = 3 if kind == "warm" else iterations
    if kind == "batch":
        rig, pitch, views, width, height = "mix", 0, rng.randint(2, 5), 4 * rng.randint(40, 160), 480
    if kind == "iterate":
        width, height, views, iterations = min(width, 960), min(height, 640), min(views, 9), rng.randint(1, 6)
    if kind == "sweep":
        width, height, views = min(width, 901), min(height, 603), min(views, 5)
    if kind == "slic":
        iterations = rng.randint(1, 12)
    return _case(kind, rig, views, width, height, pitch, perturb, fmt, labels, iterations)


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------

def _rig(kind, views, width, height):
    f = 300.0 * width / 320.0
    if kind == "arc":
        return synth.arc_rig(views, 30.0 if views > 2 else 6.0, 5.0, f, width, height)
    if kind == "line":
        return synth.line_rig(views, 0.1, f, width, height)
    rows = max(1, int(math.floor(math.sqrt(views))))
    g = synth.grid_rig(rows, -(-views // rows), 0.08, f, width, height)
    return synth.Rig(g.K[:views].copy(), g.R[:views].copy(), g.t[:views].copy(), width, height)


def _as_format(rgb, fmt):
    return synth.quantize_rgba8(rgb) if fmt == "rgba8" else synth.to_rgba_float(rgb, DTYPES[fmt])


def _light_field(rig, pitch, perturb, fmt, labels, iterations, seed, lf_index=0):
    """One light field as a program holds it: views and label maps on the device, cameras, parameters.  The scene
    has textured and untextured planes, spheres and a textured background, as the workload configurations have."""
    rng = np.random.default_rng([seed, lf_index, 11])
    scene = synth._random_scene(rng, 5, 2, 1, float(rig.K[0, 0, 0]), D_MIN, D_MAX, 1.8)
    rgb, depth, _ = synth.render(rig, scene, "cuda")
    maps, gw, gh = [], 0, 0
    for v in range(rig.V):
        m, gw, gh = synth.grid_labels_fast(rig.W, rig.H, pitch, perturb, seed=seed % 100003 + 17 * v + lf_index,
                                           device="cuda")
        maps.append(m)
    params = dict(d_min=D_MIN, d_max=D_MAX, num_labels=max(1, labels), iterations=iterations, T=TRUNCATION, sigma=0.0,
                  alpha=ALPHA, eta=ETA, kernel_size_init=0, kernel_step_sp=5.0, max_neighbor_views=8, depth_domain=0,
                  jitter=1, term_mask=7, sweep_frame=0, seed=seed, lf_index=lf_index, xy_eps=0.0, warm_iter_offset=0)
    item = dict(views=_as_format(rgb, fmt), labels=torch.stack(maps).contiguous(), K=rig.K, R=rig.R, t=rig.t, GW=gw,
                GH=gh, params=params)
    return item, depth.to(torch.float32)


def _args(item):
    return [item[k] for k in ("views", "labels", "K", "R", "t", "GW", "GH", "params")]


def _superpixels(item):
    return len(item["K"]) * item["GW"] * item["GH"]


def _outputs(items):
    """Plane and depth buffers that a program allocates once and passes to every frame."""
    planes = torch.zeros((sum(_superpixels(i) for i in items), 4), dtype=torch.float32, device="cuda")
    depths = [torch.zeros(i["views"].shape[:3], dtype=torch.float32, device="cuda") for i in items]
    return planes, depths


def _next_frame(views, seed):
    """The next video frame of a static scene: the same picture under fresh sensor noise."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    noise = torch.randint(-2, 3, views.shape, generator=g, dtype=torch.int16, device="cuda")
    return (views.to(torch.int16) + noise).clamp(0, 255).to(torch.uint8)


def _mix_items(case, seed):
    """`views` light fields of uneven camera counts, sizes, superpixel pitches and label counts."""
    rng = np.random.default_rng([case["views"], case["width"], case["labels"]])     # shapes: the case's alone
    items = []
    for l in range(case["views"]):
        n = int(rng.integers(4, 9))
        scale = (1.0, 1.25, 0.75, 1.5)[l % 4]
        w, h = int(case["width"] * scale), int(case["height"] * scale)
        rig = _rig("arc" if l % 2 == 0 else "grid", n, w, h)
        labels = max(16, int(case["labels"] * (0.66 + 0.33 * (l % 3) / 2)))
        items.append(_light_field(rig, 8 + int(rng.integers(0, 25)), True, case["fmt"], labels, case["iterations"],
                                  seed, l)[0])
    return items


def _slic_grid(case):
    return max(1, round(case["width"] / case["pitch"])), max(1, round(case["height"] / case["pitch"]))


def _noisy_depth(depth, seed):
    """Estimated depth maps: the true ones with 0.4 % noise, 4 % outliers and 2 % holes."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = torch.rand(depth.shape, generator=g, device="cuda")
    e = torch.randn(depth.shape, generator=g, device="cuda")
    d = depth * (1.0 + 0.004 * e)
    d = torch.where(r < 0.04, depth * (0.6 + 0.8 * torch.rand(depth.shape, generator=g, device="cuda")), d)
    return torch.where(r > 0.98, torch.zeros_like(d), d).contiguous()


def _noisy_planes(item, depth, seed):
    """Planes near the surface: the depth at each superpixel's median pixel, normals towards the camera."""
    g = torch.Generator(device="cuda").manual_seed(seed + 1)
    n = item["GW"] * item["GH"]
    out = []
    for v in range(depth.shape[0]):
        lab = item["labels"][v].reshape(-1).long()
        cnt = torch.bincount(lab, minlength=n).clamp(min=1)
        mean = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, lab, depth[v].reshape(-1).double()) / cnt
        nrm = torch.randn((n, 3), generator=g, dtype=torch.float64, device="cuda") * 0.2
        nrm[:, 2] -= 1.0
        out.append(torch.cat([mean[:, None], nrm / nrm.norm(dim=1, keepdim=True)], dim=1))
    return torch.cat(out).to(torch.float32).contiguous()


def _inputs(case, seed):
    """The case's light field and ground-truth depth (rendered), shared by prepare and exact."""
    rig = _rig(case["rig"], case["views"], case["width"], case["height"])
    return _light_field(rig, case["pitch"], case["perturb"], case["fmt"], case["labels"], case["iterations"], seed)


def _bound(ctx, item):
    ctx.set_input(*_args(item))


def prepare(case, seed):
    kind = case["kind"]
    state = dict(kind=kind, case=case, ctx=lfd.Context(torch.cuda.current_device()))
    ctx = state["ctx"]
    if kind == "batch":
        state["items"] = _mix_items(case, seed)
        state["out"] = _outputs(state["items"])
        return state
    item, depth = _inputs(case, seed)
    state["item"] = item
    if kind == "frame":
        state["out"] = _outputs([item])
    elif kind == "host":
        state["host"] = [item["views"].cpu().pin_memory(), item["labels"].cpu().pin_memory()]
        state["planes"] = torch.zeros((_superpixels(item), 4), dtype=torch.float32).pin_memory()
        state["depth"] = torch.zeros(tuple(item["views"].shape[:3]), dtype=torch.float32).pin_memory()
    elif kind == "warm":
        second = _light_field(_rig("grid", 9, case["width"] * 5 // 4, case["height"] * 15 // 16), 16, False,
                              case["fmt"], case["labels"], case["iterations"], seed, 1)[0]
        items = [item, second]
        cold = [dict(i, params=dict(i["params"], iterations=6)) for i in items]
        planes, _ = ctx.estimate_batch(cold, want_depth=False)
        ctx.synchronize()
        ns = _superpixels(item)
        state["warm"] = [planes[:ns].clone(), planes[ns:].clone()]
        for k, i in enumerate(items):
            i["views"] = _next_frame(i["views"], seed + k)
            i["params"] = dict(i["params"], warm_iter_offset=3)
        state["items"] = items
        state["out"] = _outputs(items)
    elif kind == "sweep":
        _bound(ctx, item)
    elif kind == "iterate":
        _bound(ctx, item)
        state["planes"] = _noisy_planes(item, depth, seed)
    elif kind == "rasterize":
        _bound(ctx, item)
        state["planes"] = _noisy_planes(item, depth, seed)
    elif kind == "fuse":
        _bound(ctx, item)
        state["depth"] = _noisy_depth(depth, seed)
    elif kind == "stats":
        n = item["GW"] * item["GH"]
        state["stats"] = torch.zeros((n, 8), dtype=torch.float32, device="cuda")
    return state


def run(state):
    kind, ctx, case = state["kind"], state["ctx"], state["case"]
    if kind == "frame":
        planes, depths = state["out"]
        return list(ctx.estimate(*_args(state["item"]), out_planes=planes, out_depth=depths[0]))
    if kind == "host":
        views, labels = state["host"]
        ctx.estimate_host(views, labels, *_args(state["item"])[2:], state["planes"], state["depth"])
        return [state["planes"], state["depth"]]
    if kind == "batch":
        return list(ctx.estimate_batch(state["items"], out=state["out"]))
    if kind == "warm":
        return list(ctx.estimate_batch(state["items"], out=state["out"], warm=state["warm"]))
    if kind == "sweep":
        return list(ctx.plane_sweep(want_labels=True, want_costs=True))
    if kind == "iterate":
        return list(ctx.iterate(case["iterations"], state["planes"], want_choice=True))
    if kind == "rasterize":
        return [ctx.rasterize(state["planes"])]
    if kind == "fuse":
        return [ctx.fuse(state["depth"])]
    if kind == "slic":
        gw, gh = _slic_grid(case)
        return list(ctx.slic(state["item"]["views"], gw, gh, iterations=case["iterations"], want_centres=True))
    item = state["item"]
    lfd.superpixel_stats_noalloc(item["labels"][0], item["views"][0], item["GW"], item["GH"], ALPHA, state["stats"])
    return [state["stats"]]


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def _grid(case):
    return max(1, int(case["width"] / case["pitch"] + 0.5)), max(1, int(case["height"] / case["pitch"] + 0.5))


def _candidates(case, iteration):
    """Candidate planes of one refinement iteration: the kernel's cells and the eight triangle normals."""
    gw, gh = _grid(case)
    cells = min(case["width"], case["height"]) / math.sqrt(case["width"] * case["height"] / (gw * gh))
    return 9 + 8 * max(1, int(cells / 5 / iteration)) + 8


def _frame_flops(case, iterations, offset=0):
    """40 operations for a bilinear truncated-SSD sample of every label, 17 for an energy sample of every candidate
    (the sums of the method's definition)."""
    samples = case["views"] * case["width"] * case["height"] * min(8, case["views"] - 1)
    cands = sum(_candidates(case, i + offset) for i in range(1, iterations + 1))
    return samples * ((40 * case["labels"] if offset == 0 else 0) + 17 * cands)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        c = dict(case, views=6, pitch=20, width=int(case["width"] * 1.1), height=int(case["height"] * 1.1))
        one = work(dict(c, kind="frame"))
        return {k: case["views"] * v for k, v in one.items()}
    px = case["views"] * case["width"] * case["height"]
    gw, gh = _grid(case)
    sp = case["views"] * gw * gh
    tb = TEXEL_BYTES[case["fmt"]]
    nnb = min(8, case["views"] - 1)
    frame_bytes = px * (tb + 4 + 4) + 16 * sp
    if kind in ("frame", "host"):
        return {"bytes": frame_bytes, "flops": _frame_flops(case, case["iterations"])}
    if kind == "warm":
        second = dict(case, views=9, width=case["width"] * 5 // 4, height=case["height"] * 15 // 16, pitch=16)
        return {"bytes": 2.4 * frame_bytes,
                "flops": _frame_flops(case, 3, 3) + _frame_flops(second, 3, 3)}
    if kind == "sweep":
        return {"bytes": px * (tb + 4) + sp * (20 + 4 * case["labels"]), "flops": 40 * px * nnb * case["labels"]}
    if kind == "iterate":
        return {"bytes": px * 4 + sp * (32 + 16), "flops": 17 * px * nnb * _candidates(case, case["iterations"])}
    if kind == "rasterize":        # pixel lists read, the visibility map of the next iteration and the depth written
        return {"bytes": px * (4 + 16 + 4) + 16 * sp, "flops": 6 * px}
    if kind == "fuse":             # every map read, every map written; each pixel projected into every other view
        return {"bytes": px * 8, "flops": 20 * px * (case["views"] - 1)}
    if kind == "slic":
        return {"bytes": px * (tb + 4), "flops": px * (60 + (case["iterations"] + 1) * 9 * 11)}
    one = case["width"] * case["height"]
    return {"bytes": one * (tb + 4) + 32 * gw * gh, "flops": 5 * one}


# --------------------------------------------------------------------------
# the same outputs in 64 bits, in plain torch
# --------------------------------------------------------------------------

def _colours(views):
    c = views[..., :3].double()
    return c / 255.0 if views.dtype == torch.uint8 else c


def _neighbours(R, t, k):
    C = -np.einsum("vji,vj->vi", R, t)
    out = []
    for v in range(len(C)):
        d = np.linalg.norm(C - C[v], axis=1)
        left, pick = [i for i in range(len(C)) if i != v], []
        for _ in range(min(k, len(left))):
            best = left[0]
            for i in left:
                if d[i] < d[best] * (1.0 - 1e-9):
                    best = i
            left.remove(best)
            pick.append(best)
        out.append(pick)
    return out


def _pair(K, R, t, v, i):
    """P, q of the plane-induced homography P + q g^T from view v to view i."""
    rel = R[i] @ R[v].T
    return K[i] @ rel @ np.linalg.inv(K[v]), K[i] @ (t[i] - rel @ t[v])


def _uniform(seed, lf, v, n_sp, n_lab):
    """SplitMix64 draws in [0, 1) for every (superpixel, label) of a view."""
    with np.errstate(over="ignore"):
        key = np.uint64(((lf << 12) + v) << 20) + np.arange(n_sp, dtype=np.uint64)[:, None]
        x = np.uint64(seed) ^ ((key << np.uint64(12)) + np.arange(n_lab, dtype=np.uint64)[None, :])
        z = x + np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return torch.from_numpy((z >> np.uint64(11)).astype(np.float64) / 9007199254740992.0).cuda()


def _pixels(width, height):
    y, x = torch.meshgrid(torch.arange(height, dtype=torch.float64, device="cuda"),
                          torch.arange(width, dtype=torch.float64, device="cuda"), indexing="ij")
    return x.reshape(-1), y.reshape(-1)


def _sum_by(lab, n, values):
    return torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, lab, values)


def _bilinear(img, x, y):
    h, w, _ = img.shape
    x, y = x.clamp(0, w - 1), y.clamp(0, h - 1)
    x0, y0 = x.floor(), y.floor()
    fx, fy = (x - x0)[:, None], (y - y0)[:, None]
    x0, y0 = x0.long(), y0.long()
    x1, y1 = (x0 + 1).clamp(max=w - 1), (y0 + 1).clamp(max=h - 1)
    flat = img.reshape(-1, 3)
    top = flat[y0 * w + x0] * (1 - fx) + flat[y0 * w + x1] * fx
    bot = flat[y1 * w + x0] * (1 - fx) + flat[y1 * w + x1] * fx
    return top * (1 - fy) + bot * fy


def _exact_sweep(item):
    K, R, t, p = item["K"], item["R"], item["t"], item["params"]
    col = _colours(item["views"])
    V, H, W, _ = col.shape
    S, L = item["GW"] * item["GH"], p["num_labels"]
    x, y = _pixels(W, H)
    nbs = _neighbours(R, t, 8)
    lo, delta = 1 / D_MAX, (1 / D_MIN - 1 / D_MAX) / L
    planes, costs = [], []
    for v in range(V):
        lab = item["labels"][v].reshape(-1).long()
        z = lo + (torch.arange(L, dtype=torch.float64, device="cuda") + _uniform(p["seed"], p["lf_index"], v, S, L)) * delta
        own = col[v].reshape(-1, 3)
        cost = torch.zeros((S, L), dtype=torch.float64, device="cuda")
        for i in nbs[v]:
            P, q = _pair(K, R, t, v, i)
            h = [P[r, 0] * x + P[r, 1] * y + P[r, 2] for r in range(3)]
            for k in range(L):
                zk = z[lab, k]
                X, Y, Z = (h[r] + q[r] * zk for r in range(3))
                u, w = X / Z, Y / Z
                ok = (Z > 0) & (u >= -0.5) & (u < W - 0.5) & (w >= -0.5) & (w < H - 0.5)
                s = _bilinear(col[i], torch.where(ok, u, 0 * u), torch.where(ok, w, 0 * w))
                ssd = ((own - s) ** 2).sum(1).clamp(max=TRUNCATION)
                cost[:, k] += _sum_by(lab, S, torch.where(ok, ssd, torch.full_like(ssd, TRUNCATION)))
        some = torch.bincount(lab, minlength=S) > 0
        d = 1 / z.gather(1, cost.argmin(1, keepdim=True))
        plane = torch.cat([d, torch.zeros((S, 2), device="cuda", dtype=torch.float64), -torch.ones_like(d)], dim=1)
        planes.append(torch.where(some[:, None], plane, torch.zeros_like(plane)))
        costs.append(torch.where(some[:, None], cost, torch.zeros_like(cost)))
    return [torch.cat(planes), None, torch.cat(costs)]


def _geometry(item):
    """Per view: labels, counts, centroids, rays K^-1 (c, 1) and mean colours of the superpixels."""
    col = _colours(item["views"])
    V, H, W, _ = col.shape
    S = item["GW"] * item["GH"]
    x, y = _pixels(W, H)
    out = []
    for v in range(V):
        lab = item["labels"][v].reshape(-1).long()
        cnt = _sum_by(lab, S, torch.ones_like(x))
        n = cnt.clamp(min=1)
        c = torch.stack([_sum_by(lab, S, x) / n, _sum_by(lab, S, y) / n, torch.ones_like(n)], dim=1)
        rgb = torch.stack([_sum_by(lab, S, col[v, ..., k].reshape(-1)) / n for k in range(3)], dim=1)
        Ki = torch.from_numpy(np.linalg.inv(item["K"][v])).cuda()
        out.append(dict(lab=lab, cnt=cnt, cen=c * (cnt > 0)[:, None], rgb=rgb, Ki=Ki, ray=c @ Ki.T))
    return out, x, y


def _to_g(planes, geo):
    """Inverse-depth vectors g (1 / depth(p) = g . (p, 1)) of planes {d, n} anchored at the centroids."""
    rho = planes[:, 0] * (planes[:, 1:] * geo["ray"]).sum(1)
    ok = (planes[:, 0] > 0) & (rho != 0) & (geo["cnt"] > 0)
    g = (planes[:, 1:] @ geo["Ki"]) / torch.where(ok, rho, torch.ones_like(rho))[:, None]
    return g * ok[:, None], ok


RING = ((1, 0), (1, -1), (0, -1), (-1, -1), (-1, 0), (-1, 1), (0, 1), (1, 1))


def _offsets(item, iteration):
    gw, gh = item["GW"], item["GH"]
    V, H, W = item["views"].shape[:3]
    size = int(min(W, H) / math.sqrt(W * H / (gw * gh)))
    steps = max(1, int(math.floor(size / 5.0 + 0.5)) // iteration)
    cells, last = [(0, 0)] + list(RING), 1
    for k in range(1, steps + 1):
        r = max(1, int(math.floor(k * (size / iteration) / steps + 0.5)))
        if r > last:
            cells += [(dx * r, dy * r) for dx, dy in RING]
            last = r
    return cells


def _shifted(item, dx, dy):
    """For each superpixel, the one dx, dy cells away (0 where there is none) and whether it exists."""
    gw, gh = item["GW"], item["GH"]
    s = torch.arange(gw * gh, device="cuda")
    gx, gy = s % gw + dx, s // gw + dy
    ok = (gx >= 0) & (gy >= 0) & (gx < gw) & (gy < gh)
    return torch.where(ok, gy * gw + gx, torch.zeros_like(s)), ok


def _energy(item, geo, maps, nbs, v, g, valid, x, y, sigma2):
    """E of one candidate plane g per superpixel of view v (-inf where it is not valid)."""
    me = geo[v]
    S, lab = g.shape[0], me["lab"]
    H, W = item["views"].shape[1:3]
    # smoothness over the present 8-neighbours
    w, e, has = [], [], []
    for dx, dy in RING:
        j, ok = _shifted(item, dx, dy)
        ok = ok & (me["cnt"][j] > 0) & (me["d"][j] > 0)
        a = ((me["rgb"][j] - me["rgb"]) ** 2).sum(1) / (2 * ALPHA ** 2)
        diff = 1 / torch.where(ok, me["d"][j], torch.ones_like(a)) - (g * me["cen"][j]).sum(1)
        w.append(torch.where(ok, a, torch.full_like(a, float("inf"))))
        e.append(torch.exp(-diff ** 2 / (2 * sigma2)))
        has.append(ok)
    a = torch.stack(w)
    any_nb = torch.stack(has).any(0)
    wt = torch.exp(-(a - torch.where(any_nb, a.min(0).values, torch.zeros_like(a[0]))))
    wt = torch.where(torch.stack(has), wt, torch.zeros_like(wt))
    Es = torch.where(any_nb, (wt * torch.stack(e)).sum(0) / wt.sum(0).clamp(min=1e-300), torch.ones_like(g[:, 0]))
    gp = g[lab, 0] * x + g[lab, 1] * y + g[lab, 2]
    Ec = torch.zeros(S, dtype=torch.float64, device="cuda")
    for i in nbs[v]:
        P, q = _pair(item["K"], item["R"], item["t"], v, i)
        X, Y, Z = (P[r, 0] * x + P[r, 1] * y + P[r, 2] + q[r] * gp for r in range(3))
        u, w_ = (X / Z + 0.5).floor(), (Y / Z + 0.5).floor()
        ok = (gp > 0) & (Z > 0) & (u >= 0) & (u < W) & (w_ >= 0) & (w_ < H)
        idx = torch.where(ok, w_ * W + u, torch.zeros_like(u)).long()
        rgb, inv = maps[i]
        om = torch.exp(-((rgb[idx] - me["rgb"][lab]) ** 2).sum(1) / (2 * ALPHA ** 2))
        D = inv[idx]
        zeta = gp / torch.where(ok, Z, torch.ones_like(Z))
        seen = ok & (D > 0)
        inX = seen & (zeta >= D)
        G = torch.exp(-(zeta - D) ** 2 / (2 * sigma2))
        cnt, nx = _sum_by(lab, S, ok.double()), _sum_by(lab, S, inX.double())
        ny = _sum_by(lab, S, (seen & ~inX).double())
        Si = _sum_by(lab, S, om * ok) / cnt.clamp(min=1)
        Vi = Si * _sum_by(lab, S, G * inX) / nx.clamp(min=1)
        Ec += Vi + torch.where(ny > 0, ETA * (1 - me["minw"]), torch.zeros_like(Vi))
    E = Es * Ec / len(nbs[v])
    return torch.where(valid, E, torch.full_like(E, -float("inf")))


def _exact_iterate(item, planes_in, iteration):
    p = item["params"]
    geo, x, y = _geometry(item)
    S = item["GW"] * item["GH"]
    V = len(geo)
    sigma2 = (2 * (1 / D_MIN - 1 / D_MAX) / p["num_labels"]) ** 2
    nbs = _neighbours(item["R"], item["t"], 8)
    maps = []
    for v in range(V):
        m = geo[v]
        pl = planes_in[v * S:(v + 1) * S].double()
        m["n"], m["d"] = pl[:, 1:], pl[:, 0]
        m["g"], m["ok"] = _to_g(pl, m)
        inv = m["g"][m["lab"], 0] * x + m["g"][m["lab"], 1] * y + m["g"][m["lab"], 2]
        maps.append((m["rgb"][m["lab"]], inv.clamp(min=0)))
        sim = []
        for dx, dy in RING:
            j, ok = _shifted(item, dx, dy)
            a = torch.exp(-((m["rgb"][j] - m["rgb"]) ** 2).sum(1) / (2 * ALPHA ** 2))
            sim.append(torch.where(ok & (m["cnt"][j] > 0), a, torch.ones_like(a)))
        m["minw"] = torch.stack(sim).min(0).values
    energies = []
    for v in range(V):
        m = geo[v]
        rn = m["ray"].norm(dim=1)
        best = torch.full((S,), -float("inf"), dtype=torch.float64, device="cuda")
        dep = m["d"].clone()
        for k, (dx, dy) in enumerate(_offsets(item, iteration)):
            j, ok = _shifted(item, dx, dy)
            g = m["g"][j]
            ok = ok & m["ok"][j] & (m["cnt"] > 0)
            ig = (g * m["cen"]).sum(1)
            if k > 0:
                ok = ok & (ig >= 1 / D_MAX) & (ig <= 1 / D_MIN) & ((m["n"][j] * m["ray"]).sum(1).abs() >= 0.1 * rn)
            E = _energy(item, geo, maps, nbs, v, g, ok, x, y, sigma2)
            better = E > best
            best = torch.where(better, E, best)
            if k > 0:
                dep = torch.where(better, 1 / ig, dep)
        prop = best.clone()
        for k in range(8):
            a, oka = _shifted(item, *RING[k])
            b, okb = _shifted(item, *RING[(k + 1) % 8])
            p0 = dep[:, None] * m["ray"]
            n = torch.linalg.cross(m["d"][a][:, None] * m["ray"][a] - p0, m["d"][b][:, None] * m["ray"][b] - p0, dim=1)
            nn = n.norm(dim=1)
            n = n / nn.clamp(min=1e-300)[:, None]
            n = torch.where(((n * m["ray"]).sum(1) > 0)[:, None], -n, n)
            ok = oka & okb & (m["cnt"][a] > 0) & (m["cnt"][b] > 0) & (m["d"][a] > 0) & (m["d"][b] > 0) & (nn > 1e-12)
            ok = ok & ((n * m["ray"]).sum(1).abs() >= 0.1 * rn) & (prop > -float("inf")) & (dep > 0)
            g, okg = _to_g(torch.cat([dep[:, None], n], dim=1), m)
            best = torch.maximum(best, _energy(item, geo, maps, nbs, v, g, ok & okg, x, y, sigma2))
        energies.append(torch.stack([prop, best], dim=1))
    return [None, None, torch.cat(energies)]     # near-equal candidates: the choice itself has no 64-bit value


def _exact_rasterize(item, planes):
    geo, x, y = _geometry(item)
    S = item["GW"] * item["GH"]
    H, W = item["views"].shape[1:3]
    out = []
    for v, m in enumerate(geo):
        g, ok = _to_g(planes[v * S:(v + 1) * S].double(), m)
        inv = g[m["lab"], 0] * x + g[m["lab"], 1] * y + g[m["lab"], 2]
        ok = ok[m["lab"]] & (inv > 0)
        out.append(torch.where(ok, 1 / torch.where(ok, inv, torch.ones_like(inv)), torch.zeros_like(inv)).reshape(H, W))
    return [torch.stack(out)]


def _exact_fuse(item, depth, tau=0.01):
    K, R, t = item["K"], item["R"], item["t"]
    V, H, W = depth.shape
    x, y = _pixels(W, H)
    d = depth.double().reshape(V, -1)
    inf = float("inf")
    out = []
    for r in range(V):
        cand = [torch.where(d[r] > 0, d[r], torch.full_like(d[r], inf))]
        for i in range(V):
            if i == r:
                continue
            A = R[r] @ R[i].T
            M, e = K[r] @ A @ np.linalg.inv(K[i]), K[r] @ (t[r] - A @ t[i])
            X, Y, Z = (d[i] * (M[k, 0] * x + M[k, 1] * y + M[k, 2]) + e[k] for k in range(3))
            u, v = X / Z, Y / Z
            ok = (d[i] > 0) & (Z > 0) & (u >= 0) & (u <= W - 1) & (v >= 0) & (v <= H - 1)
            idx = ((v[ok] + 0.5).floor() * W + (u[ok] + 0.5).floor()).long()
            z = torch.full_like(d[r], inf).scatter_reduce_(0, idx, Z[ok], "amin")
            cand.append(z)
        c = torch.stack(cand)
        real = torch.isfinite(c)
        best = torch.full_like(d[r], inf)
        for s in range(V):
            agree = (c - c[s]).abs() <= tau * c[s]
            stab = (real * torch.where(agree, 1, -1)).sum(0) - 1
            best = torch.where(real[s] & (stab >= 0), torch.minimum(best, c[s]), best)
        out.append(torch.where(torch.isfinite(best), best, torch.zeros_like(best)).reshape(H, W))
    return [torch.stack(out)]


def _lab_colour(rgb):
    lin = torch.where(rgb <= 0.04045, rgb / 12.92, ((rgb.clamp(min=0) + 0.055) / 1.055) ** 2.4)
    m = torch.tensor([[0.4124564, 0.3575761, 0.1804375], [0.2126729, 0.7151522, 0.0721750],
                      [0.0193339, 0.1191920, 0.9503041]], dtype=torch.float64, device="cuda")
    white = torch.tensor([0.95047, 1.0, 1.08883], dtype=torch.float64, device="cuda")
    q = (lin @ m.T) / white
    f = torch.where(q > 216 / 24389, q.clamp(min=0) ** (1 / 3), (24389 / 27 * q + 16) / 116)
    return torch.stack([116 * f[:, 1] - 16, 500 * (f[:, 0] - f[:, 1]), 200 * (f[:, 1] - f[:, 2])], dim=1)


def _exact_slic(views, gw, gh, iterations, compactness=10.0):
    col = _colours(views)
    V, H, W, _ = col.shape
    x, y = _pixels(W, H)
    ex = torch.tensor([(2 * k * W + gw) // (2 * gw) for k in range(gw + 1)], device="cuda")
    ey = torch.tensor([(2 * k * H + gh) // (2 * gh) for k in range(gh + 1)], device="cuda")
    cx = torch.searchsorted(ex, x.long(), right=True) - 1
    cy = torch.searchsorted(ey, y.long(), right=True) - 1
    weight = compactness ** 2 * gw * gh / (W * H)
    n = gw * gh
    out = []
    for v in range(V):
        lab = _lab_colour(col[v].reshape(-1, 3))
        feat = torch.cat([lab, x[:, None], y[:, None]], dim=1)
        sx = 0.5 * (ex[:-1] + ex[1:] - 1).double().repeat(gh)
        sy = 0.5 * (ey[:-1] + ey[1:] - 1).double().repeat_interleave(gw)
        at = ((sy + 0.5).floor().clamp(max=H - 1) * W + (sx + 0.5).floor().clamp(max=W - 1)).long()
        cen = torch.cat([lab[at], sx[:, None], sy[:, None]], dim=1)
        for _ in range(iterations):
            best = torch.full_like(x, float("inf"))
            pick = cy * gw + cx
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    ok = (cx + dx >= 0) & (cx + dx < gw) & (cy + dy >= 0) & (cy + dy < gh)
                    c = torch.where(ok, (cy + dy) * gw + cx + dx, torch.zeros_like(cx))
                    f = (feat - cen[c]) ** 2
                    D = torch.where(ok, f[:, :3].sum(1) + weight * f[:, 3:].sum(1), torch.full_like(x, float("inf")))
                    pick = torch.where(D < best, c, pick)
                    best = torch.minimum(D, best)
            cnt = _sum_by(pick, n, torch.ones_like(x))
            mean = torch.stack([_sum_by(pick, n, feat[:, k]) for k in range(5)], dim=1) / cnt.clamp(min=1)[:, None]
            cen = torch.where((cnt > 0)[:, None], mean, cen)
        out.append(cen)
    return [None, torch.stack(out)]


def _exact_stats(item):
    one = dict(item, views=item["views"][:1], labels=item["labels"][:1])
    m = _geometry(one)[0][0]
    sim = []
    for dx, dy in RING:
        j, ok = _shifted(item, dx, dy)
        a = torch.exp(-((m["rgb"][j] - m["rgb"]) ** 2).sum(1) / (2 * ALPHA ** 2))
        sim.append(torch.where(ok & (m["cnt"][j] > 0), a, torch.ones_like(a)))
    minw = torch.stack(sim).min(0).values
    return [torch.cat([m["cen"][:, :2], m["rgb"], minw[:, None], m["cnt"][:, None], torch.zeros_like(minw)[:, None]], 1)]


def exact(case, seed):
    """Outputs of `run` in 64 bits.  Whole frames have none: they chain decisions over near-equal candidates, so that
    two evaluations differ in which of two equally good planes a superpixel keeps."""
    kind = case["kind"]
    if kind in ("frame", "host", "batch", "warm"):
        return None
    item, depth = _inputs(case, seed)
    if kind == "sweep":
        return _exact_sweep(item)
    if kind == "iterate":
        return _exact_iterate(item, _noisy_planes(item, depth, seed), case["iterations"])
    if kind == "rasterize":
        return _exact_rasterize(item, _noisy_planes(item, depth, seed))
    if kind == "fuse":
        return _exact_fuse(item, _noisy_depth(depth, seed))
    if kind == "slic":
        gw, gh = _slic_grid(case)
        return _exact_slic(item["views"], gw, gh, case["iterations"])
    return _exact_stats(item)
