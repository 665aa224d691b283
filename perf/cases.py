"""The work a user of this framework has it do, as cases that can be timed.

Each case is one call chain through the public entry points of
paper_1903_07149_gb300.scalp: a whole decomposition (new inputs, ten iterations
of Algorithm 1, connectivity, labels), a batch of them, a served request mix,
the multi-scale boundary map, a video volume, and the three per-image tools
(the contour prior, the quality metrics, the label means).

Inputs are made on the GPU from the seed alone, built like synth.py's images:
Voronoi cells with a colour ramp per cell and Gaussian noise, and their blurred
boundaries as the contour prior.
"""
import math

import torch

from paper_1903_07149_gb300 import scalp, synth

ITERS = 10


def listed():
    return [
        # the smallest decomposition: a thumbnail or a crop, where launches and
        # host latency count (the size of the smoke run)
        {"name": "thumb_96x160", "kind": "solve", "H": 96, "W": 160, "K": 60, "storage": "f32", "prior": "input"},
        # the image size of the paper's data set, with the cluster descriptors
        # read back as a program that builds features on them does
        {"name": "bsd_321x481", "kind": "solve", "H": 321, "W": 481, "K": 400, "storage": "f32", "prior": "input",
         "clusters": True},
        # the headline workload: one HD frame
        {"name": "hd_1080x1920", "kind": "solve", "H": 1080, "W": 1920, "K": 2000, "storage": "f32", "prior": "input"},
        # an odd-sized photograph with no contour map at hand: FP16 planes, the
        # prior computed from the image, fine superpixels (step 15)
        {"name": "photo_1361x2047_f16", "kind": "solve", "H": 1361, "W": 2047, "K": 12000, "storage": "f16",
         "prior": "gradient"},
        # a 4K frame
        {"name": "uhd_2160x3840", "kind": "solve", "H": 2160, "W": 3840, "K": 10000, "storage": "f32",
         "prior": "input"},
        # a data set pass: 64 images of uneven size solved as one batch
        {"name": "batch_64", "kind": "batch", "count": 64, "mix": 3000, "storage": "f32"},
        # a burst of requests served by continuous batching, labels delivered
        # to pinned host memory
        {"name": "serve_12", "kind": "serve", "count": 12, "mix": 3000, "storage": "f16"},
        # the averaged boundary map of one image at 12 scales, 6 to 600 superpixels
        {"name": "multiscale_321x481", "kind": "multiscale", "H": 321, "W": 481, "k_min": 6, "k_max": 600,
         "scales": 12},
        # supervoxels of a short video clip
        {"name": "video_32x240x320", "kind": "video", "T": 32, "H": 240, "W": 320, "K": 2000},
        # the contour prior of one HD frame by itself
        {"name": "prior_1080x1920", "kind": "prior", "H": 1080, "W": 1920},
        # the superpixel metrics of one HD decomposition against its ground truth
        {"name": "quality_1080x1920", "kind": "quality", "H": 1080, "W": 1920, "K": 2000, "segments": 300},
        # mean colour and place of every superpixel of an HD frame
        {"name": "means_1080x1920", "kind": "means", "H": 1080, "W": 1920, "K": 2000},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _image_size(rng, h_max=2160):
    h = int(round(_log_uniform(rng, 64, h_max)))
    w = int(round(h * rng.uniform(0.75, 16 / 9)))
    return h, w


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "batch", "serve", "multiscale", "video", "prior", "quality",
                       "means"])
    if kind == "solve":
        h, w = _image_size(rng)
        step = _log_uniform(rng, 12, 40)
        return {"kind": kind, "H": h, "W": w, "K": max(1, round(h * w / step ** 2)),
                "storage": rng.choice(["f32", "f32", "f16"]), "prior": rng.choice(["input", "input", "gradient"]),
                "clusters": rng.random() < 0.25}
    if kind == "batch":
        return {"kind": kind, "count": int(round(_log_uniform(rng, 3, 48))), "mix": rng.randrange(10000, 100000),
                "storage": rng.choice(["f32", "f16"])}
    if kind == "serve":
        return {"kind": kind, "count": int(round(_log_uniform(rng, 2, 16))), "mix": rng.randrange(10000, 100000),
                "storage": rng.choice(["f32", "f16"])}
    if kind == "multiscale":
        h = rng.randint(120, 360)
        return {"kind": kind, "H": h, "W": int(round(h * rng.uniform(0.7, 1.6))), "k_min": rng.randint(4, 10),
                "k_max": rng.randint(200, 800), "scales": rng.randint(3, 12)}
    if kind == "video":
        t, h = rng.randint(4, 36), rng.randint(64, 240)
        w = int(round(h * rng.uniform(1.0, 16 / 9)))
        step = rng.uniform(7, 13)
        return {"kind": kind, "T": t, "H": h, "W": w, "K": max(1, round(t * h * w / step ** 3))}
    h, w = _image_size(rng)
    if kind == "prior":
        return {"kind": kind, "H": h, "W": w}
    step = _log_uniform(rng, 12, 40)
    k = min(60000, max(4, round(h * w / step ** 2)))
    if kind == "quality":
        return {"kind": kind, "H": h, "W": w, "K": k, "segments": int(round(_log_uniform(rng, 3, 400)))}
    return {"kind": kind, "H": h, "W": w, "K": k}


# --- inputs ------------------------------------------------------------------
def _nearest(sx, sy, H, W):
    """Index of the nearest of the points (sx, sy) for every pixel centre."""
    n = sx.numel()
    dx2 = (torch.arange(W, device="cuda", dtype=torch.float32)[:, None] - sx).square()
    dy2 = (torch.arange(H, device="cuda", dtype=torch.float32)[:, None] - sy).square()
    out = torch.empty((H, W), dtype=torch.int64, device="cuda")
    rows = max(1, (1 << 27) // (W * n))
    for y in range(0, H, rows):
        out[y:y + rows] = (dy2[y:y + rows, None, :] + dx2[None]).argmin(-1)
    return out


def _blur(img):
    """Separable Gaussian, sigma 1, radius 3, the edge sample repeated."""
    taps = [math.exp(-0.5 * t * t) for t in range(-3, 4)]
    for axis in (0, 1):
        n = img.shape[axis]
        at = torch.arange(n, device="cuda")
        img = sum(t / sum(taps) * img.index_select(axis, (at + i - 3).clamp(0, n - 1)) for i, t in enumerate(taps))
    return img


def _colour(cells, dx, dy, n, radius, g):
    base = torch.rand((n, 3), generator=g, device="cuda") * 175.0 + 40.0
    ramp = torch.rand((n, 3, 2), generator=g, device="cuda") * 80.0 - 40.0
    col = base[cells] + ramp[cells, :, 0] * (dx / radius)[..., None] + ramp[cells, :, 1] * (dy / radius)[..., None]
    col += 6.0 * torch.randn(col.shape, generator=g, device="cuda")
    return col.round().clamp(0, 255).to(torch.uint8)


def _contour(cells, g):
    edge = torch.zeros(cells.shape, device="cuda")
    dx, dy = cells[:, 1:] != cells[:, :-1], cells[1:] != cells[:-1]
    edge[:, 1:][dx] = 1.0
    edge[:, :-1][dx] = 1.0
    edge[1:][dy] = 1.0
    edge[:-1][dy] = 1.0
    b = _blur(edge)
    b = b / b.max().clamp(min=1e-6)
    return (b + 0.05 * torch.rand(b.shape, generator=g, device="cuda")).clamp(0, 1)


def _generator(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _grids(H, W):
    return (torch.arange(W, device="cuda", dtype=torch.float32)[None, :],
            torch.arange(H, device="cuda", dtype=torch.float32)[:, None])


def _image(H, W, seed, n=None):
    """(rgb, contour, cells) of one image."""
    g = _generator(seed)
    n = n or max(2, round(300 * H * W / 2_073_600))
    sx, sy = torch.rand(n, generator=g, device="cuda") * W, torch.rand(n, generator=g, device="cuda") * H
    cells = _nearest(sx, sy, H, W)
    xs, ys = _grids(H, W)
    rgb = _colour(cells, xs - sx[cells], ys - sy[cells], n, math.sqrt(H * W / n), g)
    return rgb, _contour(cells, g), cells


def _video(T, H, W, seed):
    """(rgb, contour) of a clip: the cells drift, reflected at the borders."""
    g = _generator(seed)
    n = 40
    size = torch.tensor([W, H], device="cuda", dtype=torch.float32)
    pos = torch.rand((n, 2), generator=g, device="cuda") * size
    vel = torch.rand((n, 2), generator=g, device="cuda") * 3.0 - 1.5
    colours = seed + 1
    xs, ys = _grids(H, W)
    rgb = torch.empty((T, H, W, 3), dtype=torch.uint8, device="cuda")
    con = torch.empty((T, H, W), device="cuda")
    for t in range(T):
        p = torch.remainder(pos + vel * t, 2 * size)
        p = torch.where(p < size, p, 2 * size - p)
        cells = _nearest(p[:, 0], p[:, 1], H, W)
        gt = _generator(colours)  # every frame's cells keep their colours
        rgb[t] = _colour(cells, xs - p[cells, 0], ys - p[cells, 1], n, math.sqrt(H * W / n), gt)
        con[t] = _contour(cells, g)
    return rgb, con


def _superpixels(H, W, K, seed):
    """A label map like a decomposition's: the Voronoi cells of a jittered grid
    of about K points, numbered in raster order of the grid, with ragged
    borders; labels without a pixel are dropped."""
    g = _generator(seed)
    step = math.sqrt(H * W / K)
    nx, ny = max(1, round(W / step)), max(1, round(H / step))
    jx = torch.rand((ny, nx), generator=g, device="cuda") * 0.6 + 0.2
    jy = torch.rand((ny, nx), generator=g, device="cuda") * 0.6 + 0.2
    cx, cy = torch.arange(nx, device="cuda"), torch.arange(ny, device="cuda")
    px, py = (cx[None, :] + jx) * (W / nx), (cy[:, None] + jy) * (H / ny)
    xs, ys = _grids(H, W)
    xs = xs + 1.5 * torch.randn((H, W), generator=g, device="cuda")
    ys = ys + 1.5 * torch.randn((H, W), generator=g, device="cuda")
    gx = (torch.arange(W, device="cuda") * nx // W)[None, :].expand(H, W)
    gy = (torch.arange(H, device="cuda") * ny // H)[:, None].expand(H, W)
    best = torch.full((H, W), math.inf, device="cuda")
    lab = torch.zeros((H, W), dtype=torch.int64, device="cuda")
    for oy in (-1, 0, 1):
        for ox in (-1, 0, 1):
            kx, ky = (gx + ox).clamp(0, nx - 1), (gy + oy).clamp(0, ny - 1)
            d = (xs - px[ky, kx]).square() + (ys - py[ky, kx]).square()
            near = d < best
            best = torch.where(near, d, best)
            lab = torch.where(near, ky * nx + kx, lab)
    return torch.unique(lab, return_inverse=True)[1].to(torch.int32).contiguous()


def _mix(case):
    """(H, W, K) of each image of a batch or a burst of requests."""
    return [(w.H, w.W, w.K) for w in synth.batch_configs(case["count"], seed=case["mix"])]


# --- states, passes -----------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("solve", "batch", "serve"):
        stream = torch.cuda.Stream()
    if kind == "solve":
        rgb, con, _ = _image(case["H"], case["W"], seed)
        if case["prior"] == "gradient":
            con = None
        torch.cuda.synchronize()
        seg = scalp.Segmenter(rgb, con, case["K"], storage=case["storage"], prior=case["prior"], stream=stream)
        out = torch.empty((case["H"], case["W"]), dtype=torch.int32, device="cuda")
        return {"kind": kind, "seg": seg, "rgb": rgb, "con": con, "out": out, "clusters": case.get("clusters", False)}
    if kind in ("batch", "serve"):
        sizes = _mix(case)
        made = [_image(h, w, seed * 1000 + i) for i, (h, w, _) in enumerate(sizes)]
        rgbs, cons = [m[0] for m in made], [m[1] for m in made]
        ks = [k for _, _, k in sizes]
        torch.cuda.synchronize()
        if kind == "batch":
            batch = scalp.Batch(rgbs, cons, ks, storage=case["storage"], stream=stream)
            # the label maps lie one behind the other in one buffer, each on a
            # 256-byte boundary
            at = [0]
            for h, w, _ in sizes:
                at.append(at[-1] + (h * w + 63) // 64 * 64)
            flat = torch.zeros(at[-1], dtype=torch.int32, device="cuda")
            outs = [flat[a:a + h * w].view(h, w) for a, (h, w, _) in zip(at, sizes)]
            torch.cuda.synchronize()
            return {"kind": kind, "batch": batch, "rgbs": rgbs, "cons": cons, "flat": flat, "outs": outs}
        pool = (64 << 20) + sum((h * w + 65536) * 64 for h, w, _ in sizes)
        server = scalp.Server(pool, max_slots=64, storage=case["storage"], iters=ITERS, stream=stream,
                              step_pixels=4_000_000)
        return {"kind": kind, "server": server, "requests": list(zip(rgbs, cons, ks))}
    if kind == "multiscale":
        rgb, con, _ = _image(case["H"], case["W"], seed, n=40)
        return {"kind": kind, "rgb": rgb, "con": con,
                "Ks": scalp.multiscale_K(case["k_min"], case["k_max"], case["scales"])}
    if kind == "video":
        rgb, con = _video(case["T"], case["H"], case["W"], seed)
        out = torch.empty((case["T"], case["H"], case["W"]), dtype=torch.int32, device="cuda")
        return {"kind": kind, "rgb": rgb, "con": con, "K": case["K"], "out": out}
    if kind == "prior":
        return {"kind": kind, "rgb": _image(case["H"], case["W"], seed)[0]}
    if kind == "quality":
        gt = _image(case["H"], case["W"], seed, n=case["segments"])[2].to(torch.int32)
        return {"kind": kind, "labels": _superpixels(case["H"], case["W"], case["K"], seed + 7), "gt": gt}
    rgb = _image(case["H"], case["W"], seed)[0]
    labels = _superpixels(case["H"], case["W"], case["K"], seed + 7)
    n = int(labels.max()) + 1
    return {"kind": kind, "rgb": rgb, "labels": labels, "n": n,
            "out": torch.empty((n, 6), dtype=torch.float64, device="cuda")}


def run(state):
    kind = state["kind"]
    if kind == "solve":
        seg = state["seg"]
        seg.reload(state["rgb"], state["con"])
        seg.iterate(ITERS)
        labels, n = seg.labels(enforce=True, out=state["out"])
        return [labels, n, seg.clusters()] if state["clusters"] else [labels, n]
    if kind == "batch":
        b = state["batch"]
        b.reload(state["rgbs"], state["cons"])
        b.iterate(ITERS)
        _, n = b.labels(enforce=True, outs=state["outs"])
        return [state["flat"], n]
    if kind == "serve":
        srv = state["server"]
        got = [srv.submit(*r) for r in state["requests"]]
        counts, waiting = {}, [rid for rid, _ in got]
        while waiting:
            srv.step()
            left = []
            for rid in waiting:
                done, n = srv.poll(rid)
                if done:
                    counts[rid] = n
                else:
                    left.append(rid)
            waiting = left
        return [[out for _, out in got], [counts[rid] for rid, _ in got]]
    if kind == "multiscale":
        bmap, labels = scalp.multiscale_boundaries(state["rgb"], state["con"], state["Ks"], iters=ITERS)
        return [bmap, labels]
    if kind == "video":
        seg = scalp.VoxelSegmenter(state["rgb"], state["con"], state["K"])
        seg.iterate(ITERS)
        labels = seg.labels(out=state["out"])
        seg.close()
        return labels
    if kind == "prior":
        return scalp.gradient_prior(state["rgb"])
    if kind == "quality":
        return scalp.quality_metrics(state["labels"], state["gt"])
    h, w = state["labels"].shape
    scalp.scalp_label_means_static(state["rgb"].data_ptr(), 0, state["labels"].data_ptr(), h, w, state["n"],
                                   state["out"].data_ptr(), torch.cuda.current_stream().cuda_stream)
    return state["out"]


# --- what a pass cannot do without ---------------------------------------------
def _solve_flops(pixels, r, dims):
    """Per iteration and pixel: one walked path (the winner's: a third of the
    grid step on average, 10 operations a sample and 30 to assemble D) and a
    bound of 12 for each other candidate (a window of side 2r holds 2^dims
    clusters)."""
    return pixels * ITERS * (10.0 * (r / 3.0 + 1.0) + 30.0 + 12.0 * (2 ** dims - 1))


def work(case):
    """Bytes: the inputs read once, the outputs written once.  Operations: the
    decomposition's as above; the CIELab conversion as 60 a pixel."""
    kind = case["kind"]
    if kind in ("batch", "serve"):
        sizes = _mix(case)
        n = sum(h * w for h, w, _ in sizes)
        return {"bytes": 11 * n, "flops": sum(_solve_flops(h * w, math.sqrt(h * w / k), 2) + 60 * h * w
                                              for h, w, k in sizes)}
    n = case["H"] * case["W"]
    if kind == "solve":
        return {"bytes": (11 if case["prior"] == "input" else 7) * n,
                "flops": _solve_flops(n, math.sqrt(n / case["K"]), 2) + 60 * n}
    if kind == "multiscale":
        ks = scalp.multiscale_K(case["k_min"], case["k_max"], case["scales"])
        return {"bytes": (7 + 4 + 4 * len(ks)) * n,
                "flops": sum(_solve_flops(n, math.sqrt(n / k), 2) for k in ks) + 60 * n}
    if kind == "video":
        n *= case["T"]
        return {"bytes": 11 * n, "flops": _solve_flops(n, (n / case["K"]) ** (1 / 3), 3) + 60 * n}
    if kind == "prior":
        return {"bytes": 7 * n, "flops": 80 * n}
    if kind == "quality":
        return {"bytes": 8 * n, "flops": 20 * n}
    return {"bytes": 7 * n + 48 * case["K"], "flops": 70 * n}


# --- the same outputs in 64 bits, where they are numbers --------------------------
def _lab64(rgb):
    c = rgb.double() / 255.0
    lin = torch.where(c <= 0.04045, c / 12.92, ((c + 0.055) / 1.055) ** 2.4)
    m = torch.tensor([[0.4124564, 0.3575761, 0.1804375], [0.2126729, 0.7151522, 0.0721750],
                      [0.0193339, 0.1191920, 0.9503041]], dtype=torch.float64, device=rgb.device)
    t = (lin @ m.T) / m.sum(1)
    f = torch.where(t > (6 / 29) ** 3, t.clamp(min=1e-12) ** (1 / 3), t * (841 / 108) + 4 / 29)
    return torch.stack([116 * f[..., 1] - 16, 500 * (f[..., 0] - f[..., 1]), 200 * (f[..., 1] - f[..., 2])], -1)


def _boundary(l):
    b = torch.zeros(l.shape, dtype=torch.bool, device=l.device)
    dx, dy = l[:, 1:] != l[:, :-1], l[1:] != l[:-1]
    b[:, 1:] |= dx
    b[:, :-1] |= dx
    b[1:] |= dy
    b[:-1] |= dy
    return b


def _exact_prior(rgb):
    lab = _lab64(rgb)
    s = torch.zeros(rgb.shape[:2], dtype=torch.float64, device=rgb.device)
    for axis in (0, 1):
        if rgb.shape[axis] > 1:
            s += torch.gradient(lab, dim=axis)[0].square().sum(-1)
    g = s.sqrt()
    return g / g.max() if g.max() > 0 else g


def _exact_quality(lab, gt, eps=2.0):
    h, w = lab.shape
    n, n_gt = int(lab.max()) + 1, int(gt.max()) + 1
    l, g = lab.long(), gt.long()
    ov = torch.bincount((l * n_gt + g).view(-1), minlength=n * n_gt).view(n, n_gt)
    area = ov.sum(1)
    edges = torch.zeros((h, w), dtype=torch.int64, device=lab.device)
    edges[0] += 1
    edges[-1] += 1
    edges[:, 0] += 1
    edges[:, -1] += 1
    dx, dy = (l[:, 1:] != l[:, :-1]).long(), (l[1:] != l[:-1]).long()
    edges[:, 1:] += dx
    edges[:, :-1] += dx
    edges[1:] += dy
    edges[:-1] += dy
    perim = torch.zeros(n, dtype=torch.int64, device=lab.device).index_add_(0, l.view(-1), edges.view(-1))
    b_gt, b_lab = _boundary(gt), _boundary(lab)
    near = torch.zeros_like(b_lab)
    r = math.ceil(eps)
    for oy in range(-r, r + 1):
        for ox in range(-r, r + 1):
            if math.hypot(ox, oy) < eps:
                ys, xs = slice(max(0, -oy), min(h, h - oy)), slice(max(0, -ox), min(w, w - ox))
                yt, xt = slice(max(0, oy), min(h, h + oy)), slice(max(0, ox), min(w, w + ox))
                near[ys, xs] |= b_lab[yt, xt]
    hits, total = int((b_gt & near).sum()), int(b_gt.sum())
    ue = torch.where(ov > 0, area[:, None] - ov, torch.zeros_like(ov)).sum()
    a, p = area.double(), perim.double()
    co = torch.where(area > 0, 4 * math.pi * a * a / (p * p), torch.zeros_like(a)).sum()
    return {"br": hits / total if total else 1.0, "asa": int(ov.max(1)[0].sum()) / (h * w), "ue": int(ue) / (h * w),
            "co": float(co) / (h * w)}


def _exact_means(rgb, labels, n):
    h, w = labels.shape
    k = labels.long().view(-1)
    xs = torch.arange(w, dtype=torch.float64, device=rgb.device)[None, :].expand(h, w)
    ys = torch.arange(h, dtype=torch.float64, device=rgb.device)[:, None].expand(h, w)
    cols = torch.cat([torch.ones((h, w, 1), dtype=torch.float64, device=rgb.device), _lab64(rgb), xs[..., None],
                      ys[..., None]], -1).view(-1, 6)
    s = torch.zeros((n, 6), dtype=torch.float64, device=rgb.device).index_add_(0, k, cols)
    s[:, 1:] /= s[:, :1]
    return s


def exact(case, seed):
    """None for the decompositions: their outputs are labels, decided by ten
    iterations that each start from the labels before."""
    if case["kind"] not in ("prior", "quality", "means"):
        return None
    s = prepare(case, seed)
    if case["kind"] == "prior":
        return _exact_prior(s["rgb"])
    if case["kind"] == "quality":
        return _exact_quality(s["labels"], s["gt"])
    return _exact_means(s["rgb"], s["labels"], s["n"])
