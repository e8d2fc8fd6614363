"""What a user of the rasterizer has it do, as measurable cases.

A case names a scene recipe (the seeded synthetic scenes of
paper_2409_08669_gb300/scenes.py, drawn here with torch so that inputs are made
on the GPU), its size, the image size, the settings and the entry point:

  frame    Rasterizer.forward: image, final transmittance and load of one camera
  noalloc  adr_render_frame_noalloc: the allocation-free small frame
  host     adr_render_host: the frame from and to pinned host memory
  train    one training step: rasterize, the total loss, its backward
  loss     the L1 + SSIM image loss with its gradient
  serve    a burst of requests to the serving scheduler

`exact` restates each in float64 torch.  The thresholds of the paper's renderer
(tile rectangles, alpha_low, t_min) are part of what is restated; the depth
order is that of the float32 view depth, which the library documents.
"""
import ctypes
import math

import numpy as np
import torch

from paper_2409_08669_gb300 import _lib
from paper_2409_08669_gb300 import scenes as S
from paper_2409_08669_gb300.autograd import l1_ssim_loss, load_balance_loss, rasterize
from paper_2409_08669_gb300.raster import Rasterizer
from paper_2409_08669_gb300.serve import Server

W_L1, W_SSIM, W_LOAD = 0.44, 0.11, 0.45     # the weights of the total loss
SERVE_SIZES = ((800, 800), (1280, 720), (1920, 1080))


def _unnamed(kind, scene, n, w, h, mode="aabb", degree=3, rect="pixel"):
    return {"kind": kind, "scene": scene, "n": n, "width": w, "height": h, "mode": mode,
            "sh_degree": degree, "rect": rect}


def _frame(name, *what):
    return {"name": name, **_unnamed(*what)}


def listed():
    return [
        # the smallest call: a thumbnail-sized frame by an application that may not allocate
        _frame("noalloc-2k-64x48", "noalloc", "uniform", 2_000, 64, 48),
        # an interactive preview of a small object (bench.py's tiny workload)
        _frame("frame-10k-256", "frame", "uniform", 10_000, 256, 256),
        # a preview while a capture is still being fitted: odd sizes, low SH degree, circle radius
        _frame("frame-150k-1001x667", "frame", "heavy", 150_001, 1001, 667, "circle", 1),
        # a frame in the original 3DGS rasterizer's mode and tile rounding, for comparison
        _frame("frame-600k-plain-720p", "frame", "cluster", 600_000, 1280, 720, "plain", 3, "3dgs"),
        # an ordinary captured scene at full HD
        _frame("frame-1m-1080p", "frame", "cluster", 1_000_000, 1920, 1080),
        # the paper's model size with uneven per-pixel load: the benchmark workload
        _frame("frame-3m-1080p", "frame", "heavy", 3_000_000, 1920, 1080),
        # the same scene at 4K, the largest frame
        _frame("frame-3m-4k", "frame", "heavy", 3_000_000, 3840, 2160),
        # a scene that lives in the application's host memory
        _frame("host-1m-720p", "host", "cluster", 1_000_000, 1280, 720),
        # one training step of a small crop, where launches count
        _frame("train-6k-136x120", "train", "uniform", 6_000, 136, 120),
        # one training step of an ordinary scene
        _frame("train-1m-720p", "train", "cluster", 1_000_000, 1280, 720),
        # the image loss alone: evaluating or fitting full-HD images
        {"name": "loss-1080p", "kind": "loss", "width": 1920, "height": 1080},
        # a burst of viewers on two resident scenes, mixed resolutions
        {"name": "serve-16", "kind": "serve", "n": 500_000, "requests": 16, "batch": 1},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "frame", "noalloc", "host", "train", "train", "loss", "serve"])
    if kind == "serve":
        return {"kind": kind, "n": _log_int(rng, 100_000, 700_000), "requests": rng.randint(6, 16),
                "batch": rng.choice([1, 1, 4])}
    w = _log_int(rng, 64, 1920)
    h = max(48, min(1080, int(w * rng.uniform(0.5, 1.0))))
    if kind == "loss":
        return {"kind": kind, "width": w, "height": h}
    mode = rng.choice(["aabb", "aabb", "aabb", "circle", "plain"])
    degree = rng.choice([3, 3, 3, 2, 1, 0])
    rect = rng.choice(["pixel", "pixel", "pixel", "3dgs"])
    if kind == "noalloc":
        return _unnamed(kind, "uniform", _log_int(rng, 1_000, 20_000), min(w, 400), min(h, 300), mode, degree, rect)
    scene = rng.choice(["uniform", "cluster", "cluster", "heavy", "heavy"])
    n = _log_int(rng, 2_000, 20_000) if scene == "uniform" else _log_int(rng, 20_000, 3_000_000 if kind == "frame" else 1_000_000)
    if kind == "frame" and mode == "aabb" and rng.random() < 0.25:      # up to 4K
        w, h = _log_int(rng, 1920, 3840), _log_int(rng, 1080, 2160)
    if kind == "train":
        w, h = min(w, 1280), min(h, 720)
    return _unnamed(kind, scene, n, w, h, mode, degree, rect)


# ---- inputs -------------------------------------------------------------------

def _gen(seed, device="cuda"):
    return torch.Generator(device).manual_seed(int(seed) % (1 << 62))


def _normal(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _uniform(g, lo, hi, *shape):
    return torch.rand(*shape, generator=g, device="cuda") * (hi - lo) + lo


def _attributes(g, n, scale_mean=-4.0, scale_std=0.5):
    scales = torch.exp(_normal(g, n, 3) * scale_std + scale_mean)
    rots = torch.nn.functional.normalize(_normal(g, n, 4), dim=1)
    opac = torch.sigmoid(_normal(g, n) * 1.5)
    sh = _normal(g, n, 16, 3) * 0.2
    sh[:, 0] += 0.5
    return scales, rots, opac, sh


def _cluster_means(g, n, clusters=64):
    centres = _uniform(g, -3.0, 3.0, clusters, 3)
    rot = torch.linalg.qr(_normal(g, clusters, 3, 3)).Q
    stds = _uniform(g, 0.1, 0.6, clusters, 3)
    which = torch.randint(0, clusters, (n,), generator=g, device="cuda")
    pts = centres[which] + torch.einsum("nij,nj->ni", rot[which], _normal(g, n, 3) * stds[which])
    background = torch.rand(n, generator=g, device="cuda") < 0.1
    return torch.where(background[:, None], _uniform(g, -10.0, 10.0, n, 3), pts)


def _scene(name, n, g):
    """(means, scales, rots, opac, sh) of a recipe of scenes.py."""
    if name == "uniform":
        means = _uniform(g, -1.0, 1.0, n, 3)
        attrs = _attributes(g, n)
    else:
        means = _cluster_means(g, n)
        attrs = _attributes(g, n)
        if name == "heavy":          # 30% in one dense central cluster of larger Gaussians
            dense = torch.rand(n, generator=g, device="cuda") < 0.3
            means = torch.where(dense[:, None], _normal(g, n, 3) * 0.22, means)
            attrs = (torch.where(dense[:, None], torch.exp(_normal(g, n, 3) * 0.7 - 3.0), attrs[0]), *attrs[1:])
    return tuple(t.contiguous() for t in (means, *attrs))


def _camera(case, seed):
    """A camera on the radius-4 orbit (the small uniform scenes: at distance 3), at an angle of the seed's."""
    a = 2.0 * math.pi * random_unit(seed)
    r = 3.0 if case["scene"] == "uniform" else 4.0
    return S.look_at((r * math.cos(a), 0.0, r * math.sin(a)), width=case["width"], height=case["height"])


def random_unit(seed):
    return float(np.random.default_rng(int(seed)).random())


def _settings(case):
    return S.Settings(mode={"plain": S.MODE_PLAIN, "circle": S.MODE_CIRCLE, "aabb": S.MODE_AABB}[case["mode"]],
                      sh_degree=case["sh_degree"],
                      rect_rule=S.RECT_3DGS if case["rect"] == "3dgs" else S.RECT_PIXEL)


def _pair_capacity(n, w, h):
    """Room for a scene's Gaussian-tile pairs (measured: 53 per Gaussian at 1080p
    on the heavy scene, 96 in plain mode; they grow with the image's area)."""
    return int(min(1 << 30, max(1 << 20, n * (24 + 160 * w * h / (1920 * 1080)))))


def _photo(g, w, h):
    """An image with the spectrum of a photograph: random fields from coarse to fine, in [0, 1]."""
    img = torch.zeros(1, 3, h, w, device="cuda")
    for cells, weight in ((4, 0.5), (16, 0.25), (64, 0.15), (256, 0.1)):
        field = torch.rand(1, 3, cells, cells, generator=g, device="cuda")
        img += weight * torch.nn.functional.interpolate(field, size=(h, w), mode="bilinear", align_corners=False)
    return img[0].contiguous()


def _loss_images(case, seed):
    """A target and a render that is close to it: a little noise and a little blur."""
    g = _gen(seed)
    ref = _photo(g, case["width"], case["height"])
    img = torch.nn.functional.avg_pool2d(ref[None], 3, 1, 1, count_include_pad=False)[0]
    return (img + 0.02 * torch.randn(ref.shape, generator=g, device="cuda")).contiguous(), ref


def _train_inputs(case, seed):
    g = _gen(seed)
    params = _scene(case["scene"], case["n"], g)
    return params, _camera(case, seed), _settings(case), _photo(g, case["width"], case["height"])


def _serve_inputs(case, seed):
    """Two resident scenes and the burst's (scene, camera) list."""
    g = _gen(seed)
    scenes = [_scene("cluster", case["n"], g), _scene("heavy", max(1, case["n"] // 2), g)]
    rng = np.random.default_rng(int(seed))
    asked = []
    for k in range(case["requests"]):
        w, h = SERVE_SIZES[k % 3]
        asked.append((int(rng.integers(0, 2)), S.sphere_camera(rng, 4.0, w, h)))
    return scenes, asked


def prepare(case, seed):
    kind = case["kind"]
    if kind == "loss":
        img, ref = _loss_images(case, seed)
        return {"kind": kind, "img": img.requires_grad_(True), "ref": ref}
    if kind == "serve":
        scenes, asked = _serve_inputs(case, seed)
        server = Server(max_slots=16, mem_budget_bytes=64 << 30, slot_pair_capacity=1 << 26,
                        slot_max_gaussians=max(case["n"], 1), max_width=1920, max_height=1080,
                        use_graphs=True, max_batch=case["batch"])
        torch.cuda.synchronize()     # the server's streams read the scenes
        ids = [server.add_scene(p, S.Settings(mode=S.MODE_AABB)) for p in scenes]
        return {"kind": kind, "server": server, "asked": [(ids[s], cam) for s, cam in asked],
                "out": [torch.empty(3, cam.height, cam.width, device="cuda") for _, cam in asked]}
    st = _settings(case)
    n, w, h = case["n"], case["width"], case["height"]
    if kind == "train":
        params, cam, st, target = _train_inputs(case, seed)
        state = {"params": tuple(p.requires_grad_(True) for p in params), "target": target}
    else:
        cam = _camera(case, seed)
        params = _scene(case["scene"], n, _gen(seed))
        state = {"params": params}
    state.update(kind=kind, cam=cam, st=st)
    if kind == "noalloc":
        return state
    state["rast"] = Rasterizer(max_gaussians=n, pair_capacity=_pair_capacity(n, w, h), max_width=w, max_height=h)
    if kind == "host":
        state["params"] = tuple(p.cpu().pin_memory() for p in params)
        state["img"] = torch.empty(3, h, w).pin_memory()
    return state


# ---- one pass -----------------------------------------------------------------

def run(state):
    kind = state["kind"]
    if kind == "frame":
        return state["rast"].forward(state["params"], state["cam"], state["st"])
    if kind == "train":
        params, rast = state["params"], state["rast"]
        for p in params:
            p.grad = None
        img, load, t_final = rasterize(params, rast, state["cam"], state["st"])
        loss = l1_ssim_loss(img, state["target"], W_L1, W_SSIM) + W_LOAD * load_balance_loss(load, rast)
        loss.backward()
        return {"loss": loss.detach(), "img": img.detach(), "load": load.detach(), "t_final": t_final,
                "grads": [p.grad for p in params]}
    if kind == "loss":
        state["img"].grad = None
        loss = l1_ssim_loss(state["img"], state["ref"], 0.8, 0.2)
        loss.backward()
        return loss.detach(), state["img"].grad
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(s, cam, out) for (s, cam), out in zip(state["asked"], state["out"])]
        for t in tickets:
            server.wait(t)
        return state["out"]
    cam, st, params = state["cam"], state["st"], state["params"]
    c, s = _lib.make_camera(cam), _lib.make_settings(st)
    stream = torch.cuda.current_stream().cuda_stream
    n = params[0].shape[0]
    if kind == "host":
        img = state["img"]
        _lib.adr_render_host(state["rast"].ctx, *(p.data_ptr() for p in params), n, c, s, img.data_ptr(), 0, 0, stream)
        return img
    img = torch.empty(3, cam.height, cam.width, device="cuda")
    t_final = torch.empty(cam.height, cam.width, device="cuda")
    load = torch.empty(cam.height, cam.width, dtype=torch.int32, device="cuda")
    _lib.check(_lib.load().adr_render_frame_noalloc(
        *(p.data_ptr() for p in params), n, ctypes.byref(c), ctypes.byref(s), img.data_ptr(),
        t_final.data_ptr(), load.data_ptr(), stream), "adr_render_frame_noalloc")
    return img, t_final, load


def work(case):
    """Bytes: each input read once, each output written once.  Flops: about 300 per
    Gaussian projected and 30 per Gaussian evaluated at a pixel, of which the
    scenes here have about 110 a pixel (measured at 1080p)."""
    kind = case["kind"]
    if kind == "serve":
        px = sum(w * h for w, h in SERVE_SIZES) / 3 * case["requests"]
        n = 0.75 * case["n"] * case["requests"]
        return {"bytes": 1.5 * case["n"] * 236 + px * 12, "flops": n * 300 + px * 110 * 30}
    px = case["width"] * case["height"]
    if kind == "loss":   # two images in, the gradient out; five blurs forward and three back, 11 taps in each direction
        return {"bytes": 3 * px * 4 * 3, "flops": 3 * px * 8 * 22 * 2}
    n, sh = case["n"], 12 * (case["sh_degree"] + 1) ** 2
    if kind == "train":
        return {"bytes": n * (2 * 236) + px * (12 + 12 + 8), "flops": n * 900 + px * 110 * 100}
    return {"bytes": n * (44 + sh) + px * (12 if kind == "host" else 20), "flops": n * 300 + px * 110 * 30}


# ---- the same in float64 ------------------------------------------------------

def _sh_basis(d):
    """Real spherical harmonics up to degree 3 of unit directions [n, 3], Condon-Shortley phase: [n, 16]."""
    x, y, z = d.unbind(1)
    xx, yy, zz = x * x, y * y, z * z
    pi = math.pi
    c0, c1 = 0.5 / math.sqrt(pi), math.sqrt(3 / (4 * pi))
    a2, b2, c2 = math.sqrt(15 / (4 * pi)), math.sqrt(5 / (16 * pi)), math.sqrt(15 / (16 * pi))
    a3, b3, c3 = math.sqrt(35 / (32 * pi)), math.sqrt(105 / (4 * pi)), math.sqrt(21 / (32 * pi))
    d3, e3 = math.sqrt(7 / (16 * pi)), math.sqrt(105 / (16 * pi))
    return torch.stack([
        torch.full_like(x, c0), -c1 * y, c1 * z, -c1 * x,
        a2 * x * y, -a2 * y * z, b2 * (2 * zz - xx - yy), -a2 * x * z, c2 * (xx - yy),
        -a3 * y * (3 * xx - yy), b3 * x * y * z, -c3 * y * (4 * zz - xx - yy),
        d3 * z * (2 * zz - 3 * xx - 3 * yy), -c3 * x * (4 * zz - xx - yy), e3 * z * (xx - yy),
        -a3 * x * (xx - 3 * yy)], 1)


def _project(params, cam, st):
    """Projection, conic, colour and tile rectangle of every Gaussian: (values [n, 9]
    = px, py, conic a, b, c, opacity, rgb, differentiable; rect [n, 4]; kept; float32 depth)."""
    means, scales, rots, opac, sh = params
    dev = means.device
    view = torch.tensor(cam.view, dtype=torch.float64, device=dev)
    fx, fy = cam.fx, cam.fy
    p = means @ view[:3, :3].T + view[:3, 3]
    v32, m32 = torch.tensor(cam.view, dtype=torch.float32, device=dev)[2], means.detach().float()
    depth = ((v32[0] * m32[:, 0] + v32[1] * m32[:, 1]) + v32[2] * m32[:, 2]) + v32[3]
    front = depth > cam.near
    z = torch.where(front, p[:, 2], torch.ones_like(p[:, 2]))
    u = torch.stack([fx * p[:, 0] / z + cam.cx, fy * p[:, 1] / z + cam.cy], 1)
    q = rots / rots.norm(dim=1, keepdim=True)
    w, x, y, k = q.unbind(1)
    rot = torch.stack([1 - 2 * (y * y + k * k), 2 * (x * y - w * k), 2 * (x * k + w * y),
                       2 * (x * y + w * k), 1 - 2 * (x * x + k * k), 2 * (y * k - w * x),
                       2 * (x * k - w * y), 2 * (y * k + w * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    m = rot * scales[:, None, :]
    lx, ly = st.jac_clamp * cam.width / (2 * fx), st.jac_clamp * cam.height / (2 * fy)
    tx, ty = (p[:, 0] / z).clamp(-lx, lx), (p[:, 1] / z).clamp(-ly, ly)
    zero = torch.zeros_like(z)
    jac = torch.stack([fx / z, zero, -fx * tx / z, zero, fy / z, -fy * ty / z], 1).view(-1, 2, 3)
    um = jac @ view[:3, :3] @ m
    cov = um @ um.transpose(1, 2)
    a, b, c = cov[:, 0, 0] + st.lowpass, cov[:, 0, 1], cov[:, 1, 1] + st.lowpass
    det = a * c - b * b
    cam_pos = torch.tensor(cam.cam_pos, dtype=torch.float64, device=dev)
    dirs = means - cam_pos
    basis = _sh_basis(dirs / dirs.norm(dim=1, keepdim=True))[:, :(st.sh_degree + 1) ** 2]
    rgb = ((basis[:, :, None] * sh[:, :basis.shape[1]]).sum(1) + 0.5).clamp(min=0)
    vals = torch.cat([u, torch.stack([c / det, -b / det, a / det, opac], 1), rgb], 1)
    with torch.no_grad():
        lam = (a + c) / 2 + (((a - c) / 2) ** 2 + b * b).sqrt()
        r_o = torch.ceil(3 * lam.sqrt())
        kept = front & (det > 0)
        rx = ry = r_o
        if st.mode != S.MODE_PLAIN:
            kept &= opac >= st.alpha_low
            gain = 2 * torch.log((opac / st.alpha_low).clamp(min=1))
            rx, ry = ((gain * lam).sqrt(),) * 2 if st.mode == S.MODE_CIRCLE else ((gain * a).sqrt(), (gain * c).sqrt())
            rx, ry = torch.minimum(rx, r_o), torch.minimum(ry, r_o)
        spans = []
        for centre, r, size in ((u[:, 0], rx, cam.width), (u[:, 1], ry, cam.height)):
            tiles = (size + 15) // 16
            if st.rect_rule == S.RECT_3DGS:
                r = torch.ceil(r)
                lo = torch.floor((centre - r) / 16).clamp(0, tiles)
                hi = torch.floor((centre + r + 15) / 16).clamp(0, tiles)
            else:
                first, last = torch.ceil(centre - r).clamp(min=0), torch.floor(centre + r).clamp(max=size - 1)
                kept &= first <= last
                lo, hi = torch.floor(first / 16), torch.floor(last / 16) + 1
            kept &= lo < hi
            spans += [lo, hi]
        rect = torch.stack(spans, 1)
    return vals, rect, kept, depth


def _blend(vals, px, py, st):
    """Front-to-back blending of the listed Gaussians at pixels (px, py): colour, transmittance, alphas, blended."""
    dx, dy = vals[:, 0, None] - px, vals[:, 1, None] - py
    q = vals[:, 2, None] * dx * dx + 2 * vals[:, 3, None] * dx * dy + vals[:, 4, None] * dy * dy
    alpha = (vals[:, 5, None] * torch.exp(-0.5 * q)).clamp(max=0.99)
    alpha = torch.where(alpha >= st.alpha_low, alpha, torch.zeros_like(alpha))
    through = torch.cumprod(1 - alpha.detach(), 0)
    going = torch.cumsum((through < st.t_min) & (alpha > 0), 0) == 0      # before the pixel's stop
    alpha = torch.where(going, alpha, torch.zeros_like(alpha))
    after = torch.cumprod(1 - alpha, 0)
    before = torch.cat([torch.ones_like(after[:1]), after[:-1]])
    rgb = (vals[:, 6:, None] * (alpha * before)[:, None]).sum(0)
    return rgb, after[-1], alpha, ~going[-1]


def _tiles(rect, order, cam):
    """Yields (tile's pixel x, pixel y, its Gaussians in depth order)."""
    x0, x1, y0, y1 = rect[order].unbind(1)
    ys = torch.arange(16, device=rect.device)
    for tx in range((cam.width + 15) // 16):
        col = torch.nonzero((x0 <= tx) & (x1 > tx))[:, 0]
        cy0, cy1 = y0[col], y1[col]
        for ty in range((cam.height + 15) // 16):
            px = (ys + 16 * tx)[None, :].expand(16, 16).reshape(-1)
            py = (ys + 16 * ty)[:, None].expand(16, 16).reshape(-1)
            inside = (px < cam.width) & (py < cam.height)
            yield px[inside], py[inside], order[col[torch.nonzero((cy0 <= ty) & (cy1 > ty))[:, 0]]]


def _exact_frame(params, cam, st):
    """(img, t_final, load) in float64."""
    vals, rect, kept, depth = _project(tuple(p.detach().double() for p in params), cam, st)
    index = torch.nonzero(kept)[:, 0]
    order = index[torch.sort(depth[index], stable=True).indices]
    img = torch.zeros(3, cam.height, cam.width, dtype=torch.float64, device=vals.device)
    t_final = torch.ones(cam.height, cam.width, dtype=torch.float64, device=vals.device)
    load = torch.zeros(cam.height, cam.width, dtype=torch.int64, device=vals.device)
    for px, py, ids in _tiles(rect, order, cam):
        T, stopped = t_final[py, px], torch.zeros_like(px, dtype=torch.bool)
        rgb, count = img[:, py, px], load[py, px]
        for k in range(0, len(ids), 1024):        # a piece of the list at a time, until every pixel stopped
            c, t, alpha, stop = _blend_more(vals[ids[k:k + 1024]], px, py, T, stopped, st)
            rgb, T, count, stopped = rgb + c, t, count + (alpha > 0).sum(0), stopped | stop
            if k + 1024 < len(ids) and bool(stopped.all()):
                break
        img[:, py, px], t_final[py, px], load[py, px] = rgb, T, count
    bg = torch.tensor(st.bg, dtype=torch.float64, device=vals.device)
    return img + t_final * bg[:, None, None], t_final, load


def _blend_more(vals, px, py, T, stopped, st):
    """_blend from a transmittance T on; pixels that stopped stay as they are."""
    dx, dy = vals[:, 0, None] - px, vals[:, 1, None] - py
    q = vals[:, 2, None] * dx * dx + 2 * vals[:, 3, None] * dx * dy + vals[:, 4, None] * dy * dy
    alpha = (vals[:, 5, None] * torch.exp(-0.5 * q)).clamp(max=0.99)
    alpha = torch.where((alpha >= st.alpha_low) & ~stopped, alpha, torch.zeros_like(alpha))
    stop = torch.cumsum((T * torch.cumprod(1 - alpha, 0) < st.t_min) & (alpha > 0), 0) > 0
    alpha = torch.where(stop, torch.zeros_like(alpha), alpha)
    after = T * torch.cumprod(1 - alpha, 0)
    before = torch.cat([T[None], after[:-1]])
    return (vals[:, 6:, None] * (alpha * before)[:, None]).sum(0), after[-1], alpha, stop[-1]


def _exact_loss(img, ref, w_l1, w_ssim):
    """w_l1 * mean |img - ref| + w_ssim * (1 - mean SSIM), float64, differentiable."""
    d = torch.arange(11, dtype=torch.float64, device=img.device) - 5
    win = torch.exp(-d * d / 4.5)
    win = win / win.sum()

    def blur(x):
        x = torch.nn.functional.conv2d(x[:, None], win[None, None, None, :], padding=(0, 5))
        return torch.nn.functional.conv2d(x, win[None, None, :, None], padding=(5, 0))[:, 0]

    mx, my = blur(img), blur(ref)
    vx, vy, cxy = blur(img * img) - mx * mx, blur(ref * ref) - my * my, blur(img * ref) - mx * my
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    ssim = ((2 * mx * my + c1) * (2 * cxy + c2)) / ((mx * mx + my * my + c1) * (vx + vy + c2))
    return w_l1 * (img - ref).abs().mean() + w_ssim * (1 - ssim.mean())


def _exact_train(case, seed):
    params, cam, st, target = _train_inputs(case, seed)
    img, t_final, load = _exact_frame(params, cam, st)
    img.requires_grad_(True)
    loss = _exact_loss(img, target.double(), W_L1, W_SSIM)
    (d_img,) = torch.autograd.grad(loss, img)
    l = load.double()
    std = l.std(unbiased=False)
    d_load = W_LOAD * (l - l.mean()) / (l.numel() * std) if std > 0 else torch.zeros_like(l)
    leaves = [p.detach().double().requires_grad_(True) for p in params]
    vals, rect, kept, depth = _project(leaves, cam, st)
    index = torch.nonzero(kept)[:, 0]
    order = index[torch.sort(depth[index], stable=True).indices]
    total = torch.zeros_like(vals)
    for px, py, ids in _tiles(rect, order, cam):
        if not len(ids):
            continue
        v = vals.detach()[ids].requires_grad_(True)
        rgb, _, alpha, _ = _blend(v, px, py, st)
        # straight-through: each blended alpha passes the load's gradient on
        out = (rgb * d_img[:, py, px]).sum() + (alpha.sum(0) * d_load[py, px]).sum()
        total.index_add_(0, ids, torch.autograd.grad(out, v)[0])
    picked = torch.nonzero(kept)[:, 0]
    grads = torch.autograd.grad(vals[picked], leaves, total[picked])
    return {"loss": loss.detach() + W_LOAD * std, "img": img.detach(), "load": l, "t_final": t_final, "grads": list(grads)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "loss":
        img, ref = _loss_images(case, seed)
        img = img.double().requires_grad_(True)
        loss = _exact_loss(img, ref.double(), 0.8, 0.2)
        return loss.detach(), torch.autograd.grad(loss, img)[0]
    if kind == "serve":      # the first request of the burst; the others are the same path
        scenes, asked = _serve_inputs(case, seed)
        s, cam = asked[0]
        return [_exact_frame(scenes[s], cam, S.Settings(mode=S.MODE_AABB))[0]] + [None] * (len(asked) - 1)
    if case["width"] * case["height"] > 2_500_000:
        return None          # tens of thousands of tiles, one by one
    if kind == "train":
        return _exact_train(case, seed) if case["width"] * case["height"] < 1_000_000 else None
    frame = _exact_frame(_scene(case["scene"], case["n"], _gen(seed)), _camera(case, seed), _settings(case))
    return frame[0] if kind == "host" else (frame[0], frame[1], None)
