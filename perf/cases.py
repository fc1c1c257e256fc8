"""The calls whose time matters to users of this renderer, as measurable cases.

A case is a dict of plain values; `prepare` builds what a program has in hand
before the call (resident scene, sized workspace, output buffers), `run` makes
one pass through the public entry points, `exact` states in plain torch FP64
what that pass returns, and `work` what it cannot do without.

Kinds:
  frame   one view into a device image (mgs_render)
  depth   colour and depth image, Eq. 5 (mgs_render_depth)
  train   forward, squared-error loss and adjoint (autograd.render)
  static  one view through the allocation-free entry point (mgs_render_static)
  open    SH decode, scene upload, first frame, unload (a viewer opening a scene)
  serve   a burst of requests through the continuous-batching server
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2603_11531_gb300 as mgs
from paper_2603_11531_gb300 import autograd, serving, synth

BG = (0.1, 0.2, 0.3)
# requests of a burst: (scene index, width, height); scenes of n, n / 2 and n / 4 Gaussians
BURST = ((0, 640, 480), (1, 1280, 720), (2, 640, 480), (0, 640, 480), (1, 640, 480), (2, 1280, 720),
         (2, 640, 480), (0, 1280, 720), (1, 640, 480), (0, 640, 480), (2, 640, 480), (1, 1280, 720))


def _case(name, kind, n, width, height, precision="fp16", mlp="bf16", residual=False,
          scene="unbounded"):
    return {"name": name, "kind": kind, "n": n, "width": width, "height": height,
            "precision": precision, "mlp": mlp, "residual": residual, "scene": scene}


def listed():
    return [
        # a thumbnail or a unit-test-sized preview: launches and latency
        _case("preview_4k_256", "frame", 4096, 256, 256, "fp32", "none", scene="uniform"),
        # an object scene in a small window
        _case("frame_50k_640x480", "frame", 50_000, 640, 480),
        # the benchmark view: a whole unbounded scene, interactive
        _case("frame_600k_1600x1063", "frame", 600_000, 1600, 1063),
        # the same view with the paper's MLP widths (256, 128, 64)
        _case("paper_mlp_600k_1600x1063", "frame", 600_000, 1600, 1063, mlp="paper"),
        # FP32 attributes (a scene being trained) viewed in an odd-sized window,
        # with the MLP's colour residual
        _case("frame_fp32_160k_1001x667", "frame", 160_000, 1001, 667, "fp32", residual=True),
        # depth image for depth distillation
        _case("depth_300k_1280x720", "depth", 300_000, 1280, 720),
        # training steps: full size, and early / low resolution
        _case("train_300k_1296x840", "train", 300_000, 1296, 840, "fp32"),
        _case("train_30k_333x251", "train", 30_000, 333, 251, "fp32", residual=True),
        # a host that may not allocate at render time
        _case("static_100k_1280x720", "static", 100_000, 1280, 720, mlp="none"),
        # a viewer opening the largest served scene: decode, load, first frame
        _case("open_3m_640x480", "open", 3_000_000, 640, 480),
        # a burst of twelve requests on three resident scenes
        _case("serve_12x160k", "serve", 160_000, 1280, 720),
        # the largest scene at 4K
        _case("large_6m_3840x2160", "frame", 6_000_000, 3840, 2160),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "depth", "train", "train", "static", "open", "serve"])
    width = _log_int(rng, 96, 1920)
    height = max(64, int(width * rng.uniform(0.5, 0.8)))
    precision = rng.choice(["fp16", "fp16", "fp32"])
    mlp = rng.choice(["bf16", "bf16", "none", "paper"])
    n_max = 1_700_000
    scene = "unbounded"
    if kind == "train":
        n_max, precision, mlp = 400_000, "fp32", rng.choice(["bf16", "none"])
    elif kind == "static":
        n_max, mlp = 120_000, "none"
    elif kind == "open":
        n_max = 3_000_000
    elif kind == "serve":
        n_max, precision, mlp, width, height = 600_000, "fp16", "bf16", 1280, 720
    elif kind == "frame" and rng.random() < 0.3:
        scene, n_max = "uniform", 100_000
    return {"kind": kind, "n": _log_int(rng, 3000, n_max), "width": width, "height": height,
            "precision": precision, "mlp": mlp,
            "residual": mlp == "bf16" and rng.random() < 0.4, "scene": scene}


# ---- inputs -------------------------------------------------------------------

def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _attrs(n, seed, precision, scene, device=None):
    """(n, 24) records of synth's distributions, drawn on the device."""
    dev = device or _device()
    g = torch.Generator(device=dev).manual_seed(seed)
    a = torch.zeros((n, 24), dtype=torch.float32, device=dev)
    if scene == "uniform":
        a[:, 0:3] = torch.rand((n, 3), generator=g, device=dev) * 2.0 - 1.0
    else:
        n_in = int(round(0.8 * n))
        d = torch.nn.functional.normalize(torch.randn((n, 3), generator=g, device=dev), dim=1)
        u = torch.rand((n, 1), generator=g, device=dev)
        radii = torch.tensor([4.0, 2.0, 4.0], device=dev)
        a[:n_in, 0:3] = d[:n_in] * u[:n_in] ** (1.0 / 3.0) * radii
        a[n_in:, 0:3] = d[n_in:] * (30.0 + 30.0 * u[n_in:])
    a[:, 3:6] = torch.exp(-3.0 + 0.5 * torch.randn((n, 3), generator=g, device=dev))
    a[:, 6:10] = torch.randn((n, 4), generator=g, device=dev)
    a[:, 10] = torch.sigmoid(torch.randn(n, generator=g, device=dev))
    a[:, 11:23] = 0.3 * torch.randn((n, 12), generator=g, device=dev)
    return a.half() if precision == "fp16" else a


def _camera(scene, width, height, seed):
    if scene == "uniform":
        th = 0.1 * (seed % 61)
        return synth.look_at((3.0 * math.sin(th), 0.0, -3.0 * math.cos(th)), (0.0, 0.0, 0.0), width,
                             height, 60.0)
    return synth.random_orbit_camera(np.random.Generator(np.random.PCG64(seed)), width, height)


def _mlp(kind, seed):
    if kind == "none":
        return None
    return synth.random_mlp_paper(seed) if kind == "paper" else synth.random_mlp(seed)


def _views(case, seed):
    """The scenes and (scene index, camera) views of a case."""
    n, prec, kind = case["n"], case["precision"], case["scene"]
    if case["kind"] != "serve":
        return ([(_attrs(n, seed, prec, kind), _mlp(case["mlp"], seed))],
                [(0, _camera(kind, case["width"], case["height"], seed))])
    scenes = [(_attrs(max(n >> k, 1), 3 * seed + k, prec, kind), _mlp(case["mlp"], 3 * seed + k))
              for k in range(3)]
    return scenes, [(s, _camera(kind, w, h, 100 * seed + k)) for k, (s, w, h) in enumerate(BURST)]


def _train_params(seed):
    """FP32 master weights of the 22-64-64-5 MLP."""
    g = torch.Generator().manual_seed(seed)
    ts = []
    for out_f, in_f, head in ((64, 22, False), (64, 64, False), (5, 64, True)):
        ts.append((torch.rand((out_f, in_f), generator=g) * 2.0 - 1.0) * math.sqrt(6.0 / in_f))
        ts.append(torch.tensor([1.0, 0.0, 0.0, 0.0, 0.0]) if head
                  else (torch.rand(out_f, generator=g) * 2.0 - 1.0) / math.sqrt(in_f))
    return ts


def _target(case, seed):
    g = torch.Generator(device=_device()).manual_seed(seed + 7)
    return torch.rand((case["height"], case["width"], 3), generator=g, device=_device())


def _features(n, seed, precision):
    g = torch.Generator(device=_device()).manual_seed(seed + 5)
    h = 0.5 * torch.randn((n, 6), generator=g, device=_device())
    return h.half() if precision == "fp16" else h


# ---- prepare and run ------------------------------------------------------------

class _Session:
    """A renderer, its resident scenes and, for bursts, a server on them."""

    def __init__(self):
        self.renderer = mgs.Renderer(0)
        self.server = None

    def __del__(self):
        if self.server is not None:
            self.server.close()
        self.renderer.close()


def prepare(case, seed):
    s = {"case": case, "session": _Session()}
    r = s["renderer"] = s["session"].renderer
    kind, mlp = case["kind"], case["mlp"] != "none"
    scenes, views = _views(case, seed)
    cam = s["cam"] = views[0][1]
    H, W = int(cam.height), int(cam.width)
    s["opts"] = mgs.render_opts(mlp, case["residual"], BG)
    s["rgb"] = torch.empty((H, W, 3), dtype=torch.float32, device="cuda")
    if kind == "train":
        s["attrs"] = scenes[0][0].requires_grad_(True)
        s["mlp"] = tuple(t.cuda().requires_grad_(True) for t in _train_params(seed)) if mlp else None
        s["target"] = _target(case, seed)
        run(s)
    elif kind == "static":
        s["attrs"] = scenes[0][0]
    elif kind == "open":
        s["attrs"], s["mlp"] = scenes[0]
        s["features"] = _features(case["n"], seed, case["precision"])
        s["decoders"] = synth.random_sh_decoders(seed)
        run(s)
    elif kind == "serve":
        s["scenes"] = [r.load_scene(a, m) for a, m in scenes]
        s["views"] = views
        s["images"] = [torch.empty((int(c.height), int(c.width), 3), dtype=torch.float32, device="cuda")
                       for _, c in views]
        s["session"].server = serving.Server(r.ctx, slots=8, max_batch=8)
        run(s)
    else:
        s["scene"] = r.load_scene(*scenes[0])
        if kind == "depth":
            s["depth"] = torch.empty((H, W), dtype=torch.float32, device="cuda")
        # sizes the workspace for this view
        mgs.mgs_render_checked(r.ws, s["scene"], cam, s["opts"], s["rgb"])
    return s


def run(s):
    case, r, cam, opts = s["case"], s["renderer"], s["cam"], s["opts"]
    kind = case["kind"]
    if kind == "frame":
        mgs.mgs_render(r.ws, s["scene"], cam, opts, s["rgb"])
        return s["rgb"]
    if kind == "depth":
        mgs.mgs_render_depth(r.ws, s["scene"], cam, opts, s["rgb"], s["depth"])
        return [s["rgb"], s["depth"]]
    if kind == "train":
        leaves = [s["attrs"], *(s["mlp"] or ())]
        img = autograd.render(r, s["attrs"], cam, s["mlp"], s["mlp"] is not None, case["residual"], BG)
        loss = 0.5 * (img - s["target"]).square().sum()
        return [img.detach(), *torch.autograd.grad(loss, leaves)]
    if kind == "static":
        mgs.mgs_render_static(s["attrs"], cam, opts, s["rgb"])
        return s["rgb"]
    if kind == "open":
        mgs.mgs_decode_sh(r.ctx, s["features"], *s["decoders"], s["attrs"])
        scene = r.load_scene(s["attrs"], s["mlp"])
        mgs.mgs_render_checked(r.ws, scene, cam, opts, s["rgb"])
        r.unload_scene(scene)
        return [s["attrs"], s["rgb"]]
    server = s["session"].server
    tickets = [server.submit(s["scenes"][k], c, opts, out) for (k, c), out in zip(s["views"], s["images"])]
    for t in tickets:
        server.wait(t)
    return s["images"]


# ---- what a pass returns, in FP64 -------------------------------------------------
#
# Visibility, tile rectangles and the per-pixel inclusion test follow the fixed
# FP32 sequence that the renderer documents (each operation rounded to FP32);
# every value is FP64.  MLP inputs and hidden activations are rounded to BF16.

SH_C0 = 0.5 / math.sqrt(math.pi)
SH_C1 = math.sqrt(3.0) * 0.5 / math.sqrt(math.pi)
CHUNK = 1 << 14   # (tile, Gaussian) pairs evaluated at once


def _r32(x):
    return x.float().double()


def _same(x):
    return x


def _f32(x):
    return float(np.float32(x))


def _quat(v, rnd):
    w, x, y, z = v[:, 6], v[:, 7], v[:, 8], v[:, 9]
    n2 = rnd(w * w + rnd(x * x + rnd(y * y + rnd(z * z))))
    qn = rnd(torch.sqrt(n2))
    return n2 > 0, [rnd(c / qn) for c in (w, x, y, z)]


def _project(v, cam, rnd):
    """View depth, pixel mean, Sigma_2D (a, b, c) and its determinant."""
    Wm = [_f32(x) for x in np.asarray(cam.R).reshape(9)]
    tc = [_f32(x) for x in np.asarray(cam.t).reshape(3)]
    fx, fy, cx, cy = _f32(cam.fx), _f32(cam.fy), _f32(cam.cx), _f32(cam.cy)
    qok, (w, x, y, z) = _quat(v, rnd)
    xx, yy, zz, xy, xz, yz = rnd(x * x), rnd(y * y), rnd(z * z), rnd(x * y), rnd(x * z), rnd(y * z)
    wx, wy, wz = rnd(w * x), rnd(w * y), rnd(w * z)
    R = [rnd(1 - 2 * rnd(yy + zz)), 2 * rnd(xy - wz), 2 * rnd(xz + wy),
         2 * rnd(xy + wz), rnd(1 - 2 * rnd(xx + zz)), 2 * rnd(yz - wx),
         2 * rnd(xz - wy), 2 * rnd(yz + wx), rnd(1 - 2 * rnd(xx + yy))]
    t = [rnd(Wm[3 * r] * v[:, 0] + rnd(Wm[3 * r + 1] * v[:, 1] + rnd(Wm[3 * r + 2] * v[:, 2] + tc[r])))
         for r in range(3)]
    rz = rnd(1.0 / t[2])
    u, vv = rnd(t[0] * rz), rnd(t[1] * rz)
    one = torch.ones((), dtype=torch.float64)
    limx = float(rnd(1.2999999523162842 * rnd(one * 0.5 * cam.width / fx)))
    limy = float(rnd(1.2999999523162842 * rnd(one * 0.5 * cam.height / fy)))
    uc, vc = u.clamp(-limx, limx), vv.clamp(-limy, limy)
    j00, j02 = rnd(fx * rz), -rnd(rnd(fx * uc) * rz)
    j11, j12 = rnd(fy * rz), -rnd(rnd(fy * vc) * rz)
    T0 = [rnd(j02 * Wm[6 + j] + rnd(j00 * Wm[j])) for j in range(3)]
    T1 = [rnd(j12 * Wm[6 + j] + rnd(j11 * Wm[3 + j])) for j in range(3)]
    M = [rnd(R[k] * v[:, 3 + k % 3]) for k in range(9)]
    V0 = [rnd(T0[2] * M[6 + j] + rnd(T0[1] * M[3 + j] + rnd(T0[0] * M[j]))) for j in range(3)]
    V1 = [rnd(T1[2] * M[6 + j] + rnd(T1[1] * M[3 + j] + rnd(T1[0] * M[j]))) for j in range(3)]
    dil = 0.30000001192092896
    a = rnd(rnd(V0[0] * V0[0] + rnd(V0[1] * V0[1] + rnd(V0[2] * V0[2]))) + dil)
    b = rnd(V0[0] * V1[0] + rnd(V0[1] * V1[1] + rnd(V0[2] * V1[2])))
    c = rnd(rnd(V1[0] * V1[0] + rnd(V1[1] * V1[1] + rnd(V1[2] * V1[2]))) + dil)
    det = rnd(a * c - rnd(b * b))
    return qok, t[2], rnd(fx * u + cx), rnd(fy * vv + cy), a, b, c, det


def _visible(v, cam):
    """Indices of the visible Gaussians, their tile rectangles and test factors."""
    qok, tz, mx, my, a, b, c, det = _project(v, cam, _r32)
    mid, hd = _r32(0.5 * _r32(a + c)), _r32(0.5 * _r32(a - c))
    lam = _r32(mid + _r32(torch.sqrt(_r32(hd * hd + _r32(b * b)))))
    rad = torch.ceil(_r32(3.0 * _r32(torch.sqrt(lam))))
    tx, ty = (cam.width + 15) // 16, (cam.height + 15) // 16
    x0 = torch.floor(_r32(mx - rad) * 0.0625).clamp(0, tx)
    y0 = torch.floor(_r32(my - rad) * 0.0625).clamp(0, ty)
    x1 = (torch.floor(_r32(mx + rad) * 0.0625) + 1).clamp(0, tx)
    y1 = (torch.floor(_r32(my + rad) * 0.0625) + 1).clamp(0, ty)
    ok = qok & (tz > _f32(cam.znear)) & (det > 0) & (x0 < x1) & (y0 < y1)
    i = ok.nonzero().squeeze(1)
    l11 = _r32(torch.sqrt(_r32(c / det)))
    l21 = -_r32(b / _r32(torch.sqrt(_r32(c * det))))
    l22 = _r32(1.0 / _r32(torch.sqrt(c)))
    rect = torch.stack([x0, y0, x1, y1], 1)[i].long()
    return i, rect, torch.stack([mx, my, l11, l21, l22], 1)[i]


def _bf16(x):
    return x + (x.detach().to(torch.bfloat16).double() - x.detach())   # identity in the backward


def _values(v, cam, layers, residual):
    """Per-Gaussian (m_x, m_y, conic A, B, C, o, w, r, g, b, d)."""
    Wm = torch.tensor(np.asarray(cam.R, np.float32).reshape(3, 3), dtype=torch.float64, device=v.device)
    tc = torch.tensor(np.asarray(cam.t, np.float32), dtype=torch.float64, device=v.device)
    _, d, mx, my, a, b, c, det = _project(v, cam, _same)
    P = torch.nn.functional.normalize(v[:, 0:3] + Wm.T @ tc, dim=1)
    Y = v[:, 11:23].reshape(-1, 4, 3)
    rgb = (SH_C0 * Y[:, 0] - SH_C1 * P[:, 1:2] * Y[:, 1] + SH_C1 * P[:, 2:3] * Y[:, 2]
           - SH_C1 * P[:, 0:1] * Y[:, 3] + 0.5)
    phi, o = torch.ones_like(d), v[:, 10]
    if layers:
        x = torch.cat([P, v[:, 3:6], torch.stack(_quat(v, _same)[1], 1), v[:, 11:23]], 1)
        for w, bias in layers[:-1]:
            x = torch.relu(_bf16(x) @ _bf16(w).T + bias)
        y = _bf16(x) @ _bf16(layers[-1][0]).T + layers[-1][1]
        phi, o = torch.relu(y[:, 0]), torch.sigmoid(y[:, 1])
        if residual:
            rgb = rgb + y[:, 2:5]
    w = phi * phi + phi / (d * d) + torch.exp(v[:, 3:6].max(dim=1).values / d)
    return torch.cat([torch.stack([mx, my, c / det, -b / det, a / det, o, w], 1),
                      rgb.clamp(min=0.0), d[:, None]], 1)


def _pairs(rect, geo, tx):
    """(Gaussian, tile) pairs of the rectangles that may hold an included pixel."""
    w, h = rect[:, 2] - rect[:, 0], rect[:, 3] - rect[:, 1]
    csum = torch.cumsum(w * h, 0).cpu().numpy()
    g0 = 0
    while g0 < len(csum):
        base = int(csum[g0 - 1]) if g0 else 0
        g1 = max(int(np.searchsorted(csum, base + (1 << 23), side="right")), g0 + 1)
        cnt = (w * h)[g0:g1]
        g = torch.repeat_interleave(torch.arange(g0, g1, device=rect.device), cnt)
        k = torch.arange(len(g), device=rect.device) - (torch.cumsum(cnt, 0) - cnt)[g - g0]
        x, y = rect[g, 0] + k % w[g], rect[g, 1] + torch.div(k, w[g], rounding_mode="floor")
        dx, dy = (16 * x + 8).double() - geo[g, 0], (16 * y + 8).double() - geo[g, 1]
        l11, l21, l22 = geo[g, 2], geo[g, 3], geo[g, 4]
        e1, s1 = (l11 * dx + l21 * dy).abs(), l11.abs() * (dx.abs() + 8) + l21.abs() * (dy.abs() + 8)
        keep = (e1 - 7.5 * (l11.abs() + l21.abs()) <= 3.01 + 1e-5 * s1) & \
               ((l22 * dy).abs() - 7.5 * l22 <= 3.01 + 1e-5 * l22 * (dy.abs() + 8))
        g, tile = g[keep], (y * tx + x)[keep]
        for p in range(0, len(g), CHUNK):
            yield g[p:p + CHUNK], tile[p:p + CHUNK]
        g0 = g1


def _alpha(val, geo, tile, tx):
    """Alpha of the tile's 256 pixels (0 where the FP32 test excludes them)."""
    k = torch.arange(256, device=tile.device)
    px = (16 * (tile % tx))[:, None].double() + (k % 16) + 0.5
    py = (16 * torch.div(tile, tx, rounding_mode="floor"))[:, None].double() + k // 16 + 0.5
    with torch.no_grad():
        dy = _r32(py - geo[:, 1:2])
        e2 = _r32(geo[:, 4:5] * dy)
        e1 = _r32(geo[:, 2:3] * _r32(px - geo[:, 0:1]) + _r32(geo[:, 3:4] * dy))
        inside = _r32(e1 * e1 + _r32(e2 * e2)) <= 9.0
        del e1, e2, dy
    dx, dy = px - val[:, 0:1], py - val[:, 1:2]
    q = (val[:, 2:3] * dx + 2.0 * val[:, 3:4] * dy) * dx + val[:, 4:5] * dy * dy
    return torch.where(inside, (val[:, 5:6] * torch.exp(-0.5 * q)).clamp(max=0.99), 0.0)


def _composite(val, rect, geo, cam, depth):
    """Per-tile sums (A_r, A_g, A_b, B, log T, sum d a w) and the images."""
    tx, ty = (cam.width + 15) // 16, (cam.height + 15) // 16
    acc = torch.zeros((tx * ty, 6 if depth else 5, 256), dtype=torch.float64, device=val.device)
    for g, tile in _pairs(rect, geo, tx):
        vg = val[g]
        a = _alpha(vg, geo[g], tile, tx)
        aw = a * vg[:, 6:7]
        parts = [aw * vg[:, 7:8], aw * vg[:, 8:9], aw * vg[:, 9:10], aw, torch.log1p(-a)]
        if depth:
            parts.append(aw * vg[:, 10:11])
        acc.index_add_(0, tile, torch.stack(parts, 1))
    B, T = acc[:, 3], torch.exp(acc[:, 4])
    covered = B > 0
    inv = torch.where(covered, 1.0 / torch.where(covered, B, 1.0), 0.0)
    bg = torch.tensor([_f32(c) for c in BG], dtype=torch.float64, device=val.device)
    img = (1 - T)[:, None] * acc[:, 0:3] * inv[:, None] + T[:, None] * bg[None, :, None]
    out = [_untile(img, cam)]
    if depth:
        out.append(_untile(acc[:, 5:6] * inv[:, None], cam)[:, :, 0])
    return acc, inv, T, bg, out


def _untile(x, cam):
    tx, ty = (cam.width + 15) // 16, (cam.height + 15) // 16
    x = x.reshape(ty, tx, -1, 16, 16).permute(0, 3, 1, 4, 2).reshape(16 * ty, 16 * tx, -1)
    return x[:cam.height, :cam.width].contiguous()


def _tiled(x, cam):
    tx, ty = (cam.width + 15) // 16, (cam.height + 15) // 16
    full = torch.zeros((16 * ty, 16 * tx, x.shape[2]), dtype=torch.float64, device=x.device)
    full[:cam.height, :cam.width] = x
    return full.reshape(ty, 16, tx, 16, -1).permute(0, 2, 4, 1, 3).reshape(tx * ty, -1, 256)


def _layers(m, device):
    if m is None:
        return None
    f = lambda b: torch.from_numpy(synth.bf16_bits_to_f32(b).astype(np.float64)).to(device)  # noqa: E731
    c = lambda b: torch.from_numpy(np.asarray(b, np.float64)).to(device)                     # noqa: E731
    ls = [(f(m.w1), c(m.b1)), (f(m.w2), c(m.b2)), (f(m.w3), c(m.b3))]
    return ls if m.w4 is None else ls + [(f(m.w4), c(m.b4))]


def _image(attrs, m, cam, residual, depth=False):
    v = attrs.double()
    i, rect, geo = _visible(v, cam)
    val = _values(v[i], cam, _layers(m, v.device), residual)
    return _composite(val, rect, geo, cam, depth)[4]


def _train(case, seed):
    scenes, views = _views(case, seed)
    cam = views[0][1]
    v = scenes[0][0].double().requires_grad_(True)
    dev = v.device
    params = [t.double().to(dev).requires_grad_(True) for t in _train_params(seed)] \
        if case["mlp"] != "none" else []
    layers = list(zip(params[0::2], params[1::2]))
    with torch.no_grad():
        i, rect, geo = _visible(v.detach(), cam)
    val = _values(v[i], cam, layers, case["residual"])
    fixed = val.detach()
    acc, inv, T, bg, (img,) = _composite(fixed, rect, geo, cam, False)
    # dL/dA, dL/dB, dL/dlog T of C = (1 - T) A / B + T c_bg
    G = _tiled(img - _target(case, seed).double(), cam)
    r = acc[:, 0:3] * inv[:, None]
    kA = ((1 - T) * inv)[:, None]
    gA, gB = G * kA, -(G * r).sum(1) * kA[:, 0]
    gT = (G * torch.where((acc[:, 3] > 0)[:, None], bg[None, :, None] - r, 0.0)).sum(1) * T
    tx = (cam.width + 15) // 16
    gval = torch.zeros_like(fixed)
    for g, tile in _pairs(rect, geo, tx):
        p = fixed[g].requires_grad_(True)
        a = _alpha(p, geo[g], tile, tx)
        s = (a * p[:, 6:7] * (p[:, 7:8] * gA[tile, 0] + p[:, 8:9] * gA[tile, 1] + p[:, 9:10] * gA[tile, 2]
                              + gB[tile])).sum() + (torch.log1p(-a) * gT[tile]).sum()
        gval.index_add_(0, g, torch.autograd.grad(s, p)[0])
    return [img, *torch.autograd.grad((val * gval).sum(), [v, *params])]


def _decode(h, mlps):
    f = lambda u: torch.from_numpy(np.asarray(u).view(np.float16).astype(np.float64)).to(h.device)  # noqa: E731
    out = []
    for m in mlps:
        out.append(torch.relu(h.double() @ f(m.w1).T + f(m.b1)) @ f(m.w2).T + f(m.b2))
    return torch.cat(out, 1)


def exact(case, seed):
    # too long in FP64: about 20 s for the (pixel, Gaussian) pairs of 6M Gaussians at 4K
    if case["n"] * case["width"] * case["height"] > 4_000_000 * 1920 * 1080:
        return None
    if case["kind"] == "train":
        return _train(case, seed)
    with torch.no_grad():
        scenes, views = _views(case, seed)
        if case["kind"] == "serve":
            return [_image(*scenes[k], cam, case["residual"])[0] for k, cam in views]
        attrs, m = scenes[0]
        cam = views[0][1]
        if case["kind"] == "open":
            y = _decode(_features(case["n"], seed, case["precision"]), synth.random_sh_decoders(seed))
            stored = attrs.clone()
            stored[:, 11:23] = y.to(attrs.dtype)
            full = attrs.double()
            full[:, 11:23] = y
            return [full, _image(stored, m, cam, case["residual"])[0]]
        out = _image(attrs, m, cam, case["residual"], case["kind"] == "depth")
        return out if case["kind"] == "depth" else out[0]


# ---- what a pass cannot do without --------------------------------------------------

def _included(n, scene, width, height):
    """Included (pixel, Gaussian) pairs of a view, from the footprint areas of a
    sample of the scene's distribution."""
    v = _attrs(16384, 1, "fp32", scene, torch.device("cpu")).double()
    v = v[torch.randperm(len(v), generator=torch.Generator().manual_seed(1))]
    cam = _camera(scene, width, height, 0)
    _, tz, mx, my, a, b, c, det = _project(v, cam, _same)
    rx, ry = 3.0 * torch.sqrt(a), 3.0 * torch.sqrt(c)
    fx = ((mx + rx).clamp(0, width) - (mx - rx).clamp(0, width)) / (2 * rx)
    fy = ((my + ry).clamp(0, height) - (my - ry).clamp(0, height)) / (2 * ry)
    area = torch.where((tz > 0.2) & (det > 0), 9.0 * math.pi * torch.sqrt(det.clamp(min=0)) * fx * fy, 0.0)
    return float(area.nan_to_num(0.0).mean()) * n


def work(case):
    kind = case["kind"]
    e = 2 if case["precision"] == "fp16" else 4
    mlp = {"none": 0, "bf16": 22 * 64 + 64 * 64 + 64 * 5,
           "paper": 22 * 256 + 256 * 128 + 128 * 64 + 64 * 5}[case["mlp"]]
    views = [(case["n"], case["width"], case["height"])]
    if kind == "serve":
        views = [(max(case["n"] >> s, 1), w, h) for s, w, h in BURST]
    nbytes = flops = 0.0
    for n, w, h in views:
        pairs = _included(n, case["scene"], w, h)
        # records in, image out; per included pair 7 operations for the test, 9
        # for alpha and the A, B, T sums, 1 exponential; per Gaussian about 250
        # for the projection and colour
        nbytes += n * 24 * e + w * h * 12
        flops += pairs * 17 + n * (250 + 2 * mlp)
        if kind == "depth":
            nbytes += w * h * 4
            flops += pairs * 2
        if kind == "train":
            # target in, gradients out; about 36 operations per pair of the
            # adjoint, and two products per MLP weight
            nbytes += n * 24 * (e + 4) + w * h * 12
            flops += pairs * 36 + n * (500 + 4 * mlp)
        if kind == "open":
            # features in, decoded coefficients out
            nbytes += n * (6 + 12) * e
            flops += n * 2 * (2 * 6 * 64 + 64 * 12)
    return {"bytes": nbytes, "flops": flops}
