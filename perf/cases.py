"""The work that users of this renderer have it do, as measurable cases.

A case is a dict of plain values.  ``op`` says which public path it takes:

    view      one forward render of a batch of views (``Context.render``)
    train     parameter update, forward, backward (``Context`` or ``autograd.render``)
    compare   the per-Gaussian comparator renderers (``Context.render_compare``)
    serve     a burst of requests through the serving loop (``submit`` / ``poll``)

``scene`` names the input distribution (those of ``synth.py``, drawn on the
GPU): ``box`` cells in [-1,1]^3, ``multi`` three decades of cell sizes in
[-10,10]^3, ``street`` a ground plane seen from street level, ``neural`` cells
whose Gaussians small MLPs decode per view, on the ``multi`` layout.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2508_03180_gb300 import autograd, synth
from paper_2508_03180_gb300.renderer import Context

DEV = "cuda"
Y00 = 0.28209479177387814
EPS, ALPHA_MAX, D_MIN, DILATION, KSIGMA = 1e-4, 0.99, 1e-10, 0.3, 3.0
TILE = 16


def _case(name, op, scene, cells, K, views, w, h, sh=3, vsh=-1, F=0, H=0, how=""):
    c = dict(op=op, scene=scene, cells=cells, K=K, sh=sh, vsh=vsh, F=F, H=H, views=views, w=w, h=h, how=how)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: the plain scene of the paper's setting, one 256 x 256 view (launch latency)
        _case("view_256", "view", "box", 2048, 8, 1, 256, 256, sh=0),
        # interactive viewing of a 1M-Gaussian scene at 1080p, one frame
        _case("view_1080p", "view", "multi", 100_000, 10, 1, 1920, 1080),
        # one 4K frame of a 10M-Gaussian street scene, most of it out of view
        _case("view_4k_street", "view", "street", 1_000_000, 10, 1, 3840, 2160),
        # ragged sizes: K the kernels have no fixed version of, SH 2, view-dependent v_n, odd resolution
        _case("view_odd", "view", "box", 12_345, 7, 3, 1237, 703, sh=2, vsh=2),
        # the smallest training step, through torch autograd
        _case("train_256", "train", "box", 2048, 8, 1, 256, 256, how="autograd"),
        # the differentiable setting: the small scene, a batch of four 1080p views
        _case("train_4x1080p", "train", "box", 2048, 8, 4, 1920, 1080),
        # the headline step: 1M Gaussians, eight 1080p views, L1 loss, fwd + bwd
        _case("train_8x1080p", "train", "multi", 100_000, 10, 8, 1920, 1080, how="l1"),
        # a ragged step that wants every gradient there is (cells and v_n too)
        _case("train_odd", "train", "box", 20_011, 5, 3, 641, 479, sh=1, vsh=1, how="cells"),
        # neural cells: decode, render and gradients to weights, features and offsets
        _case("train_neural", "train", "neural", 100_000, 10, 2, 1920, 1080, sh=0, F=32, H=32),
        # neural cells of widths beyond the common ones, one frame
        _case("view_neural_wide", "view", "neural", 30_000, 12, 1, 1280, 720, sh=0, F=48, H=64),
        # the comparison renderer: a global sort of every Gaussian, then alpha-blending
        _case("compare_alpha", "compare", "multi", 100_000, 10, 1, 1920, 1080, how="alpha"),
        # a burst of requests of mixed resolutions over two resident scenes
        _case("serve_8", "serve", "box", 62_500, 8, 8, 1280, 720, sh=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("view", "view", "view", "train", "train", "train", "compare", "serve"))
    K = rng.choice((4, 5, 8, 8, 10, 10, 12, 17, 32))
    sh = rng.choice((0, 1, 2, 3, 3))
    w = _log_int(rng, 160, 1920)
    h = max(120, min(1080, int(w * rng.uniform(0.5, 0.8))))
    if op == "serve":
        return _case("", op, "box", _log_int(rng, 2_000, 60_000), K, rng.randint(2, 12), w, h, sh=sh)
    if op == "compare":
        return _case("", op, rng.choice(("box", "multi")), _log_int(rng, 2_000, 60_000), min(K, 12), rng.randint(1, 2), w, h,
                     sh=sh, how=rng.choice(("alpha", "alpha", "wsr")))
    scene = rng.choice(("box", "multi", "multi", "neural") + (("street",) if op == "view" else ()))
    views = rng.randint(1, 4 if op == "train" else 8)
    if scene == "neural":
        return _case("", op, scene, _log_int(rng, 2_000, 60_000), min(K, 16), min(views, 2), w, h, sh=0,
                     F=rng.choice((8, 16, 32, 32, 33, 64)), H=rng.choice((16, 32, 32, 48)))
    cells = _log_int(rng, 1_000, 400_000 if scene == "street" else 30_000 if scene == "box" else 80_000)
    vsh = rng.choice((-1, -1, 0, 1, 2, 3))
    how = rng.choice(("", "autograd", "cells") if vsh < 0 else ("", "cells")) if op == "train" else ""
    return _case("", op, scene, cells, K, views, w, h, sh=sh, vsh=vsh, how=how)


# ---------------------------------------------------------------- inputs


def _rotate(q, v):
    w, r = q[:, :1], q[:, 1:]
    c = torch.linalg.cross(r, v)
    return v + 2.0 * w * c + 2.0 * torch.linalg.cross(r, c)


def _arrays(case, seed):
    """The scene's parameters, float32 CUDA tensors in the layout of the API."""
    g = torch.Generator(device=DEV).manual_seed(1_000_003 * seed + 17)
    N, K, kind = case["cells"], case["K"], case["scene"]
    G = N * K
    uni = lambda *s: torch.rand(*s, device=DEV, generator=g)
    nrm = lambda *s: torch.randn(*s, device=DEV, generator=g)
    unit = lambda x: x / x.norm(dim=1, keepdim=True)
    lo, hi, box = {"box": (0.02, 0.1, 1.0), "multi": (0.001, 1.0, 10.0), "neural": (0.001, 1.0, 10.0),
                   "street": (0.01, 2.0, 200.0)}[kind]
    center = (uni(N, 3) * 2 - 1) * box
    if kind == "street":
        center[:, 2] = (nrm(N) * 5.0).abs()
    axes = torch.exp(math.log(lo) + uni(N, 3) * math.log(hi / lo))
    out = dict(cell_center=center, cell_axes=axes, cell_quat=unit(nrm(N, 4)), cell_v=torch.ones(N, device=DEV))
    ball = unit(nrm(G, 3)) * uni(G, 1) ** (1.0 / 3.0)
    if case["vsh"] >= 0:
        nco = (case["vsh"] + 1) ** 2
        out["cell_v_sh"] = torch.cat([torch.full((N, 1), 0.8 / Y00, device=DEV), 0.15 * nrm(N, nco - 1)], 1).contiguous()
    if kind == "neural":
        F, H = case["F"], case["H"]
        mlp = []
        for n_out, bias in ((K, 1.0), (3 * K, 0.0), (3 * K, -0.85), (4 * K, None)):
            b2 = torch.tensor([1.0, 0.0, 0.0, 0.0], device=DEV).repeat(K) if bias is None else torch.full((n_out,), bias, device=DEV)
            mlp += [(nrm(H, F + 4) / math.sqrt(F + 4)).ravel(), torch.zeros(H, device=DEV), (nrm(n_out, H) / math.sqrt(H)).ravel(), b2]
        return dict(out, feat=nrm(N, F), offset=ball, mlp=torch.cat(mlp))
    axk = axes.repeat_interleave(K, 0)
    mean = center.repeat_interleave(K, 0) + _rotate(out["cell_quat"].repeat_interleave(K, 0), ball * axk)
    nco = (case["sh"] + 1) ** 2
    sh = nrm(G, nco, 3) * 0.2
    sh[:, 0] = (uni(G, 3) - 0.5) / Y00
    return dict(out, g_mean=mean, g_scale=torch.exp(torch.log(0.3 * axk) + 0.3 * nrm(G, 3)), g_quat=unit(nrm(G, 4)),
                g_logit=nrm(G), g_sh=sh)


def _cameras(case, seed):
    n, w, h = case["views"], case["w"], case["h"]
    if case["op"] == "serve":  # mixed resolutions around the case's own
        sizes = [(w, h), (w // 2, h // 2), (w * 3 // 4, h * 3 // 4), (w * 3 // 2, h * 3 // 2)]
        return [synth.sphere_cameras(1, 3.0, *sizes[i % 4], seed0=1000 * seed + i)[0] for i in range(n)]
    if case["scene"] == "street":
        return synth.street_cameras(n, w, h, seed0=1000 * seed)
    return synth.sphere_cameras(n, 3.0 if case["scene"] == "box" else 15.0, w, h, seed0=1000 * seed)


def _upload(ctx, case, a):
    meta = dict(N=case["cells"], K=case["K"], sh_degree=case["sh"], v_sh_degree=case["vsh"])
    if case["scene"] != "neural":
        return ctx.upload_scene(dict(a, **meta))
    n = {k: v.cpu().numpy() for k, v in a.items()}
    zero = np.zeros((case["cells"] * case["K"], 4), np.float32)
    return ctx.upload_scene(synth.Scene(
        K=case["K"], sh_degree=0, cell_center=n["cell_center"], cell_axes=n["cell_axes"], cell_quat=n["cell_quat"],
        cell_v=n["cell_v"], g_mean=zero[:, :3], g_scale=zero[:, :3], g_quat=zero, g_logit=zero[:, 0], g_sh=zero[:, None, :3],
        neural=dict(F=case["F"], H=case["H"], feat=n["feat"], offset=n["offset"], mlp=n["mlp"])))


def _grad_shapes(case):
    N, K = case["cells"], case["K"]
    G = N * K
    if case["scene"] == "neural":
        P = sum(case["H"] * (case["F"] + 5) + o * case["H"] + o for o in (K, 3 * K, 3 * K, 4 * K))
        s = dict(g_mlp=(P,), g_feat=(N, case["F"]), g_offset=(G, 3))
    else:
        s = dict(g_mean=(G, 3), g_log_scale=(G, 3), g_quat=(G, 4), g_logit=(G,), g_sh=(G, (case["sh"] + 1) ** 2, 3))
    if case["how"] == "cells":
        s["g_cell_v"] = (N,)
        if case["vsh"] >= 0:
            s["g_cell_v_sh"], s["g_cell_center"] = (N, (case["vsh"] + 1) ** 2), (N, 3)
    return s


PARAMS = ("g_mean", "g_scale", "g_quat", "g_logit", "g_sh")


class _State:
    """A renderer context with its resident scenes, cameras and the caller's own buffers."""

    def __init__(self, case, seed):
        self.case, self.cams = case, _cameras(case, seed)
        self.ctx = Context()
        a = _arrays(case, seed)
        self.sids = [_upload(self.ctx, case, a)]
        n = sum(3 * h * w for h, w in Context.image_sizes(self.cams))
        g = torch.Generator(device=DEV).manual_seed(seed)
        if case["op"] == "train":
            if case["scene"] != "neural":
                self.params = {k: a[k] for k in PARAMS}
            if case["how"] == "autograd":
                for k in PARAMS:
                    self.params[k].requires_grad_(True)
            else:
                self.grads = {k: torch.empty(s, device=DEV) for k, s in _grad_shapes(case).items()}
            # the images to match, or the gradient that the caller's own loss gives for each pixel
            if case["how"] == "l1":
                self.target = torch.rand(n, device=DEV, generator=g)
                self.dL, self.loss = torch.empty(n, device=DEV), torch.empty(1, device=DEV)
            else:
                self.dL = torch.randn(n, device=DEV, generator=g) / n
        if case["op"] == "serve":
            small = dict(case, cells=max(1, case["cells"] // 5))
            self.sids.append(_upload(self.ctx, small, _arrays(small, seed + 1)))
            self.outs = [torch.empty(3, h, w, device=DEV) for h, w in Context.image_sizes(self.cams)]
            torch.cuda.synchronize()
            self.ctx.serve_start(max_batch=8)

    def __del__(self):
        ctx = getattr(self, "ctx", None)
        if ctx is not None:
            ctx.close()


def prepare(case, seed):
    return _State(case, seed)


def run(s):
    c, ctx, sid = s.case, s.ctx, s.sids[0]
    if c["op"] == "view":
        return ctx.render(sid, s.cams)[0]
    if c["op"] == "compare":
        return ctx.render_compare(sid, s.cams, mode=c["how"])[0]
    if c["op"] == "serve":
        tickets = [ctx.submit(s.sids[i % 2], cam, out) for i, (cam, out) in enumerate(zip(s.cams, s.outs))]
        for t in tickets:
            r = ctx.poll(t)
            if r.status != 0:
                raise RuntimeError("request failed: %d" % r.status)
        return list(s.outs)
    if c["how"] == "autograd":
        p = [s.params[k] for k in PARAMS]
        for t in p:
            t.grad = None
        img = autograd.render(ctx, sid, c["cells"], c["K"], c["sh"], s.cams, *p)
        img.backward(s.dL)
        return dict(image=img.detach(), **{k: t.grad for k, t in zip(PARAMS, p)})
    if c["scene"] != "neural":  # the optimiser's new values
        ctx.update_scene(sid, c["cells"], c["K"], c["sh"], **s.params)
    img, fwd, _ = ctx.render(sid, s.cams, want_state=True)
    if c["how"] == "l1":
        ctx.loss_l1(img, s.target, s.dL, s.loss)
    ctx.backward(fwd, s.dL, s.grads)
    ctx.release_state(fwd)
    out = dict(image=img, **s.grads)
    return dict(out, loss=s.loss) if c["how"] == "l1" else out


# ---------------------------------------------------------------- what a pass cannot do without


def work(case):
    """Parameters read once, images and gradients written once; per pixel, the
    (pixel, Gaussian) pairs inside the Gaussians' boxes (typical of the scene;
    dgs_counts measures them) at 23 FLOP forward and 60 more in the adjoint."""
    N, K, op = case["cells"], case["K"], case["op"]
    G = N * K
    px = sum(c.W * c.H for c in _cameras(case, 0))
    if case["scene"] == "neural":
        F, H = case["F"], case["H"]
        par = 4.0 * (N * (11 + F) + 3 * G + 4 * H * (F + 5) + 11 * K * (H + 1))
        dec = 2.0 * (4 * H * (F + 4) + 11 * K * H) * N * case["views"]
    else:
        par, dec = 4.0 * (11 * N + G * (11 + 3 * (case["sh"] + 1) ** 2) + N * max(0, case["vsh"] + 1) ** 2), 0.0
    if op == "serve":
        par *= 1.2
    pairs = {"box": min(130.0, 5e-4 * G), "multi": min(125.0, 4.5e-4 * G), "neural": min(65.0, 7e-5 * G), "street": 6.2e-6 * G}[case["scene"]] * px
    if op == "compare" and case["how"] == "wsr":
        pairs *= 3
    b, f = par + 12.0 * px, 23.0 * pairs + dec
    if op == "train":
        b += 12.0 * px + 4.0 * sum(math.prod(s) for s in _grad_shapes(case).values())
        f += 60.0 * pairs + 2 * dec
    return {"bytes": b, "flops": f}


def tolerance(case):
    """About four times the distance between the renderer and exact() (2-norm:
    images 1e-6 .. 1e-5, gradients up to 1.1e-4; at single values 7e-4 and 2e-3).
    Images also leave room for a box test decided the other way at one pixel
    (an alpha of at most 0.011).  L1 gradients change sign where image and target agree
    to the last bits (a few pixels in 1e7: 2 sqrt(6e-7) of the norm).  Neural
    cells make decisions on computed values (ReLU masks, sigma <= 0 is not
    drawn): 9e-4 seen on images, 6e-4 on gradients, whole pixels at one place."""
    if case["how"] == "l1":
        return {"rel": 1e-2, "max": 0.5}
    if case["scene"] == "neural":
        return {"rel": 4e-3, "max": 0.95}
    return {"rel": 4e-4, "max": 5e-2} if case["op"] == "train" else {"rel": 4e-5, "max": 2e-2}


# ---------------------------------------------------------------- 64-bit results
# The same operation in plain torch: values in float64, and the decisions that
# the renderer makes in float32 (tile rectangles, depth order, box tests) from
# float32 values formed in the documented order.  Pixels of a tile go through
# the tile's list entry by entry, all tiles at once.


def _camera(cam, dt):
    a = cam.as_array()
    f = a.astype(np.float32 if dt == torch.float32 else np.float64)
    return int(a[0]), int(a[1]), f[2:7], f[7:16].reshape(3, 3), f[16:19], f[19:22]


def _to_view(R, t, p):
    return [((p[:, 0] * float(R[i, 0]) + p[:, 1] * float(R[i, 1])) + p[:, 2] * float(R[i, 2])) + float(t[i]) for i in range(3)]


def _rotation(q):
    w, x, y, z = (q / torch.sqrt(((q[:, 0] * q[:, 0] + q[:, 1] * q[:, 1]) + q[:, 2] * q[:, 2]) + q[:, 3] * q[:, 3])[:, None]).unbind(1)
    return [1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
            2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
            2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]


def _dot3(a, b):
    return (a[0] * b[0] + a[1] * b[1]) + a[2] * b[2]


def _cell_rects(cam, center, axes, quat):
    """float32: (visible, depth, tx0, ty0, tx1, ty1) of every cell."""
    W, H, (fx, fy, cx, cy, zn), R, t, _ = _camera(cam, torch.float32)
    c = _to_view(R, t, center)
    Q = _rotation(quat)
    M = [[_dot3([float(R[a, i]) for i in range(3)], [Q[3 * i + j] for i in range(3)]) * axes[:, j] for j in range(3)] for a in range(3)]
    szz = _dot3(M[2], M[2])
    vis = c[2] - torch.sqrt(szz) > float(zn)
    czz = c[2] * c[2]
    a = czz - szz
    lo, hi = [], []
    for ax, (f, pp) in enumerate(((fx, cx), (fy, cy))):
        suu, suz = _dot3(M[ax], M[ax]), _dot3(M[ax], M[2])
        cuz, cuu = c[ax] * c[2], c[ax] * c[ax]
        disc = ((czz * suu - (2.0 * cuz) * suz) + cuu * szz) - (suu * szz - suz * suz)
        sq = torch.sqrt(disc.clamp_min(0.0))
        b = cuz - suz
        lo.append(float(f) * ((b - sq) / a) + float(pp))
        hi.append(float(f) * ((b + sq) / a) + float(pp))
    return _tiles_of(vis, lo, hi, W, H) + (c[2],)


def _tiles_of(vis, lo, hi, W, H):
    Tx, Ty = (W + TILE - 1) // TILE, (H + TILE - 1) // TILE
    vis = vis & (hi[0] >= 0) & (lo[0] < W) & (hi[1] >= 0) & (lo[1] < H)
    fl = lambda x, n: torch.nan_to_num(x).clamp(0.0, float(n)).div(TILE).floor().long()
    return vis, fl(lo[0], W), fl(lo[1], H), fl(hi[0], W).clamp_max(Tx - 1), fl(hi[1], H).clamp_max(Ty - 1)


def _tile_lists(rects, Tx, Ty, by_depth=True):
    """Entries of every tile in (depth, index) order: (entry list, start, length)."""
    vis, x0, y0, x1, y1, z = rects
    e = torch.nonzero(vis)[:, 0]
    if by_depth:
        e = e[torch.sort(z[e], stable=True).indices]
    w, n = (x1 - x0 + 1)[e], ((x1 - x0 + 1) * (y1 - y0 + 1))[e]
    own = torch.repeat_interleave(torch.arange(e.numel(), device=DEV), n)
    local = torch.arange(own.numel(), device=DEV) - (torch.cumsum(n, 0) - n)[own]
    tile = (y0[e][own] + local // w[own]) * Tx + x0[e][own] + local % w[own]
    tile, at = torch.sort(tile, stable=True)
    length = torch.bincount(tile, minlength=Tx * Ty)
    return e[own[at]], torch.cumsum(length, 0) - length, length


def _screen(cam, mean, scale, quat):
    """Screen mean, covariance (xx, xy, yy) and depth of Gaussians, in their own precision."""
    dt = mean.dtype
    W, H, (fx, fy, cx, cy, zn), R, t, _ = _camera(cam, dt)
    num = np.float32 if dt == torch.float32 else np.float64
    fx, fy, cx, cy = (float(v) for v in (fx, fy, cx, cy))
    c = _to_view(R, t, mean)
    ok = c[2] > float(zn)
    z = torch.where(ok, c[2], torch.ones_like(c[2]))
    x, y = c[0] / z, c[1] / z
    Q = _rotation(quat)
    M = [[Q[3 * i + j] * scale[:, j] for j in range(3)] for i in range(3)]
    S = [[_dot3(M[i], M[j]) for j in range(3)] for i in range(3)]
    lx = float(num(1.3) * (num(0.5) * num(W) / num(fx)))
    ly = float(num(1.3) * (num(0.5) * num(H) / num(fy)))
    J00, J02 = fx / z, -((fx * x.clamp(-lx, lx)) / z)
    J11, J12 = fy / z, -((fy * y.clamp(-ly, ly)) / z)
    T = [[J00 * float(R[0, j]) + J02 * float(R[2, j]) for j in range(3)], [J11 * float(R[1, j]) + J12 * float(R[2, j]) for j in range(3)]]
    V = [[_dot3(T[a], [S[i][j] for i in range(3)]) for j in range(3)] for a in range(2)]
    cov = (_dot3(V[0], T[0]) + DILATION, _dot3(V[0], T[1]), _dot3(V[1], T[1]) + DILATION)
    return ok, x * fx + cx, y * fy + cy, cov, c[2]


def _sh_basis(d, deg):
    x, y, z = d.unbind(1)
    Y = [torch.full_like(x, Y00)]
    if deg >= 1:
        k = math.sqrt(3 / (4 * math.pi))
        Y += [k * y, k * z, k * x]
    if deg >= 2:
        a, b, c = (math.sqrt(v / math.pi) for v in (15 / 4, 5 / 16, 15 / 16))
        Y += [a * x * y, a * y * z, b * (3 * z * z - 1), a * x * z, c * (x * x - y * y)]
    if deg >= 3:
        a, b, c, d0, e = (math.sqrt(v / math.pi) for v in (35 / 32, 105 / 4, 21 / 32, 7 / 16, 105 / 16))
        Y += [a * y * (3 * x * x - y * y), b * x * y * z, c * y * (5 * z * z - 1), d0 * z * (5 * z * z - 3),
              c * x * (5 * z * z - 1), e * z * (x * x - y * y), a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, 1)


def _decode(case, p, eye):
    """The Gaussians of every neural cell for one eye position."""
    N, K, F, H = case["cells"], case["K"], case["F"], case["H"]
    rel = p["cell_center"] - eye
    delta = rel.norm(dim=1, keepdim=True)
    zin = torch.cat([p["feat"], delta, rel / delta], 1)
    o, outs = 0, []
    for n_out in (K, 3 * K, 3 * K, 4 * K):
        parts = []
        for shape in ((H, F + 4), (H,), (n_out, H), (n_out,)):
            n = math.prod(shape)
            parts.append(p["mlp"][o:o + n].reshape(shape))
            o += n
        outs.append(torch.relu(zin @ parts[0].T + parts[1]) @ parts[2].T + parts[3])
    off = p["offset"].reshape(N, K, 3)
    off = off / off.norm(dim=2, keepdim=True).clamp_min(1.0)
    ratio = torch.minimum(torch.sigmoid(outs[2]).reshape(N, K, 3), 1.0 - off.norm(dim=2, keepdim=True))
    S = p["cell_axes"][:, None]
    Rn = torch.stack(_rotation(p["cell_quat"]), 1).reshape(N, 3, 3)
    q = outs[3].reshape(N, K, 4)
    mean = p["cell_center"][:, None] + torch.einsum("nij,nkj->nki", Rn, off * S)
    return (mean.reshape(-1, 3), (ratio * S).reshape(-1, 3), (q / q.norm(dim=2, keepdim=True)).reshape(-1, 4),
            torch.tanh(outs[0]).reshape(-1), torch.sigmoid(outs[1]).reshape(-1, 3))


class _View:
    """One view in 64 bits: image, and with dL the gradients to the leaves."""

    def __init__(self, case, a32, leaves, cam, mode="hybrid"):
        self.mode, self.K = mode, 1 if mode != "hybrid" else case["K"]
        W, H, _, _, _, eye = _camera(cam, torch.float64)
        self.W, self.H, self.Tx, self.Ty = W, H, (W + TILE - 1) // TILE, (H + TILE - 1) // TILE
        eye = torch.tensor(eye, device=DEV)
        if case["scene"] == "neural":
            mean, scale, quat, op, rgb = _decode(case, leaves, eye)
            drawn = op > 0
        else:
            mean, scale, quat = leaves["g_mean"], leaves["g_scale"], leaves["g_quat"]
            op, drawn = torch.sigmoid(leaves["g_logit"]), True
            d = mean - eye
            rgb = (0.5 + torch.einsum("gc,gch->gh", _sh_basis(d / d.norm(dim=1, keepdim=True), case["sh"]), leaves["g_sh"])).clamp_min(0)
        if case["vsh"] >= 0 and mode == "hybrid":
            d = leaves["cell_center"] - eye
            v = (_sh_basis(d / d.norm(dim=1, keepdim=True), case["vsh"]) * leaves["cell_v_sh"]).sum(1).clamp(0, 1)
        else:
            v = leaves["cell_v"] * 1.0
        if mode != "hybrid":
            v = v.repeat_interleave(case["K"])
        ok, mx, my, (sxx, sxy, syy), _ = _screen(cam, mean, scale, quat)
        det = sxx * syy - sxy * sxy
        self.rec = [mx, my, syy / det, -sxy / det, sxx / det, op, rgb, v]
        ok32, x32, y32, (cxx, _, cyy), z32 = _screen(cam, *(t.detach().float() for t in (mean, scale, quat)))
        ex, ey = KSIGMA * torch.sqrt(cxx), KSIGMA * torch.sqrt(cyy)
        hide = ~(ok32 & drawn)
        self.box = [x32, y32, ex.masked_fill(hide, -1.0), ey.masked_fill(hide, -1.0)]
        if mode == "hybrid":
            rects = _cell_rects(cam, a32["cell_center"], a32["cell_axes"], a32["cell_quat"])
        else:
            rects = _tiles_of(ok32, [x32 - ex, y32 - ey], [x32 + ex, y32 + ey], W, H) + (z32,)
        self.list, self.start, self.len = _tile_lists(rects, self.Tx, self.Ty, mode != "wsr")
        i = torch.arange(TILE * TILE, device=DEV)
        self.pi, self.pj = i % TILE, i // TILE
        self.val = [r.detach() for r in self.rec]

    def chunks(self):
        order = torch.argsort(self.len, descending=True, stable=True)
        size = max(1, 24_000_000 // (TILE * TILE * self.K))
        return [order[i:i + size] for i in range(0, order.numel(), size)]

    def pixels(self, tiles):
        return ((tiles % self.Tx) * TILE)[:, None] + self.pi, (torch.div(tiles, self.Tx, rounding_mode="floor") * TILE)[:, None] + self.pj

    def entry(self, tiles, n, px, py):
        """Entry n of the tiles' lists at their pixels: cell ids, Gaussian ids, offsets, G, alpha and 1 - v alpha."""
        e = self.list[self.start[tiles] + n]
        g = e[:, None] * self.K + torch.arange(self.K, device=DEV)
        mx, my, qa, qb, qc, op = (t[g][:, None] for t in self.val[:6])
        bx, by, ex, ey = (t[g][:, None] for t in self.box)
        inside = ((px.float()[..., None] + 0.5 - bx).abs() <= ex) & ((py.float()[..., None] + 0.5 - by).abs() <= ey)
        dx, dy = px[..., None] + 0.5 - mx, py[..., None] + 0.5 - my
        Gv = torch.exp(-0.5 * (qa * dx * dx + 2 * qb * dx * dy + qc * dy * dy)) * inside
        raw = op * Gv
        al = raw.clamp_max(ALPHA_MAX)
        v = self.val[7][e]
        return e, g, (dx, dy, qa, qb, qc, op), Gv, raw, al, v, 1 - v[:, None, None] * al

    def forward(self, keep):
        """The image [3, H, W]; with keep, the transmittance before every entry stays for the adjoint."""
        N = torch.zeros(self.Tx * self.Ty, TILE * TILE, 3, device=DEV, dtype=torch.float64)
        D = torch.zeros_like(N[..., 0])
        self.trace = []
        for tiles in self.chunks():
            px, py = self.pixels(tiles)
            T = torch.ones_like(px, dtype=torch.float64)
            T[(px >= self.W) | (py >= self.H)] = 0.0
            n, steps = 0, []
            while tiles.numel():
                if n % 8 == 0:  # lists that ended and tiles that are opaque leave
                    live = (T >= EPS).any(1) & (self.len[tiles] > n)
                    tiles, T, px, py = tiles[live], T[live], px[live], py[live]
                    if not tiles.numel():
                        break
                some = self.len[tiles] > n
                e, g, _, _, _, al, v, om = self.entry(tiles, torch.where(some, n, 0), px, py)
                act = (T >= EPS) & some[:, None]
                w = v[:, None] * torch.where(act, T, 0.0)
                N.index_add_(0, tiles, w[..., None] * torch.einsum("tpk,tkc->tpc", al, self.val[6][g]))
                D.index_add_(0, tiles, w * al.sum(2))
                if keep:
                    steps.append((n, tiles, T, act))
                if self.mode != "wsr":
                    T = torch.where(act, T * om.prod(2), T)
                n += 1
            self.trace.append(steps)
        self.N, self.D = N, D
        img = N if self.mode == "alpha" else torch.where((D > D_MIN)[..., None], N / D.clamp_min(D_MIN)[..., None], 0.0)
        img = img.reshape(self.Ty, self.Tx, TILE, TILE, 3).permute(4, 0, 2, 1, 3).reshape(3, self.Ty * TILE, self.Tx * TILE)
        return img[:, :self.H, :self.W]

    def backward(self, dL, leaves, wanted):
        """Gradients of sum(dL * image) with respect to the wanted leaves."""
        pad = torch.zeros(3, self.Ty * TILE, self.Tx * TILE, device=DEV, dtype=torch.float64)
        pad[:, :self.H, :self.W] = dL
        gi = pad.reshape(3, self.Ty, TILE, self.Tx, TILE).permute(1, 3, 2, 4, 0).reshape(self.Tx * self.Ty, TILE * TILE, 3)
        hit = self.D > D_MIN
        gN = torch.where(hit[..., None], gi / self.D.clamp_min(D_MIN)[..., None], 0.0)
        gD = -(gN * self.N).sum(2) / self.D.clamp_min(D_MIN)
        out = [torch.zeros_like(t) for t in self.val]
        gT_all = torch.zeros_like(gD)
        for steps in self.trace:
            for n, tiles, T, act in reversed(steps):
                px, py = self.pixels(tiles)
                some = self.len[tiles] > n
                e, g, (dx, dy, qa, qb, qc, op), Gv, raw, al, v, om = self.entry(tiles, torch.where(some, n, 0), px, py)
                Ta = torch.where(act, T, 0.0)
                gt = gT_all[tiles]
                P, col = om.prod(2), self.val[6][g]
                inner = torch.einsum("tpc,tkc->tpk", gN[tiles], col) + gD[tiles][..., None]
                gw = (al * inner).sum(2)
                back = (gt * Ta * P)[..., None] / om  # dL/dP dP/d(v alpha), sign apart
                gal = v[:, None, None] * (Ta[..., None] * inner - back)
                out[7].index_add_(0, e, (Ta * gw).sum(1) - (back * al).sum((1, 2)))
                out[6].index_add_(0, g.reshape(-1), torch.einsum("tp,tpk,tpc->tkc", v[:, None] * Ta, al, gN[tiles]).reshape(-1, 3))
                gal = torch.where(raw < ALPHA_MAX, gal, 0.0) * Gv
                gq = -0.5 * gal * op
                for k, t in ((0, -gq * 2 * (qa * dx + qb * dy)), (1, -gq * 2 * (qb * dx + qc * dy)), (2, gq * dx * dx),
                             (3, gq * 2 * dx * dy), (4, gq * dy * dy), (5, gal)):
                    out[k].index_add_(0, g.reshape(-1), t.sum(1).reshape(-1))
                gT_all[tiles] = torch.where(act, v[:, None] * gw + gt * P, gt)
        pairs = [(r, o) for r, o in zip(self.rec, out) if r.requires_grad]
        return torch.autograd.grad([r for r, _ in pairs], [leaves[k] for k in wanted], [o for _, o in pairs], allow_unused=True)


LEAF = dict(g_mean="g_mean", g_scale="g_scale", g_log_scale="g_scale", g_quat="g_quat", g_logit="g_logit", g_sh="g_sh",
            g_cell_v="cell_v", g_cell_v_sh="cell_v_sh", g_cell_center="cell_center", g_mlp="mlp", g_feat="feat", g_offset="offset")


def exact(case, seed):
    if case["how"] == "l1" or case["views"] * case["w"] * case["h"] > 9_000_000 or case["cells"] * case["K"] > 12_000_000:
        return None
    cams = _cameras(case, seed)
    if case["op"] == "serve":
        small = dict(case, cells=max(1, case["cells"] // 5))
        sets = [(case, _arrays(case, seed)), (small, _arrays(small, seed + 1))]
        sets = [(c, a, {k: v.double() for k, v in a.items()}) for c, a in sets]
        return [_View(*sets[i % 2], cam).forward(False).contiguous() for i, cam in enumerate(cams)]
    a = _arrays(case, seed)
    train = case["op"] == "train"
    leaves = {k: v.double().requires_grad_(train) for k, v in a.items()}
    if not train:
        mode = case["how"] if case["op"] == "compare" else "hybrid"
        return torch.cat([_View(case, a, leaves, cam, mode).forward(False).reshape(-1) for cam in cams])
    # the state's own draw of dL
    n = sum(3 * c.W * c.H for c in cams)
    dL = (torch.randn(n, device=DEV, generator=torch.Generator(device=DEV).manual_seed(seed)) / n).double()
    names = list(PARAMS) if case["how"] == "autograd" else list(_grad_shapes(case))
    wanted = [LEAF[k] for k in names]
    total, images, at = [0.0] * len(names), [], 0
    vd = [i for i, k in enumerate(names) if k == "g_cell_v"]
    for cam in cams:
        view = _View(case, a, leaves, cam)
        images.append(view.forward(True).reshape(-1))
        m = images[-1].numel()
        v = view.rec[7]
        got = list(view.backward(dL[at:at + m].reshape(3, cam.H, cam.W), dict(leaves, cell_v=v) if vd else leaves, wanted))
        total = [t + (0.0 if x is None else x) for t, x in zip(total, got)]
        at += m
    out = dict(image=torch.cat(images))
    for k, t, shape in zip(names, total, (leaves[w].shape for w in wanted)):
        t = torch.zeros(shape, device=DEV, dtype=torch.float64) if isinstance(t, float) else t
        out[k] = t * leaves["g_scale"].detach() if k == "g_log_scale" else t
    return out
