"""Gaussians with undefined or infinite values stay within their own pixels.

* A Gaussian whose projection is not a number (a zero quaternion pads a cell with
  fewer than K Gaussians; a parameter of a diverging step is NaN) is not drawn: images and the
  other Gaussians' gradients are those of the same scene with it out of view,
  in every blend kernel.
* A colour, or a weighted sum's weight, beyond FP32 leaves the pixels alone that it does
  not reach: those outside the Gaussian's box and those finished before its cell.
"""
import copy

import numpy as np
import pytest
import torch

from paper_2508_03180_gb300 import synth
from paper_2508_03180_gb300.renderer import Context

pytestmark = pytest.mark.gpu

# beyond 2304 tiles with the second view, which sees nothing: 16x8 sub-tiles instead of 16x4
CAM = synth.small_camera(61, 43)
EMPTY = synth.look_at((0.0, -3.0, 0.0), (0.0, -6.0, 0.0), 784, 768, 60.0)


def _zero_quat(sc, g):
    sc.g_quat[g] = 0.0


def _nan_quat(sc, g):
    sc.g_quat[g, 1] = np.nan


def _nan_scale(sc, g):
    sc.g_scale[g, 2] = np.nan


def _huge_scale(sc, g):
    sc.g_scale[g] = 1e30  # a screen covariance beyond FP32


def _images(ctx, sc, cams):
    sid = ctx.upload_scene(sc)
    out = [ctx.render(sid, cams)[0].clone()]
    out += [ctx.render_compare(sid, cams, m)[0].clone() for m in ("alpha", "wsr")]
    flat, state, _ = ctx.render(sid, cams, want_state=True)
    dl = torch.randn(flat.numel(), generator=torch.Generator().manual_seed(2)).cuda()
    gr = dict(g_mean=torch.zeros(sc.G, 3, device="cuda"), g_scale=torch.zeros(sc.G, 3, device="cuda"),
              g_quat=torch.zeros(sc.G, 4, device="cuda"), g_logit=torch.zeros(sc.G, device="cuda"),
              g_sh=torch.zeros(sc.G, 1, 3, device="cuda"), g_cell_v=torch.zeros(sc.N, device="cuda"))
    ctx.backward(state, dl, gr)
    torch.cuda.synchronize()
    ctx.release_state(state)
    ctx.release_scene(sid)
    return out, gr


@pytest.mark.parametrize("damage", [_zero_quat, _nan_quat, _nan_scale, _huge_scale])
@pytest.mark.parametrize("opaque,flags,large", [(False, 0, False), (True, 0, False), (False, 0, True), (False, 2, False)])
def test_undefined_gaussian_is_not_drawn(damage, opaque, flags, large):
    sc = synth.make_scene(24, 4, synth._box(-0.5, 0.5), 0.1, 0.4, 0, seed=31)
    if opaque:
        sc.g_logit[::2] = 7.0  # beyond the alpha clamp: those batches take the minimum
    bad = np.arange(3, sc.G, 8)
    ref = copy.deepcopy(sc)
    ref.g_mean[bad, 1] = -3.0  # beside both cameras: not in front of their near planes
    damage(sc, bad)
    cams = [CAM, EMPTY] if large else [CAM]
    ctx = Context(flags=flags)
    try:
        got, g_got = _images(ctx, sc, cams)
        want, g_want = _images(ctx, ref, cams)
        for a, b in zip(got, want):
            assert torch.equal(a, b)
        assert (want[0].reshape(-1)[:CAM.W * CAM.H] > 0).float().mean() > 0.1
        live = np.setdiff1d(np.arange(sc.G), bad)
        for k in g_want:
            a, b = (g_got[k], g_want[k]) if k == "g_cell_v" else (g_got[k][live], g_want[k][live])
            # the same sums, added to by atomics in another order
            assert (a - b).norm() <= 1e-5 * b.norm(), k
    finally:
        ctx.close()


@pytest.mark.parametrize("cfg", [dict(), dict(dilation=0.0), dict(flags=2)])
def test_undefined_opacity_is_not_drawn(cfg):
    """(By the hybrid renderer; the comparators take alpha_max within the box.)"""
    sc = synth.make_scene(24, 4, synth._box(-0.5, 0.5), 0.1, 0.4, 0, seed=37)
    bad = np.arange(3, sc.G, 8)
    ref = copy.deepcopy(sc)
    ref.g_mean[bad, 1] = -3.0  # not in front of the near plane
    sc.g_logit[bad] = np.nan
    ctx = Context(**cfg)
    try:
        (got, alpha, wsr), g_got = _images(ctx, sc, [CAM])
        (want, _, _), g_want = _images(ctx, ref, [CAM])
        assert torch.equal(got, want) and want.any()
        assert torch.isfinite(alpha).all() and torch.isfinite(wsr).all()
        live = np.setdiff1d(np.arange(sc.G), bad)
        for k in g_want:
            a, b = (g_got[k], g_want[k]) if k == "g_cell_v" else (g_got[k][live], g_want[k][live])
            assert (a - b).norm() <= 1e-5 * b.norm(), k
    finally:
        ctx.close()


def test_flat_gaussian_without_dilation():
    """A needle seen obliquely: its screen covariance is singular, L infinite and its exponent
    infinite or inf - inf.  The forward draws nothing of it, and the adjoint's replay agrees."""
    sc = synth.make_scene(24, 2, synth._box(-0.5, 0.5), 0.1, 0.4, 0, seed=33)
    needle = np.arange(1, sc.G, 6)
    sc.g_scale[needle] = [[0.5, 0.0, 0.0]]
    sc.g_quat[needle] = [[1.0, 0.0, 0.0, 0.0]]
    ref = copy.deepcopy(sc)
    ref.g_mean[needle, 1] = -3.0  # not in front of the near plane
    cams = [synth.look_at((0.0, -3.0, 0.0), (0.0, 0.0, 0.0), 61, 43, 60.0, up=(0.6, 0.0, 1.0))]
    ctx = Context(dilation=0.0)
    try:
        (got, _, _), g_got = _images(ctx, sc, cams)
        (want, _, _), g_want = _images(ctx, ref, cams)
        assert torch.equal(got, want) and (want > 0).float().mean() > 0.1
        live = np.setdiff1d(np.arange(sc.G), needle)
        for k in g_want:
            a, b = (g_got[k], g_want[k]) if k == "g_cell_v" else (g_got[k][live], g_want[k][live])
            assert (a - b).norm() <= 1e-5 * b.norm(), k
    finally:
        ctx.close()


def _flat_scene(n, logit, scale):
    """n cells of one Gaussian each, one behind the other as seen from (0, -3, 0)."""
    sc = synth.make_scene(n, 1, synth._box(-0.2, 0.2), 0.9, 1.0, 0, seed=5)
    sc.cell_center[:] = [[0.0, 0.05 * i, 0.0] for i in range(n)]
    sc.g_mean[:] = sc.cell_center
    sc.g_scale[:] = scale
    sc.g_logit[:] = logit
    return sc


@pytest.mark.parametrize("large", [False, True])
def test_infinite_colour_behind_finished_pixels(large):
    """Twelve opaque layers finish the pixels in the middle of the view; behind them, over all
    of it, a Gaussian of infinite colour."""
    sc = _flat_scene(13, 9.0, 1.0)
    sc.g_scale[12] = 3.0
    cams = [synth.small_camera(32, 16)] + ([EMPTY] if large else [])
    ref = copy.deepcopy(sc)
    sc.g_sh[12] = np.inf
    ctx = Context()
    try:
        outs = []
        for s in (ref, sc):
            sid = ctx.upload_scene(s)
            img, state, _ = ctx.render(sid, cams, want_state=True)
            a = img[:3 * 16 * 32].reshape(3, 16, 32).clone()
            ctx.release_state(state)
            c = ctx.render_compare(sid, cams, "alpha")[0][:3 * 16 * 32].reshape(3, 16, 32).clone()
            ctx.release_scene(sid)
            outs.append((a, c))
        for want, got in zip(*outs):
            same = (got == want).all(0)
            # finished pixels keep their colour, the others take the huge one
            assert 0.1 < same.float().mean() < 0.9
            assert (got[:, ~same] > 1e15).any(0).all()
            assert not torch.isnan(got).any()
    finally:
        ctx.close()


@pytest.mark.parametrize("mode", ["hybrid", "alpha", "wsr", "weight"])
def test_infinite_values_stay_within_the_box(mode):
    """Two Gaussians, the nearer one over the middle of a one-tile view only."""
    sc = _flat_scene(2, 0.0, 0.3)
    sc.g_scale[1] = 2.0
    cam = synth.small_camera(16, 16)
    ref, none = copy.deepcopy(sc), copy.deepcopy(sc)
    none.g_mean[0, 1] -= 10.0
    if mode == "weight":
        sc.cell_v[0] = np.inf
    else:
        sc.g_sh[0] = np.inf
    ctx = Context()
    try:
        imgs = []
        for s in (none, ref, sc):
            sid = ctx.upload_scene(s)
            img = ctx.render(sid, [cam])[0] if mode == "hybrid" else ctx.render_compare(
                sid, [cam], "alpha" if mode == "alpha" else "wsr")[0]
            imgs.append(img.reshape(3, 16, 16).clone())
            ctx.release_scene(sid)
        out = (imgs[0] == imgs[1]).all(0)  # the pixels that the nearer one does not reach
        assert 0.2 < out.float().mean() < 0.9
        assert torch.equal(imgs[2][:, out], imgs[0][:, out])
    finally:
        ctx.close()
