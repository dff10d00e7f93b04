"""A Gaussian whose projection is not a number (a zero quaternion pads a cell with
fewer than K Gaussians; a parameter of a diverging step is NaN) is not drawn: images and the
other Gaussians' gradients are those of the same scene with it out of view, in
every blend kernel."""
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
