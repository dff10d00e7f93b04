"""Parity of the sm_103a path (through the C ABI) against the CPU oracle.

* binning (cell rectangles, depths, per-tile ordered cell lists, ranges): bit-exact
* per-Gaussian AABB inputs (mu2, half extents): bit-exact; conic, opacity,
  colour: within FP32 rounding of the FP64 projection
* images: 1e-4 max abs per channel against the FP64 oracle, which renders
  with the GPU's per-pixel processed-cell counts after checking that each is
  a valid outcome of the stopping rule (relative slack 1e-3 on T); the
  oracle's own counts may differ on at most 0.01% of pixels
"""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from paper_2508_03180_gb300 import synth
from tests.gpu_helpers import LOG2E, gpu_render, read_state, tile_lists_equal, view_slices

pytestmark = pytest.mark.gpu

IMG_TOL = 1e-4


@pytest.fixture(scope="module")
def rctx():
    from paper_2508_03180_gb300.renderer import Context
    c = Context()
    yield c
    c.close()


def check_view(scene, cam_obj, gv, cells_all, img, check_image=True, tile_rows=None):
    cam = cam_obj.as_array()
    rect, depth = oracle.cell_rects(scene, cam)
    assert np.array_equal(gv["rect"], rect), "cell rectangles differ"
    vis = rect[:, 0] >= 0
    assert np.array_equal(gv["depth"][vis].view(np.uint32), depth[vis].view(np.uint32)), "cell depths differ"
    ocells, orng = oracle.tile_lists(rect, depth, cam)
    assert tile_lists_equal(gv, cells_all, ocells, orng) == 0, "tile lists differ"
    # AABB inputs: bit-exact for Gaussians of visible cells
    mu2f, extf, valid = oracle.gauss_decisions(scene, cam)
    gvis = np.repeat(vis, scene.K)
    rec = gv["rec"]
    ok = gvis & (valid != 0)
    assert np.array_equal(rec[ok, 0:2].view(np.uint32), mu2f[ok].view(np.uint32)), "projected means differ"
    assert np.array_equal(rec[ok, 2:4].view(np.uint32), extf[ok].view(np.uint32)), "AABB extents differ"
    assert np.all(rec[gvis & (valid == 0), 2] < 0), "invalid Gaussians must never pass the AABB test"
    if not check_image:
        return None
    pv = oracle.prepare_view(scene, cam, tile_rows=tile_rows)
    pr = pv["proj"]
    # conic / opacity / colour of the records vs FP64
    # the record holds the conic's Cholesky factor L = [[p, 0], [r, t]] scaled by
    # kappa = sqrt(log2(e)/2): a = p^2, b = p r, c = r^2 + t^2 (divided by kappa^2)
    k2 = 0.5 * LOG2E
    pp, rr, tt = (rec[:, 4].astype(np.float64), rec[:, 5].astype(np.float64), rec[:, 6].astype(np.float64))
    conic = np.stack([pp * pp / k2, pp * rr / k2, (rr * rr + tt * tt) / k2], 1)
    m = pv["mask"]
    # each entry within 1e-4 of the conic's own scale
    scale = np.maximum(np.abs(pr["conic"][m][:, 0]), np.abs(pr["conic"][m][:, 2]))[:, None]
    assert np.all(np.abs(conic[m] - pr["conic"][m]) <= 1e-4 * scale), "conic differs"
    np.testing.assert_allclose(rec[m, 7], pr["opac"][m], rtol=1e-5, atol=1e-7)
    np.testing.assert_allclose(rec[m, 8:11], pr["rgb"][m], rtol=1e-4, atol=2e-5)
    r = oracle.render_view(scene, cam, forced_ndone=gv["nd"], pv=pv)
    H, W = gv["H"], gv["W"]
    ty0, ty1 = pv["rows"]
    y0, y1 = ty0 * 16, min(ty1 * 16, H)
    window = slice(y0, y1)
    n_px = (y1 - y0) * W
    assert r["bad"] <= 0, f"{r['bad']} GPU termination counts are not valid outcomes"
    diff_own = int((r["ndone"][window] != gv["nd"][window]).sum())
    assert diff_own <= max(1, int(1e-4 * n_px)), f"{diff_own} pixels stop at a different cell"
    err = np.abs(img.reshape(3, H, W)[:, window] - r["C"][:, window]).max()
    assert err <= IMG_TOL, f"image max abs error {err}"
    np.testing.assert_allclose(gv["D"][window], r["D"][window], rtol=1e-4, atol=1e-7)
    return dict(err=float(err), diff_own=diff_own, hit=float((r["D"][window] > 1e-10).mean()))


def _render_and_check(rctx, scene, cams, tile_rows=None):
    sid = rctx.upload_scene(scene)
    state = None
    try:
        flat, state, st = gpu_render(rctx, sid, cams)
        gs = read_state(rctx, state, scene, cams)
        imgs = rctx.split(flat, cams)
        res = []
        for v, cam in enumerate(cams):
            gv = view_slices(gs, v)
            res.append(check_view(scene, cam, gv, gs["cells"], imgs[v].cpu().numpy(), tile_rows=tile_rows))
        # sort length reported = sum over views of the oracle's
        assert st.sort_length == sum(oracle.sort_length(scene, c.as_array()) for c in cams)
        return res
    finally:
        if state is not None:
            rctx.release_state(state)
        rctx.release_scene(sid)


def test_small_scene_256(rctx):
    """2,048 cells x 8 Gaussians, 256x256, one view."""
    res = _render_and_check(rctx, synth.scene_small(), [synth.small_camera()])
    assert res[0]["hit"] > 0.5


def test_small_scene_sh3_batch_of_views(rctx):
    sc = synth.scene_small(sh_degree=3)
    cams = synth.sphere_cameras(4, 3.0, 200, 136, seed0=10)
    _render_and_check(rctx, sc, cams)


def test_mixed_resolutions_one_chain(rctx):
    sc = synth.make_scene(500, 5, synth._box(-1, 1), 0.03, 0.3, 2, seed=3)
    base = synth.sphere_cameras(3, 3.5, 64, 64, seed0=20)
    cams = [base[0].with_resolution(97, 45), base[1].with_resolution(16, 16), base[2].with_resolution(130, 211)]
    _render_and_check(rctx, sc, cams)


@pytest.mark.parametrize("K", [1, 3, 10, 32])
def test_gaussians_per_cell(rctx, K):
    sc = synth.make_scene(max(8, 600 // K), K, synth._box(-1, 1), 0.05, 0.3, 1, seed=K)
    _render_and_check(rctx, sc, [synth.small_camera(80, 72)])


@pytest.mark.parametrize("K", [2, 5, 8, 11, 16, 17, 31])
def test_cell_batches(rctx, K):
    """The forward blends 32 // K cells per batch: list lengths around the
    batch's, lanes without a Gaussian (K not dividing 32), lists that end or
    whose pixels finish within a batch (opaque cells)."""
    sc = synth.make_scene(max(8, 900 // K), K, synth._box(-1, 1), 0.05, 0.4, 1, seed=40 + K)
    sc.g_logit[:] += 2.0
    _render_and_check(rctx, sc, [synth.small_camera(75, 50), synth.small_camera(64, 48)])


@pytest.mark.parametrize("W", [768, 737])
def test_sub_tile_sizes_give_the_same_image(rctx, W):
    """2304 tiles and fewer (a cut last column), against 2352 (the larger sub-tiles): the common
    pixels of both images are equal bit for bit."""
    sc = synth.scene_small(n_cells=500)
    sid = rctx.upload_scene(sc)
    wide = synth.small_camera(784, 768)
    a = rctx.render(sid, [wide])[0].view(3, 768, 784)[:, :, :W].clone()
    b = rctx.render(sid, [dataclasses.replace(wide, W=W)])[0].view(3, 768, W)
    assert torch.equal(a, b)
    rctx.release_scene(sid)


def test_no_dilation_and_a_gaussian_of_no_extent():
    """Without dilation a Gaussian of no extent has an infinite conic: it is
    drawn nowhere but at its centre, and its neighbours as if it were absent."""
    cam = synth.small_camera(64, 48)
    from paper_2508_03180_gb300.renderer import Context
    images = []
    for hidden in (False, True):
        sc = synth.make_scene(40, 4, synth._box(-0.5, 0.5), 0.2, 0.4, 0, seed=9)
        sc.g_scale[::7] = 0.0
        if hidden:
            sc.g_logit[::7] = -100.0
            sc.g_scale[::7] = 0.05
        ctx = Context(dilation=0.0)
        images.append(ctx.render(ctx.upload_scene(sc), [cam])[0].cpu().numpy())
        ctx.close()
    assert np.isfinite(images[0]).all()
    assert np.abs(images[0] - images[1]).max() <= 1e-6


def test_multiscale_subset_480x270(rctx):
    sc = synth.scene_multiscale(n_cells=20_000, K=10)
    _render_and_check(rctx, sc, synth.sphere_cameras(2, 15.0, 480, 270))


def test_ragged_and_tiny_images(rctx):
    sc = synth.scene_small(n_cells=300)
    cams = [synth.small_camera(1, 1), synth.small_camera(17, 33), synth.small_camera(31, 15)]
    _render_and_check(rctx, sc, cams)


def test_empty_scene_renders_background(rctx):
    sc = synth.scene_small(n_cells=0)
    sid = rctx.upload_scene(sc)
    flat, _, st = rctx.render(sid, [synth.small_camera(40, 24)], stats=True)
    torch.cuda.synchronize()
    assert st.sort_length == 0 and torch.all(flat == 0)
    rctx.release_scene(sid)


def test_all_cells_culled(rctx):
    sc = synth.scene_small(n_cells=500)
    cam = synth.look_at((0, -3, 0), (0, -6, 0), 64, 64)  # looking away from the scene
    sid = rctx.upload_scene(sc)
    flat, _, st = rctx.render(sid, [cam], stats=True)
    torch.cuda.synchronize()
    assert st.sort_length == 0 and st.visible_cells == 0 and torch.all(flat == 0)
    rctx.release_scene(sid)


def test_one_cell_covering_the_screen(rctx):
    sc = synth.make_scene(1, 16, lambda rng, n: np.zeros((n, 3)), 1.0, 1.2, 0, seed=1)
    _render_and_check(rctx, sc, [synth.small_camera(100, 60)])


def test_termination_halving_stack(rctx):
    from tests.test_oracle_blend import _halving_stack
    sc, _ = _halving_stack(20)
    res = _render_and_check(rctx, sc, [synth.small_camera(9, 9)])
    assert res[0]["err"] <= IMG_TOL


def test_render_is_deterministic(rctx):
    sc = synth.scene_small(sh_degree=3)
    sid = rctx.upload_scene(sc)
    cams = synth.sphere_cameras(2, 3.0, 128, 128)
    a, _, _ = rctx.render(sid, cams)
    b, _, _ = rctx.render(sid, cams)
    torch.cuda.synchronize()
    assert torch.equal(a, b)
    rctx.release_scene(sid)


def test_host_output_matches_device_output(rctx):
    sc = synth.scene_small()
    sid = rctx.upload_scene(sc)
    cams = [synth.small_camera(64, 48)]
    a, _, _ = rctx.render(sid, cams)
    h = np.zeros(3 * 64 * 48, np.float32)
    rctx.render_host(sid, cams, h)
    torch.cuda.synchronize()
    assert np.array_equal(a.cpu().numpy(), h)
    rctx.release_scene(sid)


@pytest.mark.parametrize("n,bits", [(0, 8), (1, 32), (3072, 32), (3073, 13), (6145, 9), (4096, 32), (4097, 13),
                                    (1_000_003, 32), (300_001, 17)])
def test_radix_sort_pairs_stable(rctx, n, bits):
    g = torch.Generator().manual_seed(n + bits)
    keys = torch.randint(0, 2 ** 31, (n,), generator=g, dtype=torch.int64)
    if n > 10:
        keys[: n // 3] = keys[0]  # many equal keys: stability matters
    keys = (keys & ((1 << bits) - 1)).to(torch.int64)
    k32 = keys.to(torch.int32)  # values < 2^31 when bits <= 31, else reinterpret
    vals = torch.arange(n, dtype=torch.int32)
    kd, vd = k32.cuda(), vals.cuda()
    rctx.sort_pairs(kd, vd, bits)
    torch.cuda.synchronize()
    order = np.argsort(keys.numpy().astype(np.uint64), kind="stable")
    assert np.array_equal(vd.cpu().numpy(), order.astype(np.int32))
    assert np.array_equal(kd.cpu().numpy(), k32.numpy()[order])


@pytest.mark.parametrize("n", [2, 1023, 1024, 1025, 9 * 1024 + 1, 262_144, 262_145])
def test_radix_sort_partition_edges(rctx, n):
    """Around a small partition, one look-back of eight partitions, and the
    size at which the partitions grow."""
    test_radix_sort_pairs_stable(rctx, n, 32)


@pytest.mark.parametrize("n_cells", [1, 1023, 2048, 2049, 70_000])
def test_binning_with_most_cells_culled(rctx, n_cells):
    """The depth sort leaves the culled cells out: entry counts around a scan
    partition and a sort partition, a camera inside the scene."""
    sc = synth.make_scene(n_cells, 1, synth._box(-1, 1), 0.002, 0.1, 0, seed=n_cells)
    cams = [synth.look_at((0.1, 0.0, 0.0), (1.0, 0.2, 0.1), 64, 48, 60.0), synth.small_camera(40, 56)]
    _render_and_check(rctx, sc, cams)


@pytest.mark.parametrize("n_cells,sh,offset", [(1, 0, 0), (21, 1, 1), (64, 2, 2), (65, 3, 3), (683, 3, 0)])
def test_update_from_arrays_at_any_alignment(rctx, n_cells, sh, offset):
    """The rows become planes whatever the arrays' widths, row counts (tiles of
    64 rows and more) and alignment: the updated scene renders as the uploaded one."""
    sc = synth.make_scene(n_cells, 3, synth._box(-1, 1), 0.1, 0.4, sh, seed=n_cells)
    other = synth.make_scene(n_cells, 3, synth._box(-1, 1), 0.1, 0.4, sh, seed=n_cells)
    for a in (other.g_mean, other.g_scale, other.g_quat, other.g_logit, other.g_sh):
        a[:] = 0.5
    cam = synth.small_camera(96, 80)

    def shifted(a):
        buf = torch.empty(a.size + 8, device="cuda")
        t = buf[offset:offset + a.size].view(a.shape)
        t.copy_(torch.from_numpy(np.ascontiguousarray(a)))
        return t

    sid, oid = rctx.upload_scene(sc), rctx.upload_scene(other)
    ref = rctx.render(sid, [cam])[0].clone()
    rctx.update_scene(oid, sc.N, sc.K, sh, **{k: shifted(getattr(sc, k)) for k in
                                              ("g_mean", "g_scale", "g_quat", "g_logit", "g_sh")})
    img = rctx.render(oid, [cam])[0]
    assert torch.equal(img, ref)
    rctx.release_scene(sid)
    rctx.release_scene(oid)


def _street():
    sc = synth.make_scene(249_100, 10, synth._ground_plane, 0.05, 0.5, 0, seed=2)
    return sc, synth.street_cameras(1, 320, 192, seed0=3)[0], [
        synth.look_at((0.0, -900.0, 300.0 + i), (0.0, 0.0, 0.0), 48, 32, 60.0) for i in range(3)]


def test_sparse_projection_equals_dense(rctx):
    """A scene of 2.5M Gaussians seen from street level, most cells culled (the
    projection that lists the kept Gaussians first), and the same view beside others that
    see all of it (the direct one): the same image bit for bit."""
    sc, cam, far = _street()
    sid = rctx.upload_scene(sc)
    alone, _, st = rctx.render(sid, [cam], stats=True)
    assert 0 < st.visible_cells < sc.N // 2
    alone = alone.clone()
    both, _, st = rctx.render(sid, [cam] + far, stats=True)
    assert st.visible_cells > 2 * sc.N
    assert torch.equal(both[:alone.numel()], alone)
    rctx.release_scene(sid)


def test_gradients_of_the_sparse_projection(rctx):
    """It clears the gradient accumulators of what it projects: twice the same backward on the
    same buffers, and with the direct projection (the other views' gradient is zero).
    The sums' order, that of atomics, is all that differs."""
    sc, cam, far = _street()
    sid = rctx.upload_scene(sc)
    outs, n = [], 3 * cam.W * cam.H
    dl = torch.randn(n, generator=torch.Generator().manual_seed(6)).cuda()
    for cams in ([cam], [cam], [cam] + far):
        img, state, _ = rctx.render(sid, cams, want_state=True)
        full = torch.zeros(img.numel(), device="cuda")
        full[:n] = dl
        g = dict(g_mean=torch.empty(sc.G, 3, device="cuda"), g_logit=torch.empty(sc.G, device="cuda"),
                 g_sh=torch.empty(sc.G, 1, 3, device="cuda"))
        rctx.backward(state, full, g)
        torch.cuda.synchronize()
        rctx.release_state(state)
        outs.append(g)
    for k, want in outs[2].items():
        assert want.norm() > 0
        for g in outs[:2]:
            assert (g[k] - want).norm() <= 1e-5 * want.norm(), k
    rctx.release_scene(sid)


def test_more_than_65536_tiles(rctx):
    """An odd number of tile-sort passes (17 bits of tile number), the pairs counted on the
    host and on the device."""
    sc = synth.scene_small(n_cells=400)
    cams = [synth.small_camera(4112, 4112)]
    _render_and_check(rctx, sc, cams, tile_rows=(128, 130))
    sid = rctx.upload_scene(sc)
    want = rctx.render(sid, cams, stats=True)[0].clone()
    assert torch.equal(rctx.render(sid, cams)[0], want)
    rctx.release_scene(sid)


def test_loss_l1_matches_definition(rctx):
    g = torch.Generator().manual_seed(0)
    a = torch.rand(1_000_003, generator=g).cuda()
    b = torch.rand(1_000_003, generator=g).cuda()
    b[:10] = a[:10]
    dl = torch.empty_like(a)
    loss = torch.empty(1, device="cuda")
    rctx.loss_l1(a, b, dl, loss)
    torch.cuda.synchronize()
    ref = (a.double() - b.double()).abs().mean().item()
    assert abs(loss.item() - ref) <= 1e-6 * ref
    assert torch.equal(dl, torch.sign(a - b) / a.numel())


def _edge_cells(rng, n):
    # cell centres just outside the left and right edges of the small camera's
    # view at depth 3 (x = +-2.3, world y = 0 is view depth 3)
    side = np.where(np.arange(n) % 2 == 0, -1.0, 1.0)
    return np.stack([side * rng.uniform(2.1, 2.5, n), rng.uniform(-0.4, 0.4, n), rng.uniform(-1.2, 1.2, n)], 1)


def test_gaussians_beyond_the_jacobian_clamp(rctx):
    """Large cells at the frame's edges: many of their Gaussians lie where
    t_x/t_z or t_y/t_z exceeds 1.3 x the half-FOV tangent, so the EWA
    Jacobian is taken at the clamped direction; records, binning and image
    still match the oracle, and the gradients too."""
    sc = synth.make_scene(24, 16, _edge_cells, 1.1, 1.6, 3, seed=21)
    cam = synth.small_camera(96, 64)
    c = cam.as_array()
    R, t = c[7:16].reshape(3, 3).astype(np.float64), c[16:19].astype(np.float64)
    tv = sc.g_mean.astype(np.float64) @ R.T + t
    limx = 1.3 * 0.5 * cam.W / cam.fx
    frac = float((np.abs(tv[:, 0] / tv[:, 2]) > limx).mean())
    assert frac > 0.1, frac
    res = _render_and_check(rctx, sc, [cam])
    assert res[0]["hit"] > 0.2
