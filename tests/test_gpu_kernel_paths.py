"""One small test per dispatch rule of the kernels, at the sizes where a path
can go wrong (remainders of blocks, vectors and batches), against the oracle."""
import dataclasses

import numpy as np
import pytest
import torch

import oracle
from paper_2406_02518_gb300 import binding as B
from paper_2406_02518_gb300 import synthetic as syn
from _parity import check_image, compare_binning, compare_grads, gradient_weights, last_ids
from test_gpu_parity import (GRAD_NAMES, _bins, _lib, _sampled_check, _two_views, _views,  # noqa: F401
                             ws)

pytestmark = pytest.mark.gpu


def _check(scene, views, st, cloud, cfg, ws):
    """Binning, image and every gradient of one render against the oracle."""
    gv = B.views_from_arrays(views)
    img, tf, nl = B.render(cloud, gv, cfg, ws)
    torch.cuda.synchronize()
    bins = _bins(ws, scene, views, st)
    compare_binning(bins, oracle.bin32(scene, views, st))
    ids = last_ids(nl.cpu().numpy().view(np.uint32), bins, views, st.tile)
    rep = check_image(scene, views, st, img.cpu().numpy(), tf.cpu().numpy(), ids)
    w, fm = gradient_weights(rep, 3)
    g = B.render_backward(cloud, gv, cfg, ws, torch.as_tensor(w, dtype=torch.float32, device="cuda"),
                          tf, nl)
    gr = oracle.render_backward(scene, views, st, w, flip_masks=fm)
    gpu = {n: t.float().cpu().numpy() for n, t in g.items()}
    k = cloud.feat_dim
    gpu["feat"] = np.concatenate([gpu.pop("feat_iso").reshape(-1, k), gpu.pop("feat_dir").reshape(-1, k)])
    gpu["pose"] = gpu.pop("world_to_cam")
    compare_grads(gpu, gr, GRAD_NAMES)


def _shifted(t):
    """The same values one element past an allocation's start (never 16-byte aligned)."""
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    buf[1:] = t.reshape(-1)
    return buf[1:].view(t.shape)


@pytest.mark.parametrize("n,k,L,bf16,shift,entangled", [
    (255, 5, 3, False, False, False),   # rows of no whole vectors, a last feature octet of five
    (257, 12, 2, False, False, True),   # whole vectors of four, an octet of four
    (257, 12, 2, False, True, True),    # the same rows off the vector boundary: scalar loads
    (600, 20, 3, True, False, False),   # bfloat16 vectors
    (600, 20, 3, True, True, True),
    (1, 32, 3, False, False, True)])
def test_generic_radiosity_loads(n, k, L, bf16, shift, entangled, ws):
    scene = syn.uniform_cloud(n, seed=80 + k + n, dir_frac=0.5 if n > 1 else 1.0, dir_std=1.0, k=k,
                              sh_degree=L, log_scale_range=(-2.5, -1.5))
    scene = dataclasses.replace(scene, entangled=entangled)
    if bf16:
        scene.feat[scene.n_iso:] = syn.round_to_bf16(scene.feat[scene.n_iso:])
    cloud = B.cloud_from_arrays(scene, feat_dir_bf16=bf16)
    if shift:
        cloud = dataclasses.replace(cloud, feat_iso=_shifted(cloud.feat_iso), feat_dir=_shifted(cloud.feat_dir))
    st = syn.Settings(near_plane=0.2)
    _check(scene, _two_views(45, 60, 8.0 / 56), st, cloud, B.config_from_settings(st), ws)


def _column(n, seed, depths, spread):
    """n Gaussians around the source-to-detector axis, on the given depths (or
    spread over a depth range), so that a few tiles hold nearly all of them."""
    sc = syn.uniform_cloud(n, seed=seed, extent=spread, log_scale_range=(-4.5, -3.5), alpha_range=(0.02, 0.1))
    if depths is not None:
        sc.means[:, 2] = np.asarray(depths, np.float32)[np.arange(n) % len(depths)]
    return sc


@pytest.mark.parametrize("n,size,tile,depths,spread", [
    (2100, 8, 8, None, 0.3),        # two slices of one tile
    (9000, 32, 8, None, 0.3),       # sixteen tiles just past the line
    (60000, 16, 8, None, 0.3),      # the most slices a tile gets
    (30000, 24, 8, (0.0, 0.1, 0.1001), 0.2),  # three depths: most slices empty
    (20000, 16, 16, (0.05,), 0.1)])  # one depth: one slice of 20,000 (chunk sorts, merge)
def test_depth_slices(n, size, tile, depths, spread, ws):
    """Views with many Gaussians per tile: the tile lists, cut into depth
    slices, must be the oracle's whole lists."""
    scene = _column(n, 90 + size, depths, spread)
    views = _views([syn.pose_matrix(np.eye(3), np.array([0.0, 0.0, 2.0])),
                    syn.pose_matrix(syn.rot_y(0.3), np.array([0.02, 0.0, 2.1]))], 4.0, 1.2 / size, size, size)
    st = syn.Settings(near_plane=0.2, tile=tile)
    cloud, gv, cfg = B.cloud_from_arrays(scene), B.views_from_arrays(views), B.config_from_settings(st)
    img, tf, nl = B.render(cloud, gv, cfg, ws)
    torch.cuda.synchronize()
    ref = oracle.bin32(scene, views, st)
    compare_binning(_bins(ws, scene, views, st), ref)
    # the same without a synchronisation, on a workspace reserved by the public sizes, and with
    # room for about half of the pairs: whole tiles only
    tiles = views.n_views * (-(-size // tile)) ** 2
    for pairs, want in ((ref["m"], 0), (ref["m"] // 3, 2)):
        w2 = B.Workspace()
        w2.reserve(views.n_views * n, pairs, tiles)
        i2, _, _ = B.render(cloud, gv, B.config_from_settings(st, no_sync=True), w2)
        fits = ref["m"] <= pairs + pairs // 4 + 4096
        assert w2.sync_status() == (0 if fits else 2)
        got = _bins(w2, scene, views, st)
        if fits:
            compare_binning(got, ref)
            assert torch.equal(i2, img)
        else:
            gr, rr = (x["ranges"].reshape(-1, 2).astype(np.int64) for x in (got, ref))
            for t in range(tiles):
                if gr[t, 1] > gr[t, 0]:
                    assert np.array_equal(gr[t], rr[t])
                    assert np.array_equal(got["vals"][gr[t, 0]:gr[t, 1]], ref["vals"][rr[t, 0]:rr[t, 1]])
        w2.close()


def _needles(n, seed):
    """Gaussians with one axis up to a thousand times the others."""
    sc = syn.uniform_cloud(n, seed=seed, dir_frac=0.4, dir_std=1.0, log_scale_range=(-6.5, -5.5))
    sc.log_scales[: n // 2, 0] += np.float32(4.0)
    return sc


@pytest.mark.parametrize("shape,tile", [
    ((363, 363), 8),    # 2,116 regions of 8 x 8: just past the line, ragged right and bottom edges
    ((361, 359), 8),    # 2,070 regions, a single pixel row and seven columns in the last tiles
    ((352, 352), 8),    # 1,936: the 8 x 4 regions of smaller renders
    ((353, 370), 16),   # 23 x 24 tiles of four regions
    ((340, 421), 32)])  # 11 x 14 tiles of sixteen
@pytest.mark.parametrize("needles", [False, True])
def test_pixel_pair_rasterisers(shape, tile, needles, ws):
    """The rasterisers of both sides of the pixel-pair rule on the same scene:
    sampled pixels of the image and the gradients against the oracle. (The
    needles' shape gradients are left out: binary32 itself is 2e-3 to 6e-3 off
    there in every kernel, the conic of a 400:1 covariance being the cause.)"""
    H, W = shape
    scene = _needles(1500, 61) if needles else syn.uniform_cloud(2500, seed=61, dir_frac=0.4, dir_std=1.0)
    views = _views([syn.pose_matrix(syn.rot_y(0.2), np.array([0.0, 0.1, 2.0]))], 4.0, 8.0 / W, H, W)
    st = syn.Settings(near_plane=0.2, tile=tile)
    grads = [g for g in B.GRAD_FIELDS if not (needles and g in ("log_scales", "quats"))]
    _sampled_check(scene, views, st, ws, [0], 3000, 7, grads, depth=32)


@pytest.mark.parametrize("shape,tile", [((90, 75), 8), ((90, 75), 16), ((75, 90), 32), ((347, 391), 16),
                                        ((384, 381), 32)])
@pytest.mark.parametrize("per_pixel", [False, True])
def test_picked_batches(shape, tile, per_pixel, ws):
    """Lists longer than several batches, of which a region's batches pick the
    covering entries (tiles of 16 and 32), on both sides of the pixel-pair
    rule; with per-pixel rays too."""
    H, W = shape
    scene = syn.uniform_cloud(4000, seed=33, dir_frac=0.5, dir_std=1.0, extent=0.7, log_scale_range=(-4.5, -2.5),
                              alpha_range=(0.02, 0.6))
    scene = dataclasses.replace(scene, per_pixel=per_pixel)
    views = _views([syn.pose_matrix(syn.rot_y(0.2), np.array([0.0, 0.1, 2.0]))], 4.0, 4.0 / W, H, W)
    _sampled_check(scene, views, syn.Settings(near_plane=0.2, tile=tile), ws, [0], 1500, 7, B.GRAD_FIELDS)


@pytest.mark.parametrize("n,tile", [(16, 8), (17, 8), (32, 16), (33, 8), (70, 16)])
def test_pixel_ray_stretches(n, tile, ws):
    """Faint Gaussians over the whole detector: every pair of pixels adds every
    entry of a batch, so the backward's walks fill one stretch of its table
    (16 entries), one and an entry, and both halves of whole batches."""
    scene = syn.uniform_cloud(n, seed=51 + n, dir_frac=0.5, dir_std=1.0, extent=0.2, log_scale_range=(-0.9, -0.5),
                              alpha_range=(0.02, 0.06))
    scene = dataclasses.replace(scene, per_pixel=True)
    st = syn.Settings(near_plane=0.2, tile=tile)
    _check(scene, _two_views(45, 60, 1.0 / 56), st, B.cloud_from_arrays(scene), B.config_from_settings(st), ws)


def test_no_sync_render_without_room_for_slices(ws):
    """A workspace sized by a synchronising render of many tiles takes a no-sync
    render of a crowded view that fits its records, pairs and tiles, although
    it was never reserved for depth slices; a synchronising render of the same
    layout after it uses them again, and the backward of either is accepted."""
    scene = _column(30000, 95, None, 0.3)
    st = syn.Settings(near_plane=0.2, tile=8)
    pose = [syn.pose_matrix(np.eye(3), np.array([0.0, 0.0, 2.0]))]
    large, small = _views(pose, 4.0, 1.2 / 200, 200, 200), _views(pose, 4.0, 1.2 / 16, 16, 16)
    cloud = B.cloud_from_arrays(scene)
    w2 = B.Workspace()
    B.render(cloud, B.views_from_arrays(large), B.config_from_settings(st), w2)
    gv = B.views_from_arrays(small)
    ref = oracle.bin32(scene, small, st)
    for no_sync in (True, False, True):
        cfg = B.config_from_settings(st, no_sync=no_sync)
        img, tf, nl = B.render(cloud, gv, cfg, w2)
        g = B.render_backward(cloud, gv, cfg, w2, torch.ones_like(img), tf, nl)
        assert w2.sync_status() == 0
        compare_binning(_bins(w2, scene, small, st), ref)
        assert float(g["means"].abs().max()) > 0
    w2.close()
