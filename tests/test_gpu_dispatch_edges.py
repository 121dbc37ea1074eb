"""Branches of the kernels' dispatch that only larger or mixed renders reach:
crowded views (depth slices) with enough 8 x 8 regions for the pixel-pair
backward but not for the pixel-pair forward, views cut into different numbers of
slices in one batch, and RADS volumes of more crossings than one digit selects
among or one block sums."""
import numpy as np
import pytest
import torch

import oracle
from oracle import rads as orads
from paper_2406_02518_gb300 import binding as B
from paper_2406_02518_gb300 import synthetic as syn
from _parity import compare_grads
from test_gpu_kernel_paths import _column, _needles
from test_gpu_parity import _compare_view_lists, _lib, _sampled_check, _views, ws  # noqa: F401

pytestmark = pytest.mark.gpu

# The 8 x 4 forward with row-pair covers serves sliced renders of at least 2,048
# regions and fewer than one for each of the forward's 32 warps per SM.
PAIR_REGIONS = 2048


@pytest.mark.parametrize("tile,side,n_views,n,scales,dilation", [
    (32, 31, 130, 1300, (-4.5, -3.5), 0.3),   # one ragged tile of sixteen regions a view
    (16, 61, 34, 17000, (-6.5, -5.5), 0.1),   # sixteen tiles of four
    (8, 24, 240, 9500, (-6.5, -5.5), 0.05),   # nine tiles of one
    (32, 32, 129, 1300, None, 0.3)])          # needles: ellipses that rounding can take out of their boxes
def test_sliced_renders_with_few_regions(tile, side, n_views, n, scales, dilation, ws):
    nt = (-(-side // tile)) ** 2
    regions = n_views * nt * (tile // 8) ** 2
    assert PAIR_REGIONS <= regions < 32 * torch.cuda.get_device_properties(0).multi_processor_count
    assert n > 1024 * nt  # cut into slices
    scene = _needles(n, 63) if scales is None else syn.uniform_cloud(
        n, seed=64 + tile, extent=0.3, dir_frac=0.4, dir_std=1.0, log_scale_range=scales, alpha_range=(0.02, 0.1))
    poses = [syn.pose_matrix(syn.rot_y(0.2 * np.sin(v)), np.array([0.01 * np.cos(v), 0.0, 2.0])) for v in range(n_views)]
    st = syn.Settings(near_plane=0.2, tile=tile, dilation=dilation)
    # (the needles' shape gradients are 2e-3 to 6e-3 off in binary32 itself, in every kernel)
    grads = [g for g in B.GRAD_FIELDS if not (scales is None and g in ("log_scales", "quats"))]
    _sampled_check(scene, _views(poses, 4.0, 1.2 / side, side, side), st, ws, [0, n_views - 1], 1200, 7, grads)


def test_batch_of_views_with_different_slices():
    """Views cut into 1 to 32 slices, one after another: the gaps that align their
    lists, the lists against the oracle's, images and gradients against each
    request's own render."""
    st = syn.Settings(near_plane=0.2, tile=8)
    cfg = B.config_from_settings(st)
    sizes = [(1, 8), (8193, 8), (700, 20), (1025, 8), (0, 16), (40000, 16), (3, 8), (2049, 8), (9300, 24), (500, 33)]
    scenes = [_column(n, 200 + k, None, 0.3) for k, (n, _) in enumerate(sizes)]
    views = [_views([syn.pose_matrix(syn.rot_y(0.1 * k), np.array([0.0, 0.0, 2.0]))], 4.0, 1.2 / s, s, s)
             for k, (_, s) in enumerate(sizes)]
    batch = B.Batch([B.cloud_from_arrays(s) for s in scenes], [B.views_from_arrays(v) for v in views])
    wb, w1 = B.Workspace(), B.Workspace()
    img, tf, nl = B.render_batched(batch, cfg, wb)
    dL = torch.linspace(-1, 1, batch.pixels, device="cuda")
    g = B.render_batched_backward(batch, cfg, wb, dL, tf, nl)
    tiles = [(-(-s // 8)) ** 2 for _, s in sizes]
    bins = B.debug_binning(wb, 1, int(batch.n.sum()), sum(tiles))
    n_off, t_off = np.concatenate([[0], np.cumsum(batch.n)]), np.concatenate([[0], np.cumsum(tiles)])
    iso_off, dir_off = np.concatenate([[0], np.cumsum(batch.n_iso)]), np.concatenate([[0], np.cumsum(batch.n - batch.n_iso)])
    for r, (scene, view) in enumerate(zip(scenes, views)):
        if scene.n:
            ref = oracle.bin32(scene, view, st)
            part = dict(bins, ranges=bins["ranges"].reshape(-1, 2)[t_off[r]:t_off[r + 1]],
                        keys=bins["keys"] - (np.uint64(t_off[r]) << np.uint64(32)))
            _compare_view_lists(part, ref, [0], tiles[r])
        cloud, gv = B.cloud_from_arrays(scene), B.views_from_arrays(view)
        one = B.render(cloud, gv, cfg, w1)
        for a, b in zip((img, tf, nl), one):
            assert torch.equal(batch.view_slice(a, r), b[0])
        if not scene.n:
            continue
        gs = B.render_backward(cloud, gv, cfg, w1, batch.view_slice(dL, r)[None].contiguous(), one[1], one[2])
        got = {k: g[k][n_off[r]:n_off[r + 1]] for k in ("means", "log_scales", "quats", "opacity_logits")}
        got.update(feat_iso=g["feat_iso"][iso_off[r]:iso_off[r + 1]], feat_dir=g["feat_dir"][dir_off[r]:dir_off[r + 1]],
                   b_iso=g["b_iso"][r], B_dir=g["B_dir"][r], world_to_cam=g["world_to_cam"][r:r + 1])
        # equal up to the order of atomic additions
        compare_grads({k: t.cpu().numpy() for k, t in got.items()}, {k: t.cpu().numpy() for k, t in gs.items()},
                      list(got), tol=1e-5, zero_ok=list(got))
    wb.close()
    w1.close()


@pytest.mark.parametrize("shape,least", [
    ((150, 150, 152), 1 << 22),    # a second digit of the selection; rows of whole vectors
    ((183, 185, 187), 1 << 23)])   # more than 2,048 blocks of keys: scanned offsets; odd rows
def test_rads_of_many_crossings(shape, least, ws):
    hu = np.random.default_rng(5).integers(-1000, 1001, shape).astype(np.int16)
    r = B.rads(torch.as_tensor(hu, device="cuda"), (0.5, 0.5, 0.5), (1.0, 2.0, 3.0), 3000, 500, seed=9, ws=ws, debug=True)
    torch.cuda.synchronize()
    ref = orads.rads(hu, (0.5, 0.5, 0.5), (1.0, 2.0, 3.0), 3000, 500, seed=9)
    assert r["n_crossings"] == ref["n_crossings"] > least
    assert np.array_equal(r["kept_edges"].cpu().numpy(), ref["edge_ids"])
    assert np.array_equal(r["draw_voxels"].cpu().numpy(), ref["draw_voxels"])
    # as in the other RADS tests: binary32 interpolation, a few ulp at 100 mm
    assert np.abs(r["means"].cpu().numpy() - ref["means"]).max() <= 1e-4
