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
from test_gpu_parity import GRAD_NAMES, _bins, _lib, _two_views, _views, ws  # noqa: F401

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
