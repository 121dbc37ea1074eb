"""The basis gradients of the generic radiosity kernels take nothing from a
Gaussian whose weight is zero (one that no view sees, or the term of Eq. 3 that
it does not carry), whatever its features are."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2406_02518_gb300 import binding as B
from paper_2406_02518_gb300 import synthetic as syn
from test_gpu_parity import _lib, _two_views, ws  # noqa: F401

pytestmark = pytest.mark.gpu


def _basis_gradients(scene, ws):
    views, cfg = B.views_from_arrays(_two_views(45, 60, 8.0 / 56)), B.config_from_settings(syn.Settings(near_plane=0.2))
    cloud = B.cloud_from_arrays(scene)
    out = (torch.empty((2, 45, 60), device="cuda"), torch.empty((2, 45, 60), device="cuda"),
           torch.empty((2, 45, 60), dtype=torch.int32, device="cuda"))
    try:
        B.render(cloud, views, cfg, ws, out=out)
    except B.DDGSError as e:  # reported, and the outputs are written
        assert e.code == 3 and not np.isfinite(scene.feat).all()
    g = B.render_backward(cloud, views, cfg, ws, torch.ones_like(out[0]), out[1], out[2], want=("b_iso", "B_dir"))
    return {k: v.cpu().numpy() for k, v in g.items()}


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("k,L,entangled", [(5, 1, False), (12, 2, True), (32, 3, False)])
def test_features_of_weight_zero(k, L, entangled, value, ws):
    n = 300  # two blocks
    scene = syn.uniform_cloud(n, seed=70 + k, dir_frac=0.5, dir_std=1.0, k=k, sh_degree=L,
                              log_scale_range=(-2.5, -1.5))
    scene = dataclasses.replace(scene, entangled=entangled)
    unseen = [3, n - 2]  # behind the source: an isotropic and a direction-dependent one
    scene.means[unseen] = (0.0, 0.0, -50.0)
    want = _basis_gradients(scene, ws)
    scene.feat[unseen] = value
    got = _basis_gradients(scene, ws)
    for name in want:
        # the sums differ by the order of the 2D gradients' atomic additions alone
        assert np.abs(want[name]).max() > 0
        assert np.abs(got[name] - want[name]).max() <= 1e-4 * np.abs(want[name]).max(), name


@pytest.mark.parametrize("L", [1, 3])
def test_features_of_the_other_term(L, ws):
    """A visible isotropic Gaussian's features reach b_iso's gradient, never B_dir's."""
    scene = syn.uniform_cloud(300, seed=77, dir_frac=0.5, dir_std=1.0, k=6, sh_degree=L, log_scale_range=(-2.5, -1.5))
    scene.feat[5, 2] = np.inf
    scene.means[5] = (0.0, 0.0, 0.0)
    g = _basis_gradients(scene, ws)
    assert np.isfinite(g["B_dir"]).all() and np.abs(g["B_dir"]).max() > 0
