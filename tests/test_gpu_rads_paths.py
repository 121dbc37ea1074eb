"""The branches of the RADS initialisation at their edges, against plain numpy:
the neighbour search's grid on clustered, flat and tiny clouds, and the last
step of the selection where few and many keys share a prefix."""
import numpy as np
import pytest
import torch

from oracle import rads as orads
from paper_2406_02518_gb300 import binding as B
from test_gpu_parity import _lib, ws  # noqa: F401

pytestmark = pytest.mark.gpu


def _volume(shape, blobs, seed, noise):
    """Soft background with bright boxes (z, y, x, size) and integer noise."""
    rng = np.random.default_rng(seed)
    hu = rng.integers(-noise, noise + 1, shape).astype(np.int16) if noise else np.zeros(shape, np.int16)
    for z, y, x, s in blobs:
        hu[z:z + s, y:y + s, x:x + s] += 1000
    return hu


@pytest.mark.parametrize("shape,spacing,blobs,noise,n1,n2", [
    ((40, 64, 48), (0.5, 0.5, 0.5), [(3, 3, 3, 4)], 0, 400, 300),          # every point in one corner
    ((40, 63, 47), (0.5, 0.7, 2.0), [(3, 3, 3, 4), (30, 50, 40, 5)], 0, 500, 300),  # two far clusters, odd rows
    ((1, 200, 160), (1.0, 1.0, 1.0), [(0, 20, 20, 60)], 3, 300, 500),      # a single slice: a flat grid
    ((1, 1, 4096), (0.25, 1.0, 1.0), [], 900, 700, 700),                   # a line of cells
    ((16, 16, 16), (1.0, 1.0, 1.0), [(4, 4, 4, 8)], 0, 0, 3),              # fewer points than neighbours
    ((64, 64, 64), (1.0, -1.0, 1.0), [(20, 20, 20, 24)], 30, 2000, 1500),  # a descending axis
    ((96, 128, 128), (0.5, 0.5, 0.5), [], 1000, 9000, 100)])               # 2.3 M crossings: 1,100 share a prefix
def test_rads_paths(shape, spacing, blobs, noise, n1, n2, ws):
    hu = _volume(shape, blobs, 5, noise)
    origin = (-3.0, 4.0, 100.0)
    r = B.rads(torch.as_tensor(hu, device="cuda"), spacing, origin, n1, n2, seed=9, ws=ws, debug=True)
    torch.cuda.synchronize()
    means, ls = r["means"].cpu().numpy(), r["log_scales"].cpu().numpy()
    ref = orads.rads(hu, spacing, origin, n1, n2, seed=9)
    assert r["n_crossings"] == ref["n_crossings"]
    assert np.array_equal(r["kept_edges"].cpu().numpy(), ref["edge_ids"])
    assert np.array_equal(r["draw_voxels"].cpu().numpy(), ref["draw_voxels"])
    # the neighbour search over the call's own points, in binary32 like the kernel: d^2 = fma(dz,
    # dz, fma(dy, dy, dx dx)) differs from the plain sum by two roundings (2^-23 relative), and
    # the logarithm's half by half of that plus one ulp of log s (at most 2^-21 here)
    p = means.astype(np.float64)
    want = np.empty(len(p))
    for a in range(0, len(p), 512):
        d2 = ((p[a:a + 512, None] - p[None]) ** 2).sum(-1)
        d2[np.arange(len(d2)), a + np.arange(len(d2))] = np.inf
        k = min(3, len(p) - 1)
        m = np.sort(np.partition(d2, k - 1, axis=1)[:, :k], axis=1).mean(1) if k else np.zeros(len(d2))
        want[a:a + 512] = 0.5 * np.log(np.maximum(m, 1e-7))
    assert np.abs(ls - want[:, None]).max(initial=0) <= 2e-6
