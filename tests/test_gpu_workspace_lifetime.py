"""What outlives one call on a workspace: its memory, and a captured graph's tables
and buffers."""
import numpy as np
import pytest
import torch

import oracle
from paper_2406_02518_gb300 import binding as B
from paper_2406_02518_gb300 import synthetic as syn
from _parity import compare_binning
from test_gpu_kernel_paths import _column
from test_gpu_parity import _bins, _lib, _views  # noqa: F401

pytestmark = pytest.mark.gpu

POSE = [syn.pose_matrix(np.eye(3), np.array([0.0, 0.0, 2.0]))]


def _offset_launches(run):
    """Launches of the binning's offset kernels in one render: three where tiles
    are cut into depth slices, two without."""
    B.profiler_collect()
    B.profiler_enable(True)
    try:
        run()
        torch.cuda.synchronize()
        return B.profiler_collect()["bin_offsets"][1]
    finally:
        B.profiler_enable(False)


@pytest.mark.parametrize("captured", [True, False])
def test_graph_of_a_render_without_slices(captured):
    """A workspace without room for a crowded view's depth slices: the no-sync
    render goes without. Once a graph has captured it, a synchronising render of
    the same layout must leave the graph's tables and buffers as they are; where
    none has, it makes room and uses the slices."""
    scene = _column(30000, 95, None, 0.3)
    st = syn.Settings(near_plane=0.2, tile=8)
    large, small = _views(POSE, 4.0, 1.2 / 200, 200, 200), _views(POSE, 4.0, 1.2 / 16, 16, 16)
    cloud, gv = B.cloud_from_arrays(scene), B.views_from_arrays(small)
    cfg, cfg_ns = B.config_from_settings(st), B.config_from_settings(st, no_sync=True)
    ref = oracle.bin32(scene, small, st)
    w = B.Workspace()
    B.render(cloud, B.views_from_arrays(large), cfg, w)
    out = B.render(cloud, gv, cfg_ns, w)
    dL, grads = torch.ones_like(out[0]), {}
    B.render_backward(cloud, gv, cfg_ns, w, dL, out[1], out[2])
    torch.cuda.synchronize()
    want = [t.clone() for t in out]
    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            B.render(cloud, gv, cfg_ns, w, out=out)
            grads = B.render_backward(cloud, gv, cfg_ns, w, dL, out[1], out[2])
    assert _offset_launches(lambda: B.render(cloud, gv, cfg, w)) == (2 if captured else 3)
    if captured:
        for _ in range(2):
            for t in out:
                t.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert all(torch.equal(a, b) for a, b in zip(out, want))
            assert float(grads["means"].abs().max()) > 0
        assert w.sync_status() == 0
        compare_binning(_bins(w, scene, small, st), ref)
        # another layout ends the graph's claim: the slices come back
        B.render(cloud, B.views_from_arrays(large), cfg, w)
        assert _offset_launches(lambda: B.render(cloud, gv, cfg, w)) == 3
    compare_binning(_bins(w, scene, small, st), ref)
    w.close()


def test_workspaces_return_their_memory():
    """Create, reserve, render a crowded view and destroy, many times: the free
    memory comes back. (Reserving for 4 M records makes room for depth slices.)"""
    scene = _column(2100, 98, None, 0.3)
    st = syn.Settings(near_plane=0.2, tile=8)
    cloud, gv = B.cloud_from_arrays(scene), B.views_from_arrays(_views(POSE, 4.0, 1.2 / 8, 8, 8))
    cfg = B.config_from_settings(st)

    def cycles(n):
        for _ in range(n):
            w = B.Workspace()
            w.reserve(4_000_000, 1 << 20, 4096)
            B.render(cloud, gv, cfg, w)
            w.close()
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    before = cycles(4)
    assert before - cycles(60) < 8 << 20


def test_reserved_batch_of_many_views_keeps_its_slices():
    """A batch on a workspace reserved by its records, pairs and tiles: the depth
    slices of its crowded views have room, however many other views there are and
    however the lists of one view are aligned after another's."""
    st = syn.Settings(near_plane=0.2, tile=8)
    tiny, crowded = _column(1, 96, None, 0.1), _column(8193, 97, None, 0.3)
    view = B.views_from_arrays(_views(POSE, 4.0, 1.2 / 8, 8, 8))  # one tile
    for clouds in ([tiny, crowded] * 40, [tiny] * 400 + [crowded]):
        batch = B.Batch([B.cloud_from_arrays(c) for c in clouds], [view] * len(clouds))
        w = B.Workspace()
        img, _, _ = B.render_batched(batch, B.config_from_settings(st), w)
        pairs = w.pairs()
        w.close()
        w = B.Workspace()
        w.reserve(int(batch.n.sum()), pairs, len(clouds))
        out = [None]

        def run():
            out[0] = B.render_batched(batch, B.config_from_settings(st, no_sync=True), w)

        assert _offset_launches(run) == 3
        assert w.sync_status() == 0
        assert torch.equal(out[0][0], img)
        w.close()
