"""Host logic of the depth slices (ddgs::plan_slices) where views that are cut
lie between views that are not: the gaps that align their lists are part of
what a workspace reserved by records and tiles has room for. Compiled into a
small host program."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

_PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "ddgs_internal.cuh"

// views of `side` pixels at tile 8, request r of n[r % cycle] Gaussians
static int check(int V, const std::vector<int64_t> &n, const std::vector<int> &side) {
  std::vector<ddgs::ReqTab> req(V + 1);
  std::vector<ddgs::ViewTab> view(V + 1);
  int64_t tiles = 0, records = 0;
  for (int v = 0; v < V; ++v) {
    req[v].n = n[v % n.size()];
    ddgs::ViewTab &t = view[v];
    t.req = v;
    t.H = t.W = side[v % side.size()];
    t.tiles_x = (t.W + 7) / 8;
    t.tile_base = tiles;
    tiles += (int64_t)t.tiles_x * t.tiles_x;
    records += req[v].n;
  }
  view[V].tile_base = tiles;
  ddgs::RenderShape s{};
  ddgs::plan_binning(view.data(), V, req.data(), tiles, 8, s);
  ddgs::plan_slices(view.data(), V, req.data(), 8, s);
  const int64_t bound = ddgs::vtile_bound(tiles, records);
  const bool ok = s.total_vtiles <= bound && s.hist_slots < ddgs::hist_slot_bound(bound);
  printf("%d views, %lld lists, bound %lld%s\n", V, (long long)s.total_vtiles, (long long)bound, ok ? "" : " FAIL");
  return ok ? 0 : 1;
}

int main() {
  int bad = 0;
  for (int V : {2, 3, 200, 16000}) {
    bad += check(V, {1, 8193}, {8});             // one tile in 32 slices after one tile
    bad += check(V, {500, 1025}, {8});           // the least that is cut
    bad += check(V, {1, 1, 1, 2049}, {8});
    bad += check(V, {8193, 1025, 1, 2049}, {8});
    bad += check(V, {1, 40000}, {8, 16});        // four tiles
    bad += check(V, {3, 1 << 20}, {24, 64});
  }
  return bad;
}
"""


def test_gaps_between_sliced_views_are_within_the_reserved_bounds(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "gaps.cu", tmp_path / "gaps"
    src.write_text(_PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I",
                    os.path.join(ROOT, "paper_2406_02518_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    str(src), "-o", str(exe)], check=True, capture_output=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
