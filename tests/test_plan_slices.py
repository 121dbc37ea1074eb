"""Host logic of the depth slices (ddgs::plan_slices), compiled into a small host
program over the layouts of the binning plan's test: only crowded views are
cut, lists are aligned for the offsets kernel, the counters stay within bands
and below the sizes that a workspace reserved by records and tiles holds."""
import os
import shutil
import subprocess

import pytest

from test_plan_binning import _PROGRAM, ROOT

_SLICES = _PROGRAM[:_PROGRAM.index("    int64_t items = 0, slots = 0;")] + r"""
    const std::vector<ddgs::ViewTab> before = view;
    ddgs::plan_slices(view.data(), V, req.data(), tile, s, budget);
    int64_t items = 0, slots = 0, lists = 0, records = 0;
    bool any = false;
    for (int v = 0; v < V; ++v) {
      const ddgs::ViewTab &t = view[v], &b = before[v];
      const int64_t nt = (int64_t)t.tiles_x * ((t.H + tile - 1) / tile), n = req[t.req].n;
      const int lg = t.lg_slices;
      records += n;
      if (lg < 0 || (1 << lg) > ddgs::SLICE_MAX || (lg > 0 && n <= ddgs::SLICE_FROM * nt)) { printf("FAIL slices\n"); return 1; }
      if (lg == 0 && n > ddgs::SLICE_FROM * nt && 2 * nt <= ddgs::BIN_HIST_MAX) { printf("FAIL not sliced\n"); return 1; }
      if (t.vtile_base < lists || t.vtile_base % (1 << lg) || t.vtile_base - lists >= (1 << lg)) { printf("FAIL list base\n"); return 1; }
      lists = t.vtile_base + (nt << lg);
      if ((((int64_t)t.band_w * t.band_h) << lg) > ddgs::BIN_HIST_MAX) { printf("FAIL band too large\n"); return 1; }
      if (t.band_w != b.band_w || t.band_h != b.band_h || t.bands_x != b.bands_x) { printf("FAIL bands moved\n"); return 1; }
      if ((n == 0) != (t.chunks == 0) || t.chunks > b.chunks) { printf("FAIL chunks\n"); return 1; }
      if (t.item_base != items || t.hist_base != slots) { printf("FAIL bases\n"); return 1; }
      const int64_t by = ((t.H + tile - 1) / tile + t.band_h - 1) / t.band_h;
      items += (int64_t)t.chunks * t.bands_x * by;
      slots += ((int64_t)t.chunks * t.bands_x * by * t.band_w * t.band_h) << lg;
      if (t.chunks > 0 && (((int64_t)t.band_w * t.band_h) << lg) > s.hist_area) { printf("FAIL hist_area\n"); return 1; }
      any |= lg > 0;
    }
    if (lists != s.total_vtiles || view[V].vtile_base != lists || any != (s.sliced != 0) || (!any && lists != tiles)) { printf("FAIL lists\n"); return 1; }
    if (items != s.n_items || slots != s.hist_slots || view[V].item_base != items) { printf("FAIL totals\n"); return 1; }
    // what ddgs_workspace_reserve(records, pairs, tiles) makes room for
    if (lists > ddgs::vtile_bound(tiles, records)) { printf("FAIL list bound\n"); return 1; }
    if (s.hist_slots >= ddgs::hist_slot_bound(ddgs::vtile_bound(tiles, records), budget)) { printf("FAIL slot bound\n"); return 1; }
    layouts += any;
  }
  printf("ok %d\n", layouts);
  return layouts > 50 ? 0 : 1;
}
"""


def test_depth_slices_stay_within_the_reserved_bounds(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    src = tmp_path / "slices.cu"
    src.write_text(_SLICES)
    exe = tmp_path / "slices"
    inc = os.path.join(ROOT, "paper_2406_02518_gb300", "csrc")
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-I", inc, "-I",
                    os.path.join(ROOT, "include"), str(src), "-o", str(exe)], check=True,
                   capture_output=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
