"""The benchmark's byte models of the phases that build the tile lists, given the step's count of
cell entries: what the library moves, not what a sort of every pair would."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)
import bench  # noqa: E402


class _Workload:
    cameras = [{"width": 1920, "height": 1080}, {"width": 640, "height": 480},
               {"width": 17, "height": 1}]


def test_views_cells_rounds_partial_cells_up():
    # Cells of 64 x 64 pixels: 30 x 17, 10 x 8, 1 x 1.
    assert bench.views_cells(_Workload, {"tile_w": 16, "tile_h": 16}) == 30 * 17 + 80 + 1
    # Of 128 x 32: 15 x 34, 5 x 15, 1 x 1.
    assert bench.views_cells(_Workload, {"tile_w": 32, "tile_h": 8}) == 15 * 34 + 75 + 1


@pytest.mark.parametrize("entries,cells,passes", [
    (20_000, 255, 1), (20_000, 256, 2), (20_000, 65_535, 2), (20_000, 65_536, 3),
    ((1 << 20) - 1, 300, 2), (1 << 20, 300, 1), (1 << 20, 511, 1), (1 << 20, 512, 2)])
def test_list_phases_follow_the_cell_entries(entries, cells, passes):
    n, V, K, tiles, nv, pairs = 1000, 4, 16, 5000, 2500, 160_000
    stats = {"n_visible": nv, "n_pairs": pairs, "n_eval": 1}
    phases = dict.fromkeys(("preprocess", "compact", "depth_sort", "offsets", "duplicate",
                            "tile_sort", "ranges", "preprocess_backward"), 0.01)
    out = bench.phase_rooflines(phases, stats, n, V, K, tiles, 5000.0, 80.0, (entries, cells))
    assert "offsets" not in out  # the phase does nothing
    expect = {
        "preprocess": 44 * n + n * V / 8 + nv * (44 + 12 * K + 56 + 4),
        "compact": n * V / 8 + nv * (4 + 12),
        "depth_sort": 80 * nv,
        "duplicate": 44 * nv + 8 * entries,
        "tile_sort": passes * 20 * entries,
        "ranges": (4 + 4 + 8) * entries + 3 * 8 * cells + 4 * pairs + 32 * tiles,
        "preprocess_backward": 128 * nv + 8 * (11 + 3 * K) * n,
    }
    assert set(out) == set(expect)
    for name, b in expect.items():
        assert out[name]["bytes"] == pytest.approx(b), name
        assert out[name]["frac"] == pytest.approx(b / 1e-5 / 1e9 / 5000.0)
