"""The count of cell entries that a state reports: one per (cell of 4 x 4 tiles, Gaussian) of its
pair list, as long as no footprint skips a cell."""
import numpy as np
import pytest
import torch

from paper_2601_00705_gb300 import synthetic

from gpu_common import gpu_forward

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile_w,tile_h,ppt", [(16, 16, 4), (8, 8, 2), (32, 8, 4)])
def test_entries_are_the_distinct_cells_of_the_pairs(tile_w, tile_h, ppt):
    wl = synthetic.tiny(seed=12, n=3000, width=333, height=251)
    tx, ty = -(-333 // tile_w), -(-251 // tile_h)
    r, *_, state = gpu_forward(wl.gaussians.as_dict(), wl.cameras, tile_w=tile_w, tile_h=tile_h,
                               pixels_per_thread=ppt)
    vals, ranges = r.ctx.tile_lists(state, tx * ty)
    entries = r.ctx.cell_entries(state, torch.cuda.current_stream().cuda_stream)
    r.release(state)
    tile = np.repeat(np.arange(tx * ty), ranges[:, 1].astype(np.int64) - ranges[:, 0])
    cell = (tile // tx // 4) * -(-tx // 4) + tile % tx // 4
    assert entries == np.unique(cell.astype(np.int64) << 32 | vals).size > 0
