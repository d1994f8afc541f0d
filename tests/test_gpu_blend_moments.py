"""Accuracy of the backward blend's footprint moments: small footprints in every row of their tile,
for each number of pixels per thread that sums its rows in pairs. The moments of a Gaussian far
from the row they are summed about cancel; summed about the row nearest to its centre they keep
the precision of their terms."""
import numpy as np
import pytest

import oracle
from paper_2601_00705_gb300 import synthetic

from gpu_common import gpu_render, masked_l1_upstream, rel_l2

pytestmark = pytest.mark.gpu

# 32 roundings of 2^-24: a moment adds up a few dozen products of rounded factors.
MOMENT_RTOL = 32 * 2.0 ** -24


@pytest.mark.parametrize("tile_w,tile_h,bwd_ppt", [(16, 16, 2), (16, 16, 4), (16, 16, 8),
                                                   (32, 8, 4), (32, 8, 8), (8, 8, 2)])
@pytest.mark.parametrize("weight_depth", [0.0, 0.1])
def test_shape_gradients_keep_their_precision(tile_w, tile_h, bwd_ppt, weight_depth):
    wl = synthetic.tiny(seed=31)
    g = wl.gaussians.as_dict()
    orc0 = oracle.render(g, wl.cameras)
    rng = np.random.default_rng(8)
    d_color, keep = masked_l1_upstream(orc0, rng.random(orc0["color"].shape))
    d_depth = None
    if weight_depth:
        d_depth = (weight_depth * rng.choice([-1.0, 1.0], keep.size) / keep.size).astype(np.float32)
        d_depth[~keep] = 0.0
    orc = oracle.render(g, wl.cameras, d_color=d_color, d_depth=d_depth)
    gpu = gpu_render(g, wl.cameras, d_color=d_color, d_depth=d_depth, tile_w=tile_w, tile_h=tile_h,
                     pixels_per_thread=2, backward_pixels_per_thread=bwd_ppt)
    errs = {k: rel_l2(gpu[k], orc[k]) for k in ("g_log_scales", "g_quats")}
    assert all(e <= MOMENT_RTOL for e in errs.values()), errs
