"""Accuracy of the backward blend's footprint moments on thin, tilted footprints of tens to hundreds
of pixels whose centres lie in other tiles: in a tile, the pixels that such a footprint covers lie
around its ridge, many rows from the row nearest to its centre."""
import numpy as np
import pytest

import oracle
from paper_2601_00705_gb300 import synthetic

from gpu_common import gpu_render, masked_l1_upstream, rel_l2

pytestmark = pytest.mark.gpu

# A term of a moment multiplies eight rounded factors (alpha, the transmittance, the colour
# difference seen behind, the upstream gradient's weight, and the offsets across the footprint);
# what cancels in the sums must not add to that.
MOMENT_RTOL = 8 * 2.0 ** -24


def _needles(seed, n=300, w=160, h=120, f=150.0):
    """Needles through random points of the image, their centres up to 120 px along their axes."""
    rng = np.random.default_rng(seed)
    z = rng.uniform(1.0, 3.0, n)
    ang = rng.uniform(0.0, np.pi, n)
    length, width = np.exp(rng.uniform(np.log(15), np.log(120), n)), rng.uniform(0.5, 1.5, n)
    px, py = rng.uniform(0, w, n), rng.uniform(0, h, n)
    along = rng.uniform(-1, 1, n) * length
    cx, cy = px + along * np.cos(ang), py + along * np.sin(ang)
    g = dict(means=np.stack([(cx - (w - 1) / 2) / f * z, (cy - (h - 1) / 2) / f * z, z], 1),
             log_scales=np.log(np.stack([length, width, width], 1) * (z / f)[:, None]),
             quats=np.stack([np.cos(ang / 2), 0 * ang, 0 * ang, np.sin(ang / 2)], 1),
             opacity_logits=rng.uniform(-3.0, -1.0, n), sh=rng.normal(0.0, 0.5, (n, 1, 3)))
    cam = synthetic.camera(w, h, f, f, (w - 1) / 2, (h - 1) / 2, np.eye(3), np.zeros(3))
    return {k: v.astype(np.float32) for k, v in g.items()}, [cam]


@pytest.mark.parametrize("tile_w,tile_h,bwd_ppt", [(16, 16, 2), (16, 16, 4), (16, 16, 8),
                                                   (32, 8, 8), (8, 8, 2)])
@pytest.mark.parametrize("seed", [1, 2])
def test_thin_axes_keep_their_precision(tile_w, tile_h, bwd_ppt, seed):
    g, cams = _needles(seed)
    orc0 = oracle.render(g, cams)
    d_color, keep = masked_l1_upstream(orc0, np.random.default_rng(8).random(orc0["color"].shape))
    assert keep.mean() > 0.99
    orc = oracle.render(g, cams, d_color=d_color)
    gpu = gpu_render(g, cams, d_color=d_color, tile_w=tile_w, tile_h=tile_h, pixels_per_thread=2,
                     backward_pixels_per_thread=bwd_ppt)
    # The gradients of the two thin axes; the long one's follows from small differences of sums.
    err = rel_l2(gpu["g_log_scales"][:, 1:], orc["g_log_scales"][:, 1:])
    assert err <= MOMENT_RTOL, err
