"""The backward blend's pixels per thread where the caller leaves them open: just below and at the
number of tiles from which a thread takes eight, for both tile shapes that allow it."""
import numpy as np
import pytest

from paper_2601_00705_gb300 import synthetic

from gpu_common import gpu_render

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile_w,tile_h", [(16, 16), (32, 8)])
@pytest.mark.parametrize("tiles_y,height_less", [(47, 0), (48, 0), (48, 3)])
def test_open_choice_equals_explicit_settings(tile_w, tile_h, tiles_y, height_less):
    # 38 tiles by 47 (1786) or 48 (1824); a last row of tiles that the image does not fill.
    w, h = 38 * tile_w, tiles_y * tile_h - height_less
    g = synthetic.tiny(seed=3).gaussians.as_dict()
    cams = [synthetic.camera(w, h, 0.9 * w, 0.9 * w, (w - 1) / 2, (h - 1) / 2, np.eye(3),
                             np.zeros(3))]
    d_color = np.random.default_rng(4).choice([-1.0, 1.0], (w * h, 3)) / (w * h)
    cfg = dict(tile_w=tile_w, tile_h=tile_h, pixels_per_thread=4)
    out = gpu_render(g, cams, d_color=d_color, **cfg)
    for ppt in (4, 8):
        ref = gpu_render(g, cams, d_color=d_color, backward_pixels_per_thread=ppt, **cfg)
        np.testing.assert_array_equal(out["color"], ref["color"])
        # Sums in another order: a few dozen roundings of 2^-24 relative to the largest gradient.
        for k in ("g_means", "g_log_scales", "g_quats", "g_opacity_logits", "g_sh", "g_pose"):
            np.testing.assert_allclose(out[k], ref[k], rtol=1e-4, atol=1e-5 * np.abs(ref[k]).max(),
                                       err_msg=k)
