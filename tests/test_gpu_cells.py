"""The two-level tile lists (cells of 4 x 4 tiles, then tiles) where they can go wrong: images of
a fraction of a cell and of odd size, footprints of one pixel, of the whole image and thin
diagonals that skip cells, emission rounds larger than their buffer, and batches with more cells
than a masked key can number. Lists must hold every entry exactly as often as the projection
counted, in (depth, index) order, and in every tile with a pixel that the blend can cover."""
import math

import numpy as np
import pytest
import torch

from paper_2601_00705_gb300 import synthetic
from paper_2601_00705_gb300.render import Renderer

from gpu_common import gpu_forward, to_dev

pytestmark = pytest.mark.gpu


def _scene(seed, n=60):
    """Footprints from below a pixel to several screens, isotropic ones and needles, in front of
    an identity camera whose field of view they overrun."""
    rng = np.random.default_rng(seed)
    z = rng.uniform(1.0, 5.0, n)
    g = dict(means=np.stack([rng.uniform(-1.2, 1.2, n) * z, rng.uniform(-1.2, 1.2, n) * z, z], 1),
             log_scales=rng.uniform(-6.0, -1.0, (n, 3)), quats=rng.standard_normal((n, 4)),
             opacity_logits=rng.uniform(-2.0, 2.0, n), sh=rng.normal(0.0, 0.5, (n, 1, 3)))
    g["log_scales"][: n // 3, 1:] = -7.0        # needles ...
    g["log_scales"][: n // 3, 0] = rng.uniform(-1.0, 1.0, n // 3)
    g["log_scales"][-2:] = 1.0                  # ... and two that fill the image
    g["opacity_logits"][-2:] = -2.0
    return {k: v.astype(np.float32) for k, v in g.items()}


def _camera(w, h):
    return synthetic.camera(w, h, 0.6 * max(w, h), 0.6 * max(w, h), (w - 1) / 2, (h - 1) / 2,
                            np.eye(3), np.zeros(3))


@pytest.mark.parametrize("w,h,tw,th,ppt", [
    (1, 1, 16, 16, 4), (17, 1, 16, 16, 4), (65, 63, 16, 16, 4), (130, 257, 8, 8, 2),
    (257, 33, 32, 8, 4), (2051, 1100, 16, 16, 4)])
def test_lists_of_odd_sizes(w, h, tw, th, ppt):
    cfg = dict(tile_w=tw, tile_h=th, pixels_per_thread=ppt)
    g, cams = _scene(7 * w + h), [_camera(w, h), _camera(max(1, w // 2), h)]
    tiles = sum(-(-c["width"] // tw) * -(-c["height"] // th) for c in cams)
    n = g["means"].shape[0]
    r, *_, state = gpu_forward(g, cams, **cfg)
    vals, ranges = r.ctx.tile_lists(state, tiles)
    rec, counts = r.ctx.records(state, 2 * n)
    stats = r.stats(state)
    r.release(state)
    assert vals.size == int(counts.sum()) == stats["n_pairs"]
    np.testing.assert_array_equal(np.bincount(vals, minlength=2 * n), counts)
    lengths = ranges[:, 1].astype(np.int64) - ranges[:, 0]
    held = lengths > 0
    np.testing.assert_array_equal(ranges[held, 0], np.cumsum(lengths[held]) - lengths[held])
    tile = np.repeat(np.arange(tiles), lengths)
    key = (rec[vals, 11].view(np.uint32).astype(np.uint64) << np.uint64(32)) | vals
    assert np.all(key[1:][tile[1:] == tile[:-1]] > key[:-1][tile[1:] == tile[:-1]])
    # Every pixel whose exponent, from the records in double, is within 1e-4 of the coverage
    # threshold (the FP32 exponent differs by a few 1e-6) lies in a listed tile of its entry.
    base, checked = 0, 0
    for v, c in enumerate(cams):
        tx = -(-c["width"] // tw)
        y, x = np.mgrid[0:c["height"], 0:c["width"]]
        of_pixel = base + (y // th) * tx + x // tw
        for i in np.nonzero(counts[v * n:(v + 1) * n])[0]:
            r0 = rec[v * n + i].astype(np.float64)
            dx, dy = x - (r0[0] + r0[2]), y - (r0[1] + r0[3])
            e = r0[7] - (r0[4] * dx + r0[5] * dy) ** 2 - (r0[6] * dy) ** 2
            need = np.unique(of_pixel[e >= np.log2(np.float64(np.float32(1 / 255))) - 1e-4])
            assert np.isin(need, tile[vals == v * n + i]).all(), (v, i)
            checked += need.size
        base += tx * -(-c["height"] // th)
    assert checked > 0


def test_more_cells_than_a_masked_key_numbers():
    # 17 views of 64 x 64 cells (8x8 tiles): 69,632 cells. Each view must come out exactly as on
    # its own, where its cells carry masks.
    g = _scene(3, n=400)
    p = [to_dev(g[k]) for k in ("means", "log_scales", "quats", "opacity_logits", "sh")]
    cam = _camera(2048, 2048)
    cams = []
    for v in range(17):
        a = 0.02 * v
        R = np.array([[math.cos(a), 0, math.sin(a)], [0, 1, 0], [-math.sin(a), 0, math.cos(a)]])
        cams.append(dict(cam, R=R.astype(np.float32), t=np.array([0.01 * v, 0, 0], np.float32)))
    r = Renderer(0, tile_w=8, tile_h=8, pixels_per_thread=2)
    *together, state = r.forward_raw(*p, cams)
    assert r.stats(state)["status"] == 0
    r.release(state)
    P = 2048 * 2048
    for v in (0, 8, 16):
        *alone, state = r.forward_raw(*p, cams[v:v + 1])
        torch.cuda.synchronize()
        for a, b in zip(together, alone):
            assert torch.equal(a[v * P:(v + 1) * P], b), v
        r.release(state)
