"""Maps far from the origin: the rounding of float32 coordinates moves the cull's depth and pixel by
more than its slack, so its margins have to follow it. Every entry whose centre the projection of
the same float32 inputs in double sees inside the image has to be listed."""
import numpy as np
import pytest

from paper_2601_00705_gb300 import synthetic
from paper_2601_00705_gb300.render import Renderer

from gpu_common import to_dev

pytestmark = pytest.mark.gpu

W, H, F = 1000, 700, 1400.0


def _scene(shift, n, seed):
    """Small opaque Gaussians close in front of two cameras, all of it moved by `shift`."""
    rng = np.random.default_rng(seed)
    cams, means = [], []
    for yaw, pitch in ((0.7, 0.2), (-2.1, -0.4)):
        where = np.asarray(shift) + rng.uniform(-1, 1, 3)
        R, _ = synthetic.look_pose(where, yaw, pitch)
        R = np.asarray(R, np.float32)
        t = (-R.astype(np.float64) @ where).astype(np.float32)
        cams.append(synthetic.camera(W, H, F, F, (W - 1) / 2 + 40.0, (H - 1) / 2 - 25.0, R, t))
        z = np.exp(rng.uniform(np.log(0.15), np.log(3.0), n))
        # Near the image's border, on both sides of it.
        u, v = rng.uniform(-20, W + 20, n), rng.uniform(-20, H + 20, n)
        edge = rng.integers(0, 4, n)
        u = np.where(edge == 0, rng.uniform(-20, 20, n), u)
        u = np.where(edge == 1, W - 1 + rng.uniform(-20, 20, n), u)
        v = np.where(edge == 2, rng.uniform(-20, 20, n), v)
        v = np.where(edge == 3, H - 1 + rng.uniform(-20, 20, n), v)
        c = cams[-1]
        xc = np.stack([(u - c["cx"]) / F * z, (v - c["cy"]) / F * z, z], 1)
        means.append((xc - t.astype(np.float64)) @ R.astype(np.float64))
    n *= 2
    g = dict(means=np.concatenate(means), log_scales=np.full((n, 3), -9.0),
             quats=np.tile([1.0, 0, 0, 0], (n, 1)), opacity_logits=np.full(n, 3.0),
             sh=rng.normal(0.0, 0.5, (n, 1, 3)))
    return {k: v.astype(np.float32) for k, v in g.items()}, cams


@pytest.mark.parametrize("jac_clamp", [1.3, 0.0])
@pytest.mark.parametrize("shift", [(3.0, -2.0, 1.0), (1e4, -7e3, 40.0), (6e4, 5e4, -2e3)])
def test_every_entry_inside_the_image_is_listed(shift, jac_clamp):
    n = 40000
    g, cams = _scene(shift, n, 5)
    r = Renderer(0, jac_clamp=jac_clamp)
    p = [to_dev(g[k]) for k in ("means", "log_scales", "quats", "opacity_logits", "sh")]
    *_, state = r.forward_raw(*p, cams)
    assert r.stats(state)["status"] == 0
    _, counts = r.ctx.records(state, 2 * 2 * n)
    r.release(state)
    listed = np.asarray(counts).reshape(2, 2 * n) > 0
    inside = 0
    for v, c in enumerate(cams):
        xc = g["means"].astype(np.float64) @ c["R"].astype(np.float64).T + c["t"].astype(np.float64)
        z = xc[:, 2]
        with np.errstate(divide="ignore", invalid="ignore"):
            u, w = F * xc[:, 0] / z + c["cx"], F * xc[:, 1] / z + c["cy"]
        seen = (z > 0.2 + 1e-6) & (u >= 0) & (u <= W - 1) & (w >= 0) & (w <= H - 1)
        inside += int(seen.sum())
        assert listed[v][seen].all(), (v, int((~listed[v][seen]).sum()), int(seen.sum()))
    assert inside > n // 2
