"""The plane fit's neighbourhoods (oracle/seeding.py, FP64) where their search can go wrong: every
point in one cell, cells that fit one packed key, cells that need the two-word sort, cells beyond
the 21-bit range (clamped), points within rounding of the radius, and fewer points than a warp;
with and without voxel thinning. Normals as in test_gpu_seeding.py (max-abs 1e-5), the same seeds."""
import numpy as np
import pytest
import torch

from oracle import seeding as oseed
from paper_2601_00705_gb300 import seeding, synthetic
from gpu_common import renderer

pytestmark = pytest.mark.gpu

H = float(np.float32(0.05))


def _points(kind, rng, m):
    """Noisy planar patches about the cameras' room, or as the kind says."""
    patches = max(1, m // 60)
    centre = rng.uniform([1.0, 1.0, 0.5], [5.0, 4.0, 2.5], (patches, 3))
    if kind == "one cell":
        centre = np.full((patches, 3), 1.025)
    elif kind == "wide":      # 2^20 cells and more per axis: two words
        centre += rng.choice([0.0, 3e4, -3e4], (patches, 3))
    elif kind == "clamped":   # beyond 2^20 cells of 5 cm from the origin
        centre += rng.choice([0.0, 6e4, -9e4], (patches, 3))
    n = rng.standard_normal((patches, 3))
    n /= np.linalg.norm(n, axis=1, keepdims=True)
    which = np.arange(m) % patches
    d = rng.standard_normal((m, 3))
    d -= (d * n[which]).sum(1, keepdims=True) * n[which]
    d *= (0.02 if kind == "one cell" else 0.06) * rng.random((m, 1)) / np.linalg.norm(
        d, axis=1, keepdims=True)
    X = centre[which] + d + 0.001 * rng.standard_normal((m, 1)) * n[which]
    if kind == "radius":      # partners a rounding inside and outside the radius
        t = rng.standard_normal((m // 2, 3))
        t /= np.linalg.norm(t, axis=1, keepdims=True)
        X[1::2][:m // 2] = X[0::2][:m // 2] + H * t * (
            1.0 + rng.choice([-1e-9, 1e-9], (m // 2, 1)))
    return X


# (Clamped voxels merge, so the thinning of points beyond the range is not the oracle's.)
@pytest.mark.parametrize("kind,m,voxel", [
    ("room", 3001, 0.0), ("room", 3001, 0.03), ("room", 5, 0.0), ("one cell", 700, 0.0),
    ("one cell", 700, 0.03), ("wide", 1500, 0.0), ("wide", 1500, 0.03), ("clamped", 1500, 0.0),
    ("radius", 1200, 0.0)])
def test_normals_of_all_cell_layouts(kind, m, voxel):
    rng = np.random.default_rng(m)
    c = synthetic.correspondences(seed=1021, m=m)
    r = renderer()
    tri = seeding.triangulate(r.ctx, c.cameras, c.ref_view, c.ref_xy, c.nb_view, c.nb_xy,
                              c.nb_conf, r.device, r.stream_handle())
    X = _points(kind, rng, m)
    host = dict(valid=rng.random(m) < 0.95, X=X, err=rng.uniform(0.0, 1.0, m),
                angle=rng.uniform(0.05, 0.5, m), kappa=rng.random(m).astype(np.float32))
    host["valid"][:4] = True
    for k, v in host.items():
        tri[k].copy_(torch.from_numpy(np.ascontiguousarray(v)).to(tri[k].dtype))
    cfg = dict(oseed.DEFAULTS, plane_radius=H, voxel=voxel)
    cfg = {k: float(np.float32(v)) for k, v in cfg.items()}
    host["kappa"] = host["kappa"].astype(np.float64)
    gpu = seeding.init_seeds(r.ctx, c.cameras, tri, c.observed, c.gain_bias, r.device, 1,
                             r.stream_handle(), **cfg)
    ref = oseed.init_seeds(c.cameras, host, c.ref_view, c.nb_view, c.observed, c.gain_bias,
                           sh_degree=1, config=cfg)
    np.testing.assert_array_equal(gpu["index"].cpu().numpy(), ref["index"])
    np.testing.assert_allclose(gpu["means"].cpu().numpy(), ref["means"], rtol=1e-6, atol=1e-6)
    np.testing.assert_allclose(gpu["normals"].cpu().numpy(), ref["normals"], rtol=0, atol=1e-5)
    assert not gpu["sh"][:, 1:].any()
