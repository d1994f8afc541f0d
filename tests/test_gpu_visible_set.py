"""What counts as seen (observation counts, n_visible) on views whose edge tiles reach past the
image: an entry in the overhang is seen exactly when its footprint's bounding radius, widened by
2 % and 4 px, reaches the image, whatever test picks the candidates. Expected counts come from the
parameters, in double."""
import numpy as np
import pytest

from paper_2601_00705_gb300 import binding, synthetic
from paper_2601_00705_gb300.mapping import MapRegularizer
from paper_2601_00705_gb300.render import Renderer

from gpu_common import to_dev

pytestmark = pytest.mark.gpu

# Entries this close (px) to a decision are left out: the float32 centre and radius are within a
# few ulps of 1200 px of the double ones, the tile cover is padded by 1/16 px, and where a footprint
# barely reaches the grid of tiles the count is not checked.
NEAR, REACH = 1e-2, 0.25


def _scene(n, seed):
    rng = np.random.default_rng(seed)
    z = rng.uniform(0.6, 8.0, n)
    g = dict(means=np.stack([rng.uniform(-1.3, 1.3, n) * z, rng.uniform(-0.9, 0.9, n) * z, z], 1),
             log_scales=rng.normal(-5.0, 0.4, (n, 3)), quats=rng.standard_normal((n, 4)),
             opacity_logits=rng.uniform(-1.0, 4.0, n), sh=rng.normal(0.0, 0.5, (n, 1, 3)))
    return {k: v.astype(np.float32) for k, v in g.items()}


def _decide(g, cam, alpha_min=float(np.float32(1 / 255)), eps=float(np.float32(0.3)), tile=16):
    """(seen, undecided) of every Gaussian in one view."""
    m, ls, q, lg = (g[k].astype(np.float64) for k in ("means", "log_scales", "quats",
                                                      "opacity_logits"))
    R, t = np.asarray(cam["R"], np.float64), np.asarray(cam["t"], np.float64)
    f = np.array([np.float32(cam["fx"]), np.float32(cam["fy"])], np.float64)
    c = np.array([np.float32(cam["cx"]), np.float32(cam["cy"])], np.float64)
    size = np.array([cam["width"], cam["height"]], np.float64)
    xc = m @ R.T + t
    z = xc[:, 2]
    front = z > 0.2
    zs = np.where(front, z, 1.0)[:, None]
    u = xc[:, :2] / zs
    lim = float(np.float32(1.3)) * 0.5 * size / f
    uc = np.clip(u, -lim, lim)
    centre = f * u + c
    kappa = 2.0 * np.log(1.0 / (1.0 + np.exp(-lg)) / alpha_min)
    jf2 = ((f * f) * (1.0 + uc * uc)).sum(1) / zs[:, 0] ** 2
    rad = np.sqrt(kappa * (jf2 * np.exp(2.0 * ls.max(1)) + eps)) * 1.02 + 4.0
    past = np.maximum(-centre - rad[:, None], centre - rad[:, None] - (size - 1)).max(1)
    # The footprint's box: half-extents sqrt(kappa Sigma^I_aa).
    qn = q / np.linalg.norm(q, axis=1, keepdims=True)
    w, x, y, zq = qn.T
    Rq = np.stack([1 - 2 * (y * y + zq * zq), 2 * (x * y - w * zq), 2 * (x * zq + w * y),
                   2 * (x * y + w * zq), 1 - 2 * (x * x + zq * zq), 2 * (y * zq - w * x),
                   2 * (x * zq - w * y), 2 * (y * zq + w * x), 1 - 2 * (x * x + y * y)],
                  1).reshape(-1, 3, 3)
    J = np.zeros((len(m), 2, 3))
    J[:, 0, 0], J[:, 1, 1] = f[0] / zs[:, 0], f[1] / zs[:, 0]
    J[:, :, 2] = -f * uc / zs
    A = J @ R @ (Rq * np.exp(ls)[:, None, :])
    half = np.sqrt(kappa[:, None] * (np.einsum("nij,nij->ni", A, A) + eps))
    grid = np.ceil(size / tile) * tile  # a cover's box is listed up to where it leaves [0, grid)
    inside = (centre > 0.5) & (centre < grid - 0.5)
    off = ((centre + half < -REACH) | (centre - half > grid + REACH)).any(1)
    seen = front & inside.all(1) & (past < 0)
    never = ~front | off | (past > 0)
    return seen, (np.abs(past) < NEAR) | (np.abs(z - 0.2) < 1e-3) | ~(seen | never)


@pytest.mark.parametrize("width,height", [(601, 347), (786, 529), (1200, 673)])
def test_counts_of_edge_tiles_follow_the_footprints_radius(width, height):
    n = 400000
    g = _scene(n, width)
    cams = []
    for a in (0.0, 0.3):
        R = np.array([[np.cos(a), 0, np.sin(a)], [0, 1, 0], [-np.sin(a), 0, np.cos(a)]])
        cams.append(synthetic.camera(width, height, 0.6 * width, 0.6 * width, (width - 1) / 2,
                                     (height - 1) / 2, R.astype(np.float32),
                                     np.array([0.05, -0.02, 0.1], np.float32)))
    expect, skip, overhang = np.zeros(n, np.int64), np.zeros(n, bool), 0
    for cam in cams:
        seen, undecided = _decide(g, cam)
        expect += seen
        skip |= undecided
    r = Renderer(0)
    p = [to_dev(g[k]) for k in ("means", "log_scales", "quats", "opacity_logits", "sh")]
    color, _, _, state = r.forward_raw(*p, cams)
    mr = MapRegularizer(r.ctx, p[0])
    r.backward_raw(state, n, 1, len(cams), color, reg=mr.reg(), grad_mask=binding.GRAD_OPACITY)
    counts = mr.obs_count.cpu().numpy()
    r.release(state)
    assert skip.mean() < 0.05 and 0 < expect.sum() < 2 * n
    wrong = np.nonzero(~skip & (counts != expect))[0]
    assert wrong.size == 0, (wrong.size, wrong[:8], counts[wrong[:8]], expect[wrong[:8]])
