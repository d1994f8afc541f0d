"""The per-Gaussian backward at the edges of its warps and blocks: scene sizes around multiples of
32 and 128, every SH degree, warps without a visible Gaussian among mixed ones. Gradients match
the oracle, those of unseen Gaussians are exactly zero, and nothing is written past the arrays."""
import numpy as np
import pytest
import torch

import oracle
from paper_2601_00705_gb300 import synthetic

from gpu_common import GRAD_REL_L2, gpu_forward, masked_l1_upstream, rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,degree", [(1, 3), (31, 2), (32, 0), (33, 3), (127, 1), (129, 3),
                                      (130, 2), (401, 0), (401, 1), (401, 3)])
def test_ragged_sizes_and_unseen_gaussians(n, degree):
    rng = np.random.default_rng(100 * n + degree)
    K = (degree + 1) ** 2
    whole = synthetic.tiny(seed=5, n=max(n, 2)).gaussians.as_dict()
    g = {k: v[:n].copy() for k, v in whole.items()}
    rest = 0.2 * rng.standard_normal((n, K - 1, 3))
    g["sh"] = np.concatenate([g["sh"], rest], 1).astype(np.float32)
    g["log_scales"] += 1.0
    unseen = np.arange(n) % 5 == 2
    unseen[128:256] = True  # whole warps
    g["means"][unseen, 2] = -3.0
    cams = [synthetic.camera(w, 61, 70.0, 70.0, (w - 1) / 2, 30.0, np.eye(3), np.zeros(3))
            for w in (75, 40)]
    orc0 = oracle.render(g, cams)
    d_color, _ = masked_l1_upstream(orc0, rng.random(orc0["color"].shape))
    orc = oracle.render(g, cams, d_color=d_color)
    r, *_, state = gpu_forward(g, cams)
    shapes = dict(means=(n, 3), log_scales=(n, 3), quats=(n, 4), opacity_logits=(n,),
                  sh=(n, K, 3), pose=(2, 6))
    whole = {k: torch.full((int(np.prod(s)) + 256,), float("nan"), device="cuda")
             for k, s in shapes.items()}
    grads = {k: whole[k][:int(np.prod(s))].view(s) for k, s in shapes.items()}
    r.backward_raw(state, n, K, 2, to_dev(d_color), out=grads)
    torch.cuda.synchronize()
    r.release(state)
    for k, s in shapes.items():
        a = grads[k].cpu().numpy().astype(np.float64)
        assert rel_l2(a, orc["g_" + k]) <= GRAD_REL_L2, k
        if k != "pose":
            assert not a[unseen].any(), k
        assert torch.isnan(whole[k][int(np.prod(s)):]).all(), k
