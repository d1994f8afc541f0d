"""A state whose reserved cell list is longer than its pair list keeps the pairs in the buffer that
the cell sort leaves free: lists, images and gradients are those of a state without a reserve, for
short and long cell sorts, eagerly and under capture."""
import numpy as np
import pytest
import torch

from paper_2601_00705_gb300 import synthetic
from paper_2601_00705_gb300.render import Renderer

from gpu_common import GRAD_REL_L2, rel_l2, to_dev

pytestmark = pytest.mark.gpu

KEYS = ("means", "log_scales", "quats", "opacity_logits", "sh")


@pytest.mark.parametrize("n,width,height", [(300, 64, 48), (3000, 160, 120), (90000, 640, 480)])
@pytest.mark.parametrize("tile_w,tile_h,ppt", [(16, 16, 4), (8, 8, 2)])
def test_reserved_states_give_the_same_results(n, width, height, tile_w, tile_h, ppt):
    wl = synthetic.tiny(seed=n, n=n, width=width, height=height)
    p = [to_dev(wl.gaussians.as_dict()[k]) for k in KEYS]
    P, tiles = wl.n_pixels, -(-width // tile_w) * -(-height // tile_h)
    up = torch.randn((P, 3), generator=torch.Generator("cuda").manual_seed(1), device="cuda") / P
    r = Renderer(0, tile_w=tile_w, tile_h=tile_h, pixels_per_thread=ppt)
    *ref, plain = r.forward_raw(*p, wl.cameras)
    ref_grads = r.backward_raw(plain, n, 1, 1, up)
    ref_vals, ref_ranges = r.ctx.tile_lists(plain, tiles)
    pairs = r.stats(plain)["n_pairs"]
    state = r.ctx.reserve(0, 4 * pairs, r.stream_handle())
    for capture in (False, True, False):
        out = tuple(torch.zeros_like(x) for x in ref)
        if capture:
            graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
            s.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(s), torch.cuda.graph(graph, stream=s):
                r.forward_raw(*p, wl.cameras, state=state, out=out)
                grads = r.backward_raw(state, n, 1, 1, up)
            torch.cuda.current_stream().wait_stream(s)
            graph.replay()
        else:
            r.forward_raw(*p, wl.cameras, state=state, out=out)
            grads = r.backward_raw(state, n, 1, 1, up)
        torch.cuda.synchronize()
        stats = r.stats(state)
        assert stats["status"] == 0 and stats["pair_capacity"] >= 4 * pairs
        vals, ranges = r.ctx.tile_lists(state, tiles)
        np.testing.assert_array_equal(vals, ref_vals)
        np.testing.assert_array_equal(ranges, ref_ranges)
        for a, b in zip(out, ref):
            assert torch.equal(a, b)
        for k, g in grads.items():
            assert rel_l2(g.cpu().numpy(), ref_grads[k].cpu().numpy()) <= GRAD_REL_L2, k
    r.release(state)
    r.release(plain)


def test_a_backward_after_a_replay_reads_the_replayed_lists():
    # The eager cell sort is short (one cluster), the captured one as long as the reserve.
    n, wl = 3000, synthetic.tiny(seed=9, n=3000, width=320, height=240)
    p = [to_dev(wl.gaussians.as_dict()[k]) for k in KEYS]
    up = torch.randn((wl.n_pixels, 3), generator=torch.Generator("cuda").manual_seed(1),
                     device="cuda") / wl.n_pixels
    for reserve in (60_000, 300_000, 600_000, 2_000_000):
        r = Renderer(0)
        state = r.ctx.reserve(0, reserve, r.stream_handle())
        *out, state = r.forward_raw(*p, wl.cameras, state=state)
        ref = r.backward_raw(state, n, 1, 1, up)
        graph, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(s), torch.cuda.graph(graph, stream=s):
            r.forward_raw(*p, wl.cameras, state=state, out=tuple(out))
        torch.cuda.current_stream().wait_stream(s)
        r.forward_raw(*p, wl.cameras, state=state, out=tuple(out))
        graph.replay()
        torch.cuda.synchronize()
        vals, _ = r.ctx.tile_lists(state, 20 * 15)
        assert r.stats(state)["status"] == 0 and vals.size and vals.max() < n
        grads = r.backward_raw(state, n, 1, 1, up)
        torch.cuda.synchronize()
        for k, g in grads.items():
            assert rel_l2(g.cpu().numpy(), ref[k].cpu().numpy()) <= GRAD_REL_L2, (reserve, k)
        r.release(state)
