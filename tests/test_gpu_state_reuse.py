"""Released states are reused by the forwards that create a state: whatever ran on the memory
before (another size, another tile shape, a forward without its backward), on whatever stream,
the results equal those of a context that never released one."""
import pytest
import torch

from paper_2601_00705_gb300 import binding, synthetic
from paper_2601_00705_gb300.render import Renderer

from gpu_common import GRAD_REL_L2, rel_l2, to_dev

pytestmark = pytest.mark.gpu

KEYS = ("means", "log_scales", "quats", "opacity_logits", "sh")


def _load(n, width, height, seed):
    wl = synthetic.tiny(seed=seed, n=n, width=width, height=height)
    g = wl.gaussians.as_dict()
    gen = torch.Generator(device="cuda").manual_seed(seed)
    up = torch.randn((wl.n_pixels, 3), generator=gen, device="cuda") / wl.n_pixels
    return [to_dev(g[k]) for k in KEYS], wl.cameras, up


def _step(r, load, backward=True):
    p, cams, up = load
    *img, state = r.forward_raw(*p, cams)
    grads = r.backward_raw(state, p[0].shape[0], 1, 1, up) if backward else {}
    return state, img, grads


def test_reused_states_give_a_fresh_contexts_results():
    loads = [_load(n, w, h, s) for s, (n, w, h) in enumerate(
        [(3000, 160, 120), (1, 17, 1), (3000, 160, 120), (9001, 333, 251), (500, 64, 48)])]
    r = Renderer(0)
    sizes = []
    for backward in (True, False, True):
        for load in loads:
            state, img, grads = _step(r, load, backward)
            sizes.append(r.stats(state)["state_bytes"])
            r.release(state)
            fresh = Renderer(0)
            ref_state, ref_img, ref_grads = _step(fresh, load, backward)
            torch.cuda.synchronize()
            for a, b in zip(img, ref_img):
                assert torch.equal(a, b)
            for k in grads:
                assert rel_l2(grads[k].cpu().numpy(), ref_grads[k].cpu().numpy()) <= GRAD_REL_L2, k
            fresh.release(ref_state)
    # From the second round on a spare state holds every size: nothing grows any more.
    assert max(sizes[len(loads):]) == max(sizes[:len(loads)])


def test_a_state_released_while_its_work_is_queued_is_safe_on_another_stream():
    a, b = _load(3000, 160, 120, 1), _load(2500, 150, 100, 2)
    r = Renderer(0)
    refs = []
    for load in (a, b):
        state, img, _ = _step(Renderer(0), load, False)
        refs.append([x.clone() for x in img])
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    warm, *_ = _step(r, a, False)
    torch.cuda.synchronize()
    torch.cuda._sleep(20_000_000)  # the first forward is still queued when the second begins
    first, img_a, _ = _step(r, a, False)
    r.release(first)
    with torch.cuda.stream(side):
        second, img_b, _ = _step(r, b, False)
    torch.cuda.synchronize()
    for got, ref in zip((img_a, img_b), refs):
        for x, y in zip(got, ref):
            assert torch.equal(x, y)
    r.release(warm)
    r.release(second)


def test_a_state_used_under_capture_is_freed_and_handles_end_with_their_release():
    load = _load(2000, 160, 120, 3)
    p, cams, up = load
    r = Renderer(0)
    imgs = tuple(torch.empty(s, device="cuda") for s in ((160 * 120, 3), (160 * 120,), (160 * 120,)))
    *_, state = r.forward_raw(*p, cams, out=imgs)
    graph = torch.cuda.CUDAGraph()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s), torch.cuda.graph(graph, stream=s):
        r.forward_raw(*p, cams, state=state, out=imgs)
    torch.cuda.current_stream().wait_stream(s)
    graph.replay()
    r.release(state)
    other, img, _ = _step(r, load, False)
    torch.cuda.synchronize()
    for x, y in zip(img, imgs):
        assert torch.equal(x, y)
    r.release(other)
    for h in (state, other):
        with pytest.raises(binding.RGSError) as e:
            r.release(h)
        assert e.value.status == binding.RGS_ERR_STATE
