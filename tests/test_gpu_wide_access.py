"""The elementwise and loss kernels that take four elements per access, where that can go wrong:
sizes that are no multiple of four, views that start anywhere in the concatenated images, arrays
that are not 16-byte aligned. Against the oracles (tolerances of test_gpu_tracking.py and
test_gpu_mapping.py) or exactly."""
import numpy as np
import pytest
import torch

from oracle import mapping as omap
from oracle import tracking as otrack
from paper_2601_00705_gb300 import binding, synthetic
from gpu_common import renderer

pytestmark = pytest.mark.gpu


def _dev(a, shift):
    """`a` on the device, `shift` elements past a 256-byte boundary."""
    buf = torch.empty(a.size + 64, dtype=torch.from_numpy(a).dtype, device="cuda")
    t = buf[shift:shift + a.size]
    t.copy_(torch.from_numpy(np.ascontiguousarray(a)).reshape(-1))
    return t


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("fit", [0, 1])
@pytest.mark.parametrize("sizes", [[(1, 1)], [(3, 1), (2, 1), (5, 3)], [(37, 23), (64, 48), (1, 2)],
                                   [(333, 251), (128, 2)]])
def test_track_loss_of_any_layout(sizes, fit, shift):
    rng = np.random.default_rng(len(sizes) + shift)
    cams = [synthetic.camera(w, h, 50.0, 50.0, w / 2, h / 2, np.eye(3), np.zeros(3))
            for w, h in sizes]
    P = sum(w * h for w, h in sizes)
    f32 = lambda *s: rng.random(s).astype(np.float32)  # noqa: E731
    color, alpha, obs, wg = f32(P, 3), f32(P), f32(P, 3), f32(P)
    r = renderer()
    c, a, o, w = (_dev(x, shift) for x in (color, alpha, obs, wg))
    d = _dev(np.zeros(3 * P, np.float32), shift)
    loss = torch.full((len(sizes),), 7.0, dtype=torch.float64, device="cuda")
    gb = torch.empty((len(sizes), 2), device="cuda")
    r.ctx.track_loss(cams, binding.default_track_config(fit_exposure=fit), c.data_ptr(),
                     a.data_ptr(), o.data_ptr(), w.data_ptr(), d.data_ptr(), loss.data_ptr(),
                     gb.data_ptr(), r.stream_handle())
    torch.cuda.synchronize()
    f64 = lambda x: x.astype(np.float64)  # noqa: E731
    ref, d_ref, gb_ref = otrack.track_loss(f64(color), f64(alpha), f64(obs), f64(wg), cams, 0.5,
                                           fit_exposure=bool(fit))
    first = 0
    for v, (wd, h) in enumerate(sizes):
        px = slice(first, first + wd * h)
        first += wd * h
        # The fit divides differences of sums of FP32 partial sums (about 16 units of roundoff).
        x = f64(color[px]).ravel()
        amp = x.size * (x @ x) / max(x.size * (x @ x) - x.sum() ** 2, 1e-30)
        tol = (16 * 2.0 ** -24 * amp if fit else 0.0) * (1.0 + np.abs(gb_ref[v]).max()) + 1e-7
        np.testing.assert_allclose(gb.cpu().numpy()[v], gb_ref[v], rtol=0, atol=tol)
        np.testing.assert_allclose(loss.cpu().numpy()[v], ref[v], rtol=1e-5, atol=6 * tol * x.size)
        res = f64(obs[px]) - (gb_ref[v][0] * f64(color[px]) + gb_ref[v][1])
        sure = np.abs(res) > 1e-5 + 2 * tol  # the gradient is the residual's sign
        got = d.cpu().numpy().reshape(P, 3)[px]
        np.testing.assert_allclose(got[sure], d_ref[px][sure], rtol=1e-5, atol=tol)


@pytest.mark.parametrize("shift", [0, 1, 4])
@pytest.mark.parametrize("n", [1, 3, 4, 1023, 100001])
def test_upkeep_of_any_alignment(n, shift):
    rng = np.random.default_rng(n)
    f32 = lambda *s: rng.normal(-1.0, 2.0, s).astype(np.float32)  # noqa: E731
    means, ema, ls, lg = f32(n, 3), f32(n, 3), f32(n, 3), f32(n)
    obs = rng.integers(0, 10, n).astype(np.int32)
    vis = rng.uniform(0, 3, n).astype(np.float32)
    r = renderer()
    s = r.stream_handle()
    m, e = _dev(means, shift), _dev(ema, shift)
    r.ctx.map_ema(n, m.data_ptr(), e.data_ptr(), 0.25, s)
    arrays = [_dev(x, shift) for x in (ls, lg, obs, vis)]
    keep = _dev(np.full(n, 9, np.uint8), shift)
    count = torch.full((1,), 77, dtype=torch.int32, device="cuda")
    r.ctx.prune_mask(n, *[x.data_ptr() for x in arrays], binding.default_prune_config(),
                     keep.data_ptr(), count.data_ptr(), s)
    a, b = rng.random((3, n)).astype(np.float32), rng.random((3, n)).astype(np.float32)
    ad, bd = _dev(a, shift), _dev(b, shift)
    counts = torch.empty((3, 2), dtype=torch.int64, device="cuda")
    iou = torch.empty(3, device="cuda")
    r.ctx.covisibility(ad.data_ptr(), bd.data_ptr(), n, 3, 0.25, counts.data_ptr(),
                       iou.data_ptr(), s)
    torch.cuda.synchronize()
    np.testing.assert_allclose(e.cpu().numpy().reshape(n, 3), omap.ema(means, ema, 0.25), rtol=0,
                               atol=1e-6)
    # Every FP32 decision is far from its bound: alpha within 1e-5 of it, or the trace, is left out.
    ref = omap.prune_mask(ls, lg, obs, vis, min_opacity=np.float32(0.005), max_trace=1.0,
                          min_observations=5, min_visibility=1.0)
    alpha = 1.0 / (1.0 + np.exp(-lg.astype(np.float64)))
    trace = np.exp(2.0 * ls.astype(np.float64)).sum(1)
    sure = (np.abs(alpha - 0.005) > 1e-6) & (np.abs(trace - 1.0) > 1e-5)
    got = keep.cpu().numpy()
    np.testing.assert_array_equal(got[sure], ref[sure])
    assert int(count.item()) == int(got.sum()) and set(np.unique(got)) <= {0, 1}
    inter, union, ref_iou = otrack.covisibility(a, b, np.float32(0.25))
    np.testing.assert_array_equal(counts.cpu().numpy(), np.stack([inter, union], 1))
    np.testing.assert_array_equal(iou.cpu().numpy(), ref_iou.astype(np.float32))


@pytest.mark.parametrize("V", [1, 5, 6, 11, 64])
def test_pose_steps_of_any_number_of_views_and_rotation(V):
    # Rates up to 2 rad per step cross from the series to sin and cos.
    rng = np.random.default_rng(V)
    T = np.tile(np.eye(3, 4), (V, 1, 1)) + 0.0
    T[:, :, 3] = rng.normal(size=(V, 3))
    T = T.astype(np.float32)
    grad = (rng.normal(size=(V, 6)) * 10.0 ** rng.integers(-5, 2, size=(V, 1))).astype(np.float32)
    r = renderer()
    f32 = lambda x: float(np.float32(x))  # noqa: E731
    for lr, k in ((1e-3, 0), (0.25, 7), (2.0, 30)):
        pose = torch.from_numpy(T.reshape(V, 12).copy()).cuda()
        m = (0.01 * rng.normal(size=(V, 6)) * (k > 0)).astype(np.float32)
        v = (0.01 * rng.random((V, 6)) * (k > 0)).astype(np.float32)
        state = torch.from_numpy(np.concatenate([m, v], 1)).cuda()
        step = torch.tensor([k], dtype=torch.int32, device="cuda")
        g = torch.from_numpy(grad).cuda()
        r.ctx.pose_adam_step(V, binding.default_adam_config(lr=lr, iterations=60), g.data_ptr(),
                             state.data_ptr(), step.data_ptr(), pose.data_ptr(),
                             r.stream_handle())
        torch.cuda.synchronize()
        Tn, mn, vn, _ = otrack.adam_pose_step(T.astype(np.float64), grad.astype(np.float64),
                                              m.astype(np.float64), v.astype(np.float64), k,
                                              lr=f32(lr), beta1=f32(0.9), beta2=f32(0.999),
                                              eps=f32(1e-8), iterations=60)
        np.testing.assert_allclose(pose.cpu().numpy().reshape(V, 3, 4), Tn, rtol=0, atol=1e-6 * (
            1 + np.abs(Tn).max()))
        st = state.cpu().numpy()
        np.testing.assert_allclose(st[:, :6], mn, rtol=1e-6, atol=1e-12)
        np.testing.assert_allclose(st[:, 6:], vn, rtol=1e-6, atol=1e-18)
        assert int(step.item()) == k + 1
