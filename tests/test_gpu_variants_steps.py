"""Variants of a stage that are chosen by size, beyond their second step; sizes that depend on the
number of SMs.  (test_gpu_variants.py has the smaller ones.)"""
import numpy as np
import pytest

from paper_2310_08528_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2310_08528_gb300 import fs4d  # noqa: E402

import oracle  # noqa: E402
import test_gpu_backward as views  # noqa: E402


# A step of a directly composited tile is 131072 ranks, a queue 2048 of its list.  Faint Gaussians,
# so that no tile is saturated in its first step.
@pytest.mark.parametrize("n,w,h,scale", [(140_000, 64, 48, -3.0), (131_073, 33, 100, -4.0), (270_000, 48, 48, -3.5)])
def test_direct_frame_of_several_steps_equals_listed_frame(n, w, h, scale):
    s = sg.make_object(9, n=n, log_scale_mean=scale, mlp_std=0.1)
    s.opacity_logits = np.full(n, -9.0, np.float32)
    s.opacity_logits[::5000] = -5.0  # (above 1/255: these blend)
    s.opacity_logits[1::97] = -5.4
    cam = sg.hemisphere_cameras(5, width=w, height=h, seed=3)[2]
    ctx = fs4d.Context(0)
    try:
        sid = ctx.load_scene(s)
        want = ctx.render(sid, cam, 0.3, with_aux=True)
        assert int(want[2].max()) > 2048 and float(want[1].min()) > 1e-3
        ctx.set_band_pairs(ctx.last_pairs() - 1)
        got = ctx.render(sid, cam, 0.3, with_aux=True)
        assert ctx.last_bands() >= 2
        first = 16  # (the first band, a row of tiles or more, has the whole frame's principal point)
        for a, b in zip(got, want):
            assert torch.equal(a[:first], b[:first])
        assert float((got[0] - want[0]).abs().max()) < 2e-2
        assert torch.equal(ctx.render(sid, cam, 0.3), got[0])
    finally:
        ctx.close()


@pytest.mark.parametrize("per_sm,more", [(64, 0), (64, 1), (128, 5)])
def test_fp32_deform_tiles_agree_at_this_device(per_sm, more):
    """Tiles of 32 and of 128 Gaussians, at the size where the one gives way to the other on this
    device's number of SMs."""
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + more
    s = sg.make_object(4, n=2 * n + 3000, res_spatial=(8, 12), res_time=5, mlp_std=0.2)
    part = s.copy()
    for k in ("means", "log_scales", "quats", "opacity_logits", "sh"):
        setattr(part, k, np.ascontiguousarray(getattr(s, k)[:n]))
    ctx = fs4d.Context(0)
    try:
        a = ctx.deform(ctx.load_scene(s), [0.37], fs4d.FP32)
        b = ctx.deform(ctx.load_scene(part), [0.37], fs4d.FP32)
        for x, y in zip(a, b):
            assert torch.equal(x[:, :n], y)
    finally:
        ctx.close()


# three levels are two blocks of 64 inputs of the first layer (32 features) or one of 48 (16);
# 300 Gaussians are two whole tiles of the delta chain and a ragged one, 513 one chunk of the
# weight sums and one more
@pytest.mark.parametrize("h,n", [(16, 300), (32, 300), (32, 513)])
def test_backward_of_three_levels_matches_oracle(h, n):
    s = sg.make_object(23, n=n, res_spatial=(5, 7, 9), res_time=4, h=h, mlp_std=0.12)
    s.means *= 0.8
    s.log_scales += 1.0
    cam = views.small_camera()
    dl = views.masked_dl(s, cam, 0.4, 5)
    ctx = fs4d.Context(0)
    try:
        _, g = views.gpu_grads(ctx, s, cam, 0.4, dl)
    finally:
        ctx.close()
    views.check_groups(g, oracle.render_backward(s, cam, 0.4, dl, plane_terms=True))
