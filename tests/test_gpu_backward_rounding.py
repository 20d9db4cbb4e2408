"""The backward's products and their sums within a warp are rounded as they always were.

Adam's first steps take the sign of a gradient alone, so a gradient that is as exact but
rounded in another way sends the elements whose sum cancels the other way.  The values in
golden/backward_bits.json are the float32 gradients of a small frame as the library gave
them at commit f798696 in every one of 40 runs.  The order in which warps add to a term's
sum is free, so each Gaussian here has two pixels in a tile, or all of them in one warp:
its sums have one value.  They are compared bit for bit."""
import json
import os

import numpy as np
import pytest

from paper_2310_08528_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2310_08528_gb300 import fs4d  # noqa: E402

GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "backward_bits.json")
GROUPS = ("means", "log_scales", "quats", "opacity_logits", "sh")  # (planes and mlp sum over all Gaussians)


def scene():
    """64 faint Gaussians, many of them on top of one another: round ones that reach two pixels
    of a tile at most (0.7 pixels around the mean), and level ones, 0.46 pixels high and several
    wide, which lie within one row."""
    s = sg.make_tiny(21, n=64, mlp_std=0.02)
    rng = np.random.default_rng(5)
    s.means = (s.means * np.float32(0.25)).astype(np.float32)
    s.log_scales = rng.normal(-5.0, 0.2, s.log_scales.shape).astype(np.float32)
    s.log_scales[32:, 0] += np.float32(3.7)
    s.quats[32:] = np.float32([1, 0, 0, 0]) + rng.normal(0, 0.01, (32, 4)).astype(np.float32)
    op = rng.uniform(0.0045, 0.0085, s.opacity_logits.shape)
    op[32:] = rng.uniform(0.0045, 0.0054, 32)
    s.opacity_logits = np.log(op / (1 - op)).astype(np.float32)
    return s, sg.tiny_camera(64, 48)


def gradients():
    s, cam = scene()
    dl = torch.from_numpy(np.random.default_rng(6).normal(size=(cam.height, cam.width, 3)).astype(np.float32)).cuda()
    ctx = fs4d.Context(0)
    try:
        _, frame = ctx.render_saved(ctx.load_scene(s), cam, 0.4, fs4d.FP32)
        grads = {k: torch.zeros(np.shape(getattr(s, k)), device="cuda") for k in fs4d.PARAMS}
        ctx.render_backward(frame, dl, grads)
        ctx.frame_free(frame)
        return {k: grads[k].cpu().numpy().ravel().view(np.uint32) for k in GROUPS}
    finally:
        ctx.close()


def record(path, runs=40):
    """Writes the values of the library in use, null where its runs differ."""
    all_runs = [gradients() for _ in range(runs)]
    out = {k: [int(v) if all(int(r[k][i]) == int(v) for r in all_runs) else None for i, v in enumerate(all_runs[0][k])]
           for k in GROUPS}
    with open(path, "w") as f:
        f.write("{\n" + ",\n".join('"%s": %s' % (k, json.dumps(v, separators=(",", ":"))) for k, v in out.items()) + "\n}\n")


def test_gradient_bits():
    with open(GOLDEN) as f:
        want = json.load(f)
    got = gradients()
    for k in GROUPS:
        at = [i for i, v in enumerate(want[k]) if v is not None]
        assert len(at) == len(want[k])
        bad = [i for i in at if int(got[k][i]) != want[k][i]]
        assert not bad, f"{k}: {len(bad)} of {len(at)} elements rounded otherwise"
