"""A frame queued right behind a training step renders with the step's weights: it is the frame
that the same call gives once everything has finished."""
import pytest

from paper_2310_08528_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2310_08528_gb300 import fs4d  # noqa: E402


@pytest.mark.parametrize("prec", [fs4d.FP32, fs4d.BF16])
@pytest.mark.parametrize("n", [500, 30_000])
def test_frame_right_behind_a_training_step(n, prec):
    s = sg.make_object(11, n=n, mlp_std=0.1)
    cam = sg.hemisphere_cameras(5, width=240, height=180, seed=1)[3]
    ctx = fs4d.Context(0)
    try:
        sid = ctx.load_scene(s)
        target = torch.zeros(cam.height, cam.width, 3, device="cuda")
        trainer = fs4d.Trainer(ctx, sid, 100, lr_mlp=(1e-2, 1e-2))
        last = ctx.render(sid, cam, 0.4, prec)
        for _ in range(5):
            torch.cuda.synchronize()
            trainer.step(cam, 0.4, target, prec)
            behind = ctx.render(sid, cam, 0.4, prec)
            torch.cuda.synchronize()
            after = ctx.render(sid, cam, 0.4, prec)
            assert torch.equal(behind, after) and not torch.equal(after, last)
            last = after
        trainer.close()
    finally:
        ctx.close()
