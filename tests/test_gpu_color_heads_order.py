"""A frame with colour heads projects with its own colours: frames at two times in turn, on
buffers that hold the other frame's, are the frames that follow one of the same time."""
import pytest

from paper_2310_08528_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2310_08528_gb300 import fs4d  # noqa: E402


# SH degrees whose rows the projection copies ahead of its geometry (1, 3), and one it reads late
@pytest.mark.parametrize("n,degree", [(3000, 3), (40_000, 1), (40_000, 2), (150_000, 3)])
@pytest.mark.parametrize("prec", [fs4d.BF16, fs4d.FP32])
def test_frames_at_two_times_in_turn(n, degree, prec):
    s = sg.with_color_heads(sg.make_object(7, n=n, mlp_std=0.1, sh_degree=degree), 3, std=0.2)
    cam = sg.hemisphere_cameras(5, width=400, height=300, seed=2)[1]
    ctx = fs4d.Context(0)
    try:
        sid = ctx.load_scene(s)
        want = {}
        for t in (0.1, 0.9):
            for _ in range(2):  # the second frame finds its own colours in the buffers
                want[t] = ctx.render(sid, cam, t, prec)
                torch.cuda.synchronize()
        assert float((want[0.1] - want[0.9]).abs().max()) > 1e-2
        for _ in range(10):
            for t in (0.1, 0.9):
                assert torch.equal(ctx.render(sid, cam, t, prec), want[t])
    finally:
        ctx.close()
