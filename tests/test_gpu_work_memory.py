"""Work memory that calls of several kinds and sizes share: what one call sized is enough for
the next, whatever came before it."""
import numpy as np
import pytest

from paper_2310_08528_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2310_08528_gb300 import fs4d  # noqa: E402


@pytest.fixture()
def ctx():
    c = fs4d.Context(0)
    yield c
    c.close()


def long_row(ctx, n, tiles):
    """A bin_sort of n Gaussians over one row of tiles."""
    depth = torch.linspace(1, 2, n, device="cuda")
    x = (torch.arange(n, device="cuda") * (tiles // n)).int()
    rect = torch.stack([x, 0 * x, x + 1, 0 * x + 1], 1).contiguous()
    _, vals, _, k = ctx.bin_sort(depth, rect, tiles, 1, n)
    assert k == n and torch.equal(vals, torch.arange(n, device="cuda", dtype=torch.int32))


@pytest.mark.parametrize("tiles", [6000, 100_000])
def test_async_frame_after_a_long_row_of_tiles(ctx, tiles):
    """bin_sort sizes the tiles' buffers for a grid that is no image (without length classes); a
    larger frame than the reserved one then has its lists by another route, with the same image."""
    s = sg.make_object(3, n=3000, mlp_std=0.1)
    cam = sg.hemisphere_cameras(5, width=1200, height=1200, seed=3)[1]
    sid = ctx.load_scene(s)
    other = fs4d.Context(0)
    try:
        want = other.render(other.load_scene(s), cam, 0.3)
        pairs = other.last_pairs()
    finally:
        other.close()
    long_row(ctx, 1000, tiles)
    ctx.reserve(sid, 64, 64, 2 * pairs)
    d_cam = torch.from_numpy(np.frombuffer(bytes(fs4d.camera_struct(cam)), np.float32).copy()).cuda()
    image = torch.empty(1200, 1200, 3, device="cuda")
    ctx.render_async(sid, cam, d_cam, torch.tensor([0.3], device="cuda"), image)
    assert ctx.last_binning() == fs4d.BINNING_SORT
    torch.cuda.synchronize()
    assert torch.equal(image, want)
    ctx.check_device_status()


def test_sizes_of_different_calls_do_not_multiply(ctx):
    """Bit rows are sized for one call's tiles and Gaussians: many tiles with few Gaussians (128 MB
    of bits) and many Gaussians with few tiles (1.3 MB) take no product of the two (25 GB)."""
    s = sg.make_object(5, n=200_000, mlp_std=0.1)
    cam = sg.hemisphere_cameras(5, width=300, height=200, seed=3)[2]
    sid = ctx.load_scene(s)
    want = ctx.render(sid, cam, 0.6)
    for _ in range(2):
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        long_row(ctx, 1000, 1_000_000)
        assert torch.equal(ctx.render(sid, cam, 0.6), want)
        torch.cuda.synchronize()
        assert free - torch.cuda.mem_get_info()[0] < 2 << 30
    ctx.unload_scene(sid)
    fresh = fs4d.Context(0)  # the other order
    try:
        long_row(fresh, 1000, 1_000_000)
        free = torch.cuda.mem_get_info()[0]
        assert torch.equal(fresh.render(fresh.load_scene(s), cam, 0.6), want)
        assert free - torch.cuda.mem_get_info()[0] < 2 << 30
    finally:
        fresh.close()


@pytest.mark.parametrize("before", [False, True])
def test_a_failed_allocation_leaves_a_working_context(ctx, before):
    """A capacity beyond the device's memory is refused, and the buffers that made room for it are
    allocated again by the next call (before: the context has rendered already)."""
    s = sg.make_object(6, n=5000, mlp_std=0.1)
    cam = sg.hemisphere_cameras(5, width=300, height=200, seed=3)[2]
    sid = ctx.load_scene(s)
    if before:
        want = ctx.render(sid, cam, 0.6)
    with pytest.raises(fs4d.Fs4dError):
        ctx.reserve(sid, 300, 200, 40_000_000_000)
    got = ctx.render(sid, cam, 0.6)
    image, frame = ctx.render_saved(sid, cam, 0.6)
    ctx.render_backward(frame, torch.ones_like(image), {"means": torch.zeros(s.n, 3, device="cuda")})
    ctx.frame_free(frame)
    assert torch.equal(got, image)
    if before:
        assert torch.equal(got, want)
    ctx.check_device_status()


def test_set_stream_within_a_capture(ctx):
    """A context that keeps freed frames may be given another stream inside a capture."""
    s = sg.make_object(6, n=3000, mlp_std=0.1)
    cam = sg.hemisphere_cameras(5, width=160, height=120, seed=3)[2]
    sid = ctx.load_scene(s)
    want, frame = ctx.render_saved(sid, cam, 0.6)
    ctx.reserve(sid, 160, 120, 2 * ctx.last_pairs())
    d_cam = torch.from_numpy(np.frombuffer(bytes(fs4d.camera_struct(cam)), np.float32).copy()).cuda()
    d_t, image = torch.tensor([0.6], device="cuda"), torch.zeros(120, 160, 3, device="cuda")
    ctx.frame_free(frame)
    torch.cuda.synchronize()
    before, graph = ctx.stream, torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        ctx.set_stream(torch.cuda.current_stream())
        ctx.render_async(sid, cam, d_cam, d_t, image)
    ctx.set_stream(before)
    graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(image, want)
    # frames kept from before the other stream are not taken over, and the next ones are right
    for _ in range(3):
        again, frame = ctx.render_saved(sid, cam, 0.6)
        assert torch.equal(again, want)
        ctx.frame_free(frame)


def test_saved_frames_on_two_streams(ctx):
    """Frames rendered on one stream, used and freed on another."""
    s = sg.make_object(8, n=20_000, mlp_std=0.1)
    cam = sg.hemisphere_cameras(5, width=320, height=240, seed=3)[2]
    sid = ctx.load_scene(s)
    dl = torch.ones(240, 320, 3, device="cuda")

    def grads(frame):
        g = {"sh": torch.zeros(s.sh.shape, device="cuda"), "opacity_logits": torch.zeros(s.n, device="cuda")}
        torch.cuda.synchronize()
        ctx.render_backward(frame, dl, g)
        return g

    image, frame = ctx.render_saved(sid, cam, 0.2)
    want = grads(frame)
    torch.cuda.synchronize()
    ctx.frame_free(frame)
    first, side = ctx.stream, torch.cuda.Stream()
    for k in range(6):
        got, frame = ctx.render_saved(sid, cam, 0.2)
        torch.cuda.synchronize()
        ctx.set_stream(side if ctx.stream is first else first)
        g = grads(frame)
        if k % 2:
            ctx.frame_free(frame)
        torch.cuda.synchronize()
        if not k % 2:
            ctx.frame_free(frame)
        assert torch.equal(got, image)
        for n, v in g.items():  # (the order among warps is free)
            assert float((v - want[n]).abs().max()) <= 1e-5 * float(want[n].abs().max())
    ctx.set_stream(first)


def test_kept_frames_make_room(ctx):
    """What frame_free keeps is given back when the context would run out of memory: with 48 MB of
    the device left beside two kept frames of 500,000 Gaussians (66 MB each), a scene of 75 MB is
    loaded."""
    big = sg.make_object(9, n=500_000, log_scale_mean=-7.0)
    sid = ctx.load_scene(big)
    cam = sg.hemisphere_cameras(5, width=64, height=64, seed=3)[2]
    frames = [ctx.render_saved(sid, cam, 0.5)[1] for _ in range(2)]
    torch.cuda.synchronize()
    for f in frames:
        ctx.frame_free(f)
    part = big.copy()
    for k in ("means", "log_scales", "quats", "opacity_logits", "sh"):
        setattr(part, k, np.ascontiguousarray(getattr(big, k)[:300_000]))
    hogs = []
    try:
        left = torch.cuda.mem_get_info()[0] - (48 << 20)
        while left > 0:  # pieces that the device has free ranges for
            try:
                hogs.append(torch.empty(left, dtype=torch.uint8, device="cuda"))
            except torch.OutOfMemoryError:
                hogs.append(torch.empty(left // 2, dtype=torch.uint8, device="cuda"))
            left = torch.cuda.mem_get_info()[0] - (48 << 20)
        other = ctx.load_scene(part)
        assert ctx.read_scene(other)["means"].shape == part.means.shape
    finally:
        hogs.clear()
        torch.cuda.empty_cache()


def view_gradients(ctx, sid, s, cam, t):
    image, frame = ctx.render_saved(sid, cam, t)
    g = {k: torch.zeros(np.shape(getattr(s, k)), device="cuda") for k in fs4d.PARAMS}
    ctx.render_backward(frame, torch.ones_like(image), g)
    ctx.frame_free(frame)
    return image, g


@pytest.mark.parametrize("modes", [(fs4d.BINNING_AUTO,), (fs4d.BINNING_SORT,), (fs4d.BINNING_AUTO, fs4d.BINNING_SORT)])
def test_saved_frames_of_changing_size(ctx, modes):
    """Frames that take over the buffers of frames of other sizes, scenes and binnings, growing
    past their lists' capacity and shrinking again, are those of a context that has rendered
    nothing yet."""
    scenes = [sg.make_object(12, n=900, mlp_std=0.1), sg.make_object(13, n=15_000, log_scale_mean=-3.0, mlp_std=0.1)]
    ids = [ctx.load_scene(s) for s in scenes]
    turns = [(0, 64, 48), (1, 300, 200), (0, 500, 300), (1, 120, 500), (1, 640, 480), (0, 33, 17), (1, 300, 200)]
    for k, (which, w, h) in enumerate(turns):
        mode = modes[k % len(modes)]
        cam = sg.hemisphere_cameras(5, width=w, height=h, seed=4)[k % 5]
        fresh = fs4d.Context(0)
        try:
            fresh.set_binning(mode)
            want, wg = view_gradients(fresh, fresh.load_scene(scenes[which]), scenes[which], cam, 0.3)
        finally:
            fresh.close()
        ctx.set_binning(mode)
        got, gg = view_gradients(ctx, ids[which], scenes[which], cam, 0.3)
        assert torch.equal(got, want)
        for n, v in wg.items():  # (the order among warps, and of a plane cell's terms, is free)
            scale = float(v.abs().max())
            assert float((gg[n] - v).abs().max()) <= 1e-4 * scale, (k, n)
    ctx.check_device_status()


def test_saved_frames_hold_what_their_lists_need(ctx):
    """After a generous reservation a saved frame holds its own list, not the reserved one."""
    s = sg.make_object(14, n=10_000, mlp_std=0.1)
    cam = sg.hemisphere_cameras(5, width=200, height=150, seed=4)[1]
    sid = ctx.load_scene(s)
    ctx.reserve(sid, 200, 150, 100_000_000)
    view_gradients(ctx, sid, s, cam, 0.3)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    frames = [ctx.render_saved(sid, cam, 0.1 * k)[1] for k in range(4)]
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] < 4 * (32 << 20)  # (their lists at the reservation: 400 MB each)
    for f in frames:
        ctx.frame_free(f)


@pytest.mark.parametrize("n,w,h,ppg", [(1_000_000, 800, 600, 10.0), (600_000, 1920, 1080, 4.0)])
def test_scene_bytes_are_what_a_frame_allocates(ctx, n, w, h, ppg):
    """The per-frame figure that admission goes by, against the device memory that a reservation
    of that size takes (allocations come in 2 MB, fewer than 40 of them)."""
    sid = ctx.load_scene(sg.make_object(15, n=n, log_scale_mean=-7.0))
    _, per_frame = ctx.scene_bytes(sid, w, h, ppg)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ctx.reserve(sid, w, h, int(ppg * n) + 4096)
    used = free - torch.cuda.mem_get_info()[0]
    want = per_frame - w * h * 12  # (the image is the caller's)
    assert want <= used <= want + 40 * (2 << 20)


def test_bin_sort_allocates_no_frame(ctx):
    """A context's first bin_sort takes the depth order, the lists and the bit rows (48 bytes per
    Gaussian and pair, 10 MB of bits), none of a frame's 140 bytes per Gaussian and 20 per pair."""
    n = 1_000_000
    depth = torch.rand(n, device="cuda") + 1
    x = (torch.arange(n, device="cuda") % 40).int()
    y = (torch.arange(n, device="cuda") // 40 % 40).int()
    rect = torch.stack([x, y, x + 1, y + 1], 1).contiguous()
    ctx.bin_sort(depth[:1], rect[:1].contiguous(), 40, 40, 1)  # (the modules are loaded)
    warm = ctx.bin_sort(depth, rect, 40, 40, n)
    torch.cuda.synchronize()
    other = fs4d.Context(0)
    try:
        free = torch.cuda.mem_get_info()[0]
        got = other.bin_sort(depth, rect, 40, 40, n)
        assert other.last_binning() == fs4d.BINNING_BITMAP
        torch.cuda.synchronize()
        assert free - torch.cuda.mem_get_info()[0] < 120 << 20  # (12 bytes per pair of them torch's)
        assert all(torch.equal(a, b) for a, b in zip(got[:3], warm[:3]))
    finally:
        other.close()
