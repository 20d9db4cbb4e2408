"""Variants of a stage that are chosen by size give the same bits.  Frames composited
straight from the depth order: columns and rows of tiles as bits per depth rank.  A frame
whose pairs exceed a band goes that way; its first band has the whole frame's principal
point, so its pixels are the listed tiles' bit for bit, with full lists (the last
contributors are list positions)."""
import numpy as np
import pytest

from paper_2310_08528_gb300 import scenegen as sg

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2310_08528_gb300 import fs4d  # noqa: E402


# 32768 ranks are one step of a tile, 4096 of its list one queue, 1024 ranks one CTA of the bit rows
@pytest.mark.parametrize("n,w,h,scale", [(33, 48, 40, -2.0), (1023, 130, 120, -2.5), (1025, 1100, 64, -3.0),
                                         (6000, 64, 64, -1.0), (33000, 333, 211, -3.0)])
def test_direct_frame_equals_listed_frame(n, w, h, scale):
    s = sg.make_object(9, n=n, log_scale_mean=scale, mlp_std=0.1)
    cam = sg.hemisphere_cameras(5, width=w, height=h, seed=3)[2]
    ctx = fs4d.Context(0)
    try:
        sid = ctx.load_scene(s)
        want = ctx.render(sid, cam, 0.3, with_aux=True)
        k = ctx.last_pairs()
        assert ctx.last_bands() == 1
        ctx.set_band_pairs(k - 1)
        rows = (h + 15) // 16
        for _ in range(2):  # cut into bands, then with the bands of the frame before
            got = ctx.render(sid, cam, 0.3, with_aux=True)
            bands = ctx.last_bands()
            assert bands >= 2
            first = 16 * (rows // 4)  # at most four bands at half the limit each: the first holds these rows
            for a, b in zip(got, want):
                assert torch.equal(a[:first], b[:first])
                assert np.isfinite(a.float().cpu().numpy()).all()
            # a row's principal point is rounded differently in the other bands
            far = (got[0] - want[0]).abs().amax(-1) > 2e-2
            assert int(far.sum()) <= 1e-3 * w * h
        plain = ctx.render(sid, cam, 0.3)
        assert torch.equal(plain, got[0])
    finally:
        ctx.close()


@pytest.mark.parametrize("n", [1, 31, 33, 64 * 152, 64 * 152 + 1, 128 * 152 + 5])
@pytest.mark.parametrize("levels", [1, 2, 3])
def test_fp32_deform_tiles_agree(n, levels):
    """Tiles of 32 and of 128 Gaussians give the same sums in the same order: a scene's first
    Gaussians deform alike, bit for bit, alone and within a larger set."""
    res = (8, 12, 16)[:levels]
    s = sg.make_object(4, n=40000, res_spatial=res, res_time=5, mlp_std=0.2)
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


# up to 131072 Gaussians a tile's words stay in registers
@pytest.mark.parametrize("n,tx,ty,side", [(131072, 50, 41, 3), (131073, 7, 300, 2), (393217, 33, 9, 2),
                                          (700, 40, 30, 30), (3000, 700, 1, 40)])
def test_lists_equal_sorted_pairs(n, tx, ty, side):
    """Tile lists from column and row bits are the radix-sorted pairs: keys, values, ranges, count."""
    g = torch.Generator(device="cuda").manual_seed(n)
    lo = torch.stack([torch.randint(0, t, (n,), generator=g, device="cuda") for t in (tx, ty)], 1)
    size = torch.randint(0, side + 1, (n, 2), generator=g, device="cuda")  # (0: no tiles)
    hi = torch.minimum(lo + size, torch.tensor([tx, ty], device="cuda"))
    rect = torch.cat([lo, hi], 1).int().contiguous()
    depth = (torch.rand(n, generator=g, device="cuda") * 4).round(decimals=3).contiguous()  # with ties
    cap = int((hi - lo).prod(1).sum())
    ctx = fs4d.Context(0)
    try:
        ctx.set_binning(fs4d.BINNING_SORT)
        want = [v.clone() if torch.is_tensor(v) else v for v in ctx.bin_sort(depth, rect, tx, ty, cap)]
        ctx.set_binning(fs4d.BINNING_AUTO)
        got = ctx.bin_sort(depth, rect, tx, ty, cap)
        assert ctx.last_binning() == fs4d.BINNING_BITMAP
        assert got[3] == want[3] == cap
        for a, b in zip(got[:3], want[:3]):
            assert torch.equal(a, b)
        with pytest.raises(fs4d.Fs4dError):
            ctx.bin_sort(depth, rect, tx, ty, cap - 1)
    finally:
        ctx.close()


@pytest.mark.parametrize("thin", [1.0, 30.0, 1000.0])
def test_block_masks_miss_no_pixel(thin):
    """One Gaussian per tile, round to a thousand times longer than wide, its mean within a few
    of its sizes of the tile: every pixel whose alpha passes the threshold in 64 bits is
    blended, with that alpha, as far as float32 can tell: each term of the exponent is three
    roundings (offset, product, sum) from its value twice over, so the exponent in powers of
    two is within 10 2^-24 of the sum of its terms' magnitudes."""
    tiles = 48
    n = tiles * tiles
    rng = np.random.default_rng(int(thin))
    long, wide = np.exp(rng.uniform(0, 3, n)) * thin ** 0.5 + 0.55, rng.uniform(0.55, 3, n)
    th, k, ph = rng.uniform(0, np.pi, n), rng.uniform(0, 3.3, n), rng.uniform(0, 2 * np.pi, n)
    c, s = np.cos(th), np.sin(th)
    u, v = k * long * np.cos(ph), k * wide * np.sin(ph)
    t = np.arange(n)
    xy = np.stack([t % tiles * 16 + 8 + u * c - v * s, t // tiles * 16 + 8 + u * s + v * c], 1).astype(np.float32)
    a, b, d = [x.astype(np.float32) for x in ((c / long) ** 2 + (s / wide) ** 2, c * s * (long ** -2.0 - wide ** -2.0),
                                             (s / long) ** 2 + (c / wide) ** 2)]
    op = rng.uniform(0.02, 0.98, n).astype(np.float32)
    co = np.stack([a, b, d, op], 1)
    dev = lambda z: torch.from_numpy(np.ascontiguousarray(z)).cuda()  # noqa: E731
    ranges = np.stack([t, t + 1], 1).astype(np.int32)
    ctx = fs4d.Context(0)
    try:
        img, _, _ = ctx.composite(16 * tiles, 16 * tiles, dev(ranges), dev(t.astype(np.int32)), dev(xy), dev(co),
                                  dev(np.ones((n, 3), np.float32)))
        got = img[..., 0].cpu().numpy().reshape(tiles, 16, tiles, 16).transpose(0, 2, 1, 3).reshape(n, 16, 16)
    finally:
        ctx.close()
    px = np.arange(16) + 0.5
    dx = (xy[:, 0].astype(np.float64) - t % tiles * 16)[:, None, None] - px[None, None, :]
    dy = (xy[:, 1].astype(np.float64) - t // tiles * 16)[:, None, None] - px[None, :, None]
    A, B, C, O = [co[:, i].astype(np.float64)[:, None, None] for i in range(4)]
    alpha = np.minimum(0.99, O * np.exp(-0.5 * (A * dx * dx + 2 * B * dx * dy + C * dy * dy)))
    e = 10 * 2.0 ** -24 * 0.7213475 * (A * dx * dx + 2 * np.abs(B * dx * dy) + C * dy * dy) + 1e-6
    need = alpha * 2.0 ** -e > 1 / 255
    assert need.sum() > n / 2
    assert (np.abs(got - alpha)[need] <= (alpha * (2.0 ** e - 1) + 1e-6)[need]).all()


# depths by bucket (at most 1024 in one), a full bucket (radix sort after all), out of the buckets' range
@pytest.mark.parametrize("n,lo,hi", [(1, 1.0, 1.0), (1000, 2.0, 2.0), (1024, 3.0, 3.0), (1025, 3.0, 3.0),
                                     (100000, 2.0, 5.0), (100000, 4.0, 4.01), (60000, 1e-4, 3e3), (5000, -2.0, 2.0),
                                     (20000, 1e-4, 3e3), (24576, 2.0, 5.0), (24577, 2.0, 5.0)])
def test_depth_order_by_buckets(n, lo, hi):
    """(depth bits, index) order of the Gaussians with tiles, whatever the depths: bin_sort with
    lists against the sorted pairs."""
    g = torch.Generator(device="cuda").manual_seed(n)
    depth = lo + (hi - lo) * torch.rand(n, generator=g, device="cuda")
    if n < 10000:
        depth[::3] = float(depth[0])  # ties (more than a bucket holds, with 5000)
    x = torch.randint(0, 9, (n, 1), generator=g, device="cuda")
    size = torch.randint(0, 3, (n, 1), generator=g, device="cuda")
    rect = torch.cat([x, x, torch.clamp(x + size, max=9), torch.clamp(x + size, max=9)], 1).int().contiguous()
    cap = int(((rect[:, 2] - rect[:, 0]) * (rect[:, 3] - rect[:, 1])).sum())
    ctx = fs4d.Context(0)
    try:
        ctx.set_binning(fs4d.BINNING_SORT)
        want = [v.clone() if torch.is_tensor(v) else v for v in ctx.bin_sort(depth, rect, 9, 9, cap)]
        ctx.set_binning(fs4d.BINNING_AUTO)
        got = ctx.bin_sort(depth, rect, 9, 9, cap)
        assert got[3] == want[3] == cap
        for a, b in zip(got[:3], want[:3]):
            assert torch.equal(a, b)
    finally:
        ctx.close()


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 8, 255, 256, 257, 259, 513, 1100])
def test_composite_list_lengths(n):
    """Lists that end anywhere in a step of the walk, a batch or after saturation (from about 300
    terms): sums in float64.  Every term is far above 1/255, so only the cut at T < 1e-4 can fall
    on the other side: it moves less than 0.08 * 1e-4.  Rounding of 600 terms' products: 1e-4."""
    g = torch.Generator(device="cuda").manual_seed(n)
    w, h = 27, 15  # a whole tile and a ragged one
    xy = (torch.rand(n, 2, generator=g, device="cuda") * torch.tensor([27.0, 15.0], device="cuda")).contiguous()
    conic = torch.tensor([1e-3, 2e-4, 2e-3], device="cuda").repeat(n, 1)
    opac = 0.03 + 0.05 * torch.rand(n, 1, generator=g, device="cuda")
    co = torch.cat([conic, opac], 1).contiguous()
    rgb = torch.rand(n, 3, generator=g, device="cuda")
    half = (n + 1) // 2
    values = torch.cat([torch.arange(n), torch.arange(half)]).int().cuda()
    ranges = torch.tensor([[0, n], [n, n + half]], dtype=torch.int32, device="cuda")
    ctx = fs4d.Context(0)
    try:
        img, t_final, last = [v.cpu() for v in ctx.composite(w, h, ranges, values, xy, co, rgb)]
    finally:
        ctx.close()
    p, c, col = xy.double().cpu(), co.double().cpu(), rgb.double().cpu()
    yy, xx = torch.meshgrid(torch.arange(h) + 0.5, torch.arange(w) + 0.5, indexing="ij")
    dx, dy = p[:, 0, None, None] - xx, p[:, 1, None, None] - yy
    al = c[:, 3, None, None] * torch.exp(-0.5 * (1e-3 * dx * dx + 2 * 2e-4 * dx * dy + 2e-3 * dy * dy))
    assert float(al.min()) > 2 / 255
    al[half:, :, 16:] = 0  # the second tile's list is the first half
    T = torch.cumprod(1 - al, 0)
    before = torch.cat([torch.ones(1, h, w, dtype=torch.float64), T[:-1]])
    live = T >= 1e-4
    want = torch.einsum("nhw,nc->hwc", al * before * live, col)
    assert float((img - want).abs().max()) < 1e-4 + 0.08 * 1e-4
    count = torch.minimum(live.sum(0), torch.tensor([n] * 16 + [half] * 11))
    assert int((last - count).abs().max()) <= 1
    if n < 100:
        assert torch.equal(last.long(), count)
    assert float((t_final / T.gather(0, (last.long() - 1)[None])[0] - 1).abs().max()) < 1e-4
