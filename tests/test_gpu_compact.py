"""The automatic path's compact integral histogram: Eq. 1 numerators bit-exact
against the oracle and outputs bit-identical to the other paths, at the edges
of its chunks (32 columns), threshold groups (32) and row segments, with the
16- and 32-bit vectors and in several groups of a batch."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2102_01289_gb300 as tm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    tm.build()


def _image(H, W, seed, kind):
    if kind == "scene":
        return synth.wdr_image(H, W, seed=seed)
    rng = np.random.default_rng(seed)  # every chunk holds every bin
    return (10.0 ** rng.uniform(-2, 4, (H, W, 1)) * np.ones(3)).astype(np.float32)


def _forward(img, p, path, debug, out_dtype=torch.float32):
    x = torch.from_numpy(np.ascontiguousarray(img)).cuda()
    y = torch.empty(x.shape, dtype=out_dtype, device="cuda")
    ctx = tm.tm_create(p)
    try:
        tm.tm_set_debug(ctx, debug)
        tm.tm_set_option(ctx, tm.TM_OPT_HIST_PATH, path)
        tm.tm_forward(ctx, x, y)
        cnt = None
        if debug:
            cnt = tm.tm_debug_export(ctx, tm.TM_DBG_COUNTS).cpu().numpy().view(np.uint32)
            cnt = cnt.reshape(p.n_fields, *img.shape[:2])
        torch.cuda.synchronize()
        return y, cnt
    finally:
        tm.tm_destroy(ctx)


# W below, at and above whole chunks; H below and above the 32 row segments;
# K = n - 1 of 1, 4, 5, 31, 32, 33 and 255 thresholds; windows larger than the image
@pytest.mark.parametrize("flags", [0, tm.TM_FLAG_CDF_INCLUSIVE | tm.TM_FLAG_AREA_LITERAL])
@pytest.mark.parametrize("H,W,n,radii,kind", [
    (1, 1, 2, [0], "scene"), (1, 64, 5, [3], "scene"), (37, 31, 6, [2, 40], "scene"),
    (33, 32, 32, [4, 9], "scene"), (31, 33, 33, [1, 5, 16], "noise"), (65, 96, 34, [2, 8, 30], "scene"),
    (130, 161, 64, [8, 32, 128], "noise"), (70, 200, 256, [3, (50, 2)], "noise"),
])
def test_counts_match_oracle(orc, H, W, n, radii, kind, flags):
    img = _image(H, W, 11, kind)
    p = tm.make_params(n, radii, flags=flags)
    op = orc.make_params(n, radii, eps=float(np.float32(0.1)), sat=float(np.float32(0.6)), flags=flags)
    y, cnt = _forward(img, p, 0, True)
    ref, fl = orc.forward(img, op)
    assert np.array_equal(cnt, fl.cnt)
    got = y.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - ref) <= 1e-4 * np.maximum(np.abs(ref), 1e-3))


# windows of at most and more than 65535 / 31 = 2114 rows: 16- and 32-bit vectors
@pytest.mark.parametrize("ry", [1056, 1057, 3000])
@pytest.mark.parametrize("kind", ["scene", "noise"])
def test_tall_windows(ry, kind):
    img = _image(2300, 66, 5, kind)
    p = tm.make_params(12, [(3, ry), (40, 20)])
    y0, c0 = _forward(img, p, 0, True)
    y2, c2 = _forward(img, p, 2, True)
    assert np.array_equal(c0, c2) and torch.equal(y0, y2)
    for dt in (torch.float32, torch.float16, torch.uint8):  # the variants without debug planes
        a, _ = _forward(img, p, 0, False, dt)
        b, _ = _forward(img, p, 2, False, dt)
        assert torch.equal(a, b)


@pytest.mark.parametrize("radii", [[3, 12, 40], [5, (300, 280)]])  # small windows and others
@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
def test_outputs_equal_the_materialised_path(radii, dtype):
    img = synth.wdr_image(300, 411, seed=3, dtype=np.float32 if dtype == torch.float32 else np.float16)
    p = tm.make_params(48, radii)
    for out in (torch.float32, torch.float16, torch.uint8):
        a, _ = _forward(img, p, 0, False, out)
        b, _ = _forward(img, p, 2, False, out)
        assert torch.equal(a, b)


def test_batch_in_several_groups():
    """Six 2048 x 1536 images with 256 bins: the compact integral histograms
    (1.9 GB each) take two groups. Outputs equal the single calls', and the
    backward's count planes (kept, or counted for it) those of the sweep."""
    xs = [synth.wdr_device(1536, 2048, seed=k, device="cuda") for k in range(6)]
    ys = [torch.empty_like(x) for x in xs]
    gs = [torch.randn_like(x) for x in xs]
    p = tm.make_params(256, [8, 32])
    grads = {}
    for path, reuse in ((0, 0), (0, 1), (1, 0)):
        ctx = tm.tm_create(p)
        try:
            tm.tm_set_option(ctx, tm.TM_OPT_HIST_PATH, path)
            tm.tm_set_option(ctx, tm.TM_OPT_BACKWARD_REUSE, reuse)
            gin = [torch.empty_like(x) for x in xs]
            for _ in range(2):
                tm.tm_forward_batch(ctx, xs, ys)
            tm.tm_backward_batch(ctx, xs, gs, gin, torch.empty(7, device="cuda"))
            torch.cuda.synchronize()
            grads[path, reuse] = gin
            if path == 0 and not reuse:
                for x, y in zip(xs, ys):
                    z = torch.empty_like(x)
                    tm.tm_forward(ctx, x, z)
                    assert torch.equal(y, z)
        finally:
            tm.tm_destroy(ctx)
    for a, b, c in zip(grads[0, 0], grads[0, 1], grads[1, 0]):
        assert torch.equal(a, c) and torch.equal(b, c)


def test_batch_of_16_and_32_bit_vectors():
    """One image of the batch has windows taller than the 16-bit vectors
    allow, the others not: the batch takes 32-bit vectors throughout, and every
    output equals the image's own call."""
    p = tm.make_params(24, [(3, 1200), (20, 8)])
    xs = [torch.from_numpy(_image(h, w, 5 + h, "noise")).cuda() for h, w in ((300, 200), (2400, 70), (64, 257))]
    ys = [torch.empty_like(x) for x in xs]
    ctx = tm.tm_create(p)
    try:
        tm.tm_forward_batch(ctx, xs, ys)
        for x, y in zip(xs, ys):
            z = torch.empty_like(x)
            tm.tm_forward(ctx, x, z)
            torch.cuda.synchronize()
            assert torch.equal(y, z)
    finally:
        tm.tm_destroy(ctx)


# both sides of the rule that takes strips to the sweep: one image, and two
@pytest.mark.parametrize("H,W,count", [
    (8, 1024, 1), (8, 1025, 1), (4096, 128, 1), (4097, 128, 1), (4095, 20, 1), (4, 1023, 2), (4, 1024, 2),
])
def test_strips_equal_the_materialised_path(H, W, count):
    p = tm.make_params(33, [2, (40, 3)])
    xs = [torch.from_numpy(_image(H, W, 7 + k, "scene")).cuda() for k in range(count)]
    gs = [torch.ones_like(x) for x in xs]
    got = {}
    for path in (0, 1, 2):
        ys, gin = [torch.empty_like(x) for x in xs], [torch.empty_like(x) for x in xs]
        ctx = tm.tm_create(p)
        try:
            tm.tm_set_option(ctx, tm.TM_OPT_HIST_PATH, path)
            if count == 1:
                tm.tm_forward(ctx, xs[0], ys[0])
            else:
                tm.tm_forward_batch(ctx, xs, ys)
            if path != 2:  # the backward refuses the materialised path
                tm.tm_backward_batch(ctx, xs, gs, gin, torch.empty(7, device="cuda"))
            torch.cuda.synchronize()
            got[path] = ys, gin
        finally:
            tm.tm_destroy(ctx)
    for k in range(count):
        assert torch.equal(got[0][0][k], got[2][0][k])
        assert torch.equal(got[0][1][k], got[1][1][k])


# the largest sums of a launch without small windows: windows of the whole
# image, the luminance at both ends of the range, uneven halves
@pytest.mark.parametrize("H,W,cut", [(513, 700, 350), (3000, 4000, 4000), (3000, 4000, 7), (3001, 3999, 2500)])
def test_large_windows_equal_the_materialised_path(H, W, cut):
    x = synth.wdr_device(H, W, seed=9, device="cuda")
    x[:, :cut] = 1e-3
    x[-1, -1] = 1e4
    p = tm.make_params(6, [(W, H), (W // 2, H // 2), (W // 4, 60), 9])
    got = []
    for path in (0, 2):
        y = torch.empty_like(x)
        ctx = tm.tm_create(p)
        try:
            tm.tm_set_option(ctx, tm.TM_OPT_HIST_PATH, path)
            tm.tm_forward(ctx, x, y)
            torch.cuda.synchronize()
            got.append(y)
        finally:
            tm.tm_destroy(ctx)
    assert torch.equal(got[0], got[1])
