"""Which histogram path a forward takes, as its stages say, and the batched
passes that the automatic path no longer takes by itself."""
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


def _stages(ctx, call):
    """The stages that `call` reports."""
    tm.tm_set_option(ctx, tm.TM_OPT_STAGE_TIMING, 1)
    tm.tm_stage_times(ctx)
    call()
    names = set(tm.tm_stage_times(ctx))
    tm.tm_set_option(ctx, tm.TM_OPT_STAGE_TIMING, 0)
    return names


def _forward(x, p, path):
    y = torch.empty_like(x)
    ctx = tm.tm_create(p)
    try:
        tm.tm_set_option(ctx, tm.TM_OPT_HIST_PATH, path)
        tm.tm_forward(ctx, x, y)
        torch.cuda.synchronize()
    finally:
        tm.tm_destroy(ctx)
    return y


def _images(sizes, seed):
    return [synth.wdr_device(h, w, seed=seed + i, device="cuda") for i, (w, h) in enumerate(sizes)]


def test_stage_names_say_the_path():
    """One image, and batches with and without an image whose fields are too
    wide for the sweep: the names tell the compact histogram from the others."""
    p = tm.make_params(16, [4, (700, 600)])
    wide, small = _images([(1600, 1200), (300, 200)], 1)
    for path, single, batch in ((0, "compact_histogram", "batch_compact"), (2, "integral_histogram", None),
                                (1, "fused_sweep", None)):
        ctx = tm.tm_create(p)
        try:
            tm.tm_set_option(ctx, tm.TM_OPT_HIST_PATH, path)
            names = _stages(ctx, lambda: tm.tm_forward(ctx, small, torch.empty_like(small)))
            assert names & {"compact_histogram", "integral_histogram", "fused_sweep"} == {single}
            for xs in ([small, small.clone()], [small, wide]):
                if path == 1 and wide is xs[1]:
                    continue  # refused
                ys = [torch.empty_like(x) for x in xs]
                names = _stages(ctx, lambda: tm.tm_forward_batch(ctx, xs, ys))
                if path == 1:
                    assert names == {"batch"}
                else:
                    assert names == {"batch_materialised"} | ({batch} if batch else set())
        finally:
            tm.tm_destroy(ctx)


def test_uneven_batch_on_the_materialised_path():
    """The paper's preset over uneven sizes with the materialised path asked
    for: one batched pass, captured and then replayed, each output that of the
    image's own call."""
    p = tm.tm_params_pyramid(2000, 1500, 5, 5)
    xs = _images([(2000, 1500), (1024, 768), (640, 480), (97, 61)], 300)
    refs = [_forward(x, p, 2) for x in xs]
    ys = [torch.empty_like(x) for x in xs]
    ctx = tm.tm_create(p)
    try:
        tm.tm_set_option(ctx, tm.TM_OPT_HIST_PATH, 2)
        for _ in range(3):
            for y in ys:
                y.zero_()
            assert _stages(ctx, lambda: tm.tm_forward_batch(ctx, xs, ys)) == {"batch_materialised"}
            torch.cuda.synchronize()
            for y, r in zip(ys, refs):
                assert torch.equal(y, r)
    finally:
        tm.tm_destroy(ctx)


def test_batch_splits_over_two_passes():
    """A batch that the compact histogram refuses (an image of 66000 rows) with
    one image whose fields are too wide for the sweep: the automatic path runs
    a sweep pass and a materialised pass, and all images in a materialised pass
    while it measures that, each image equal to its own call."""
    p = tm.make_params(64, [4, (700, 600)])
    xs = _images([(1600, 1200), (300, 1900), (3, 66000), (900, 1500), (1400, 1000)], 400)
    refs = [_forward(x, p, 2) for x in xs]
    ys = [torch.empty_like(x) for x in xs]
    ctx = tm.tm_create(p)
    try:
        for rep in range(10):
            for y in ys:
                y.zero_()
            names = _stages(ctx, lambda: tm.tm_forward_batch(ctx, xs, ys))
            torch.cuda.synchronize()
            assert "batch_compact" not in names and (rep >= 2 or names == {"batch", "batch_materialised"}), names
            for y, r in zip(ys, refs):
                assert torch.equal(y, r)
    finally:
        tm.tm_destroy(ctx)


def _all_but(leave):
    """Device memory held so that about `leave` bytes are free."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")


def _path(ctx, x):
    names = _stages(ctx, lambda: tm.tm_forward(ctx, x, torch.empty_like(x)))
    return names & {"compact_histogram", "integral_histogram", "fused_sweep"}


def test_short_memory_holds_for_what_did_not_fit():
    """The compact histogram of a 12 MP image (1.8 GB) that cannot be had keeps
    neither smaller images from it nor, once there is memory again, the same
    image: after the option is set, or after 256 calls."""
    p = tm.make_params(64, [4, 16])
    big, small = _images([(4000, 3000), (300, 200)], 7)
    for again in ("option", "calls"):
        ctx = tm.tm_create(p)
        hold = None
        try:
            torch.empty_like(big)  # (the caching allocator's block for the outputs)
            hold = _all_but(900 << 20)
            assert _path(ctx, big) == {"fused_sweep"}  # (nor is there memory for the planes)
            assert _path(ctx, small) == {"compact_histogram"}
            hold = None
            torch.cuda.empty_cache()
            if again == "option":
                tm.tm_set_option(ctx, tm.TM_OPT_HIST_PATH, 0)
            else:
                y = torch.empty_like(small)
                for _ in range(256):
                    tm.tm_forward(ctx, small, y)
            assert _path(ctx, big) == {"compact_histogram"}
        finally:
            tm.tm_destroy(ctx)
            hold = None
            torch.cuda.empty_cache()


def test_calls_that_failed_for_memory_have_all_paths_again():
    """A 12 MP image for which no path's memory can be had: the call fails, and
    the next one with memory takes the sweep (the compact histogram is tried
    again later), not whatever path was tried last."""
    p = tm.make_params(64, [4, 16])
    (x,) = _images([(4000, 3000)], 7)
    ctx = tm.tm_create(p)
    hold = None
    try:
        y = torch.empty_like(x)
        hold = _all_but(100 << 20)
        for _ in range(2):
            with pytest.raises(tm.TmError) as e:
                tm.tm_forward(ctx, x, y)
            assert e.value.status == tm.TM_ENOMEM
        hold = None
        torch.cuda.empty_cache()
        assert _path(ctx, x) == {"fused_sweep"}
    finally:
        tm.tm_destroy(ctx)
        hold = None
        torch.cuda.empty_cache()


def test_batch_in_smaller_groups_when_memory_is_short():
    """Sixteen images whose compact histograms (0.9 GB each) would run in two
    groups: with 4 GB free they run one image at a time, the forward and the
    backward's recomputation, and give the same outputs."""
    p = tm.make_params(128, [8, 32])
    xs = [synth.wdr_device(1536, 2048, seed=k, device="cuda") for k in range(16)]
    gs = [torch.randn_like(x) for x in xs]
    got = []
    for short in (False, True):
        ys, gin = [torch.empty_like(x) for x in xs], [torch.empty_like(x) for x in xs]
        gp = torch.empty(7, device="cuda")
        ctx = tm.tm_create(p)
        hold = None
        try:
            if short:
                hold = _all_but(4 << 30)
            for _ in range(2):
                assert "batch_compact" in _stages(ctx, lambda: tm.tm_forward_batch(ctx, xs, ys))
            if not short:
                tm.tm_backward_batch(ctx, xs, gs, gin, gp)
            else:  # (four images: the backward's own workspace takes the rest)
                tm.tm_destroy(ctx)
                ctx = tm.tm_create(p)
                tm.tm_backward_batch(ctx, xs[:4], gs[:4], gin[:4], gp)
            torch.cuda.synchronize()
        finally:
            tm.tm_destroy(ctx)
            del hold
            torch.cuda.empty_cache()
        got.append((ys, gin))
    for a, b in zip(*[g[0] for g in got]):
        assert torch.equal(a, b)
    for a, b in zip(got[0][1][:4], got[1][1][:4]):
        assert torch.equal(a, b)


def _white(h, w, seed):
    """White noise over six decades: every 32-pixel run spans nearly all bins."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return (10.0 ** (torch.rand((h, w, 1), generator=g, device="cuda") * 6 - 2)).expand(h, w, 3).contiguous()


def test_rough_images_take_the_measured_path():
    """White noise at 12 MP and 64 bins runs faster on the sweep: the calls
    settle on it, a photograph of the same size is back on the compact
    histogram after one call, and every output is the forced sweep's."""
    p = tm.make_params(64, [8, 32, 128])
    noise, photo = _white(3000, 4000, 3), synth.wdr_device(3000, 4000, seed=4, device="cuda")
    refs = {id(x): _forward(x, p, 1) for x in (noise, photo)}
    y = torch.empty_like(noise)
    ctx = tm.tm_create(p)

    def run(x, times):
        for _ in range(times):
            y.zero_()
            tm.tm_forward(ctx, x, y)
            torch.cuda.synchronize()
            assert torch.equal(y, refs[id(x)])

    try:
        run(photo, 15)
        assert _path(ctx, photo) == {"compact_histogram"}
        run(noise, 15)
        assert _path(ctx, noise) == {"fused_sweep"}
        run(photo, 1)
        assert _path(ctx, photo) == {"compact_histogram"}
        run(noise, 1)
        assert _path(ctx, noise) == {"fused_sweep"}
    finally:
        tm.tm_destroy(ctx)


def test_rough_backward_equals_the_sweeps():
    """The backward's recomputation on rough images, while it is measured and
    after: the gradients of the forced sweep."""
    p = tm.make_params(64, [4, 16])
    xs = [_white(700, 900, 5), _white(64, 3000, 6)]
    gs = [torch.randn_like(x) for x in xs]
    got = {}
    for path in (1, 0):
        ctx = tm.tm_create(p)
        try:
            tm.tm_set_option(ctx, tm.TM_OPT_HIST_PATH, path)
            for _ in range(1 if path else 12):
                gin, gp = [torch.empty_like(x) for x in xs], torch.empty(7, device="cuda")
                tm.tm_backward_batch(ctx, xs, gs, gin, gp)
                torch.cuda.synchronize()
                got.setdefault(path, gin)
                for a, b in zip(got[1], gin):
                    assert torch.equal(a, b)
        finally:
            tm.tm_destroy(ctx)


def test_long_images_take_the_measured_path():
    """A hundred images of 2048 x 16 with 64 bins run faster on the sweep."""
    p = tm.make_params(64, [4, 16, 64])
    xs = [synth.wdr_device(16, 2048, seed=k % 7, device="cuda") for k in range(100)]
    ys = [torch.empty_like(x) for x in xs]
    refs = [_forward(x, p, 2) for x in xs[:7]]
    ctx = tm.tm_create(p)
    try:
        for _ in range(15):
            for y in ys:
                y.zero_()
            tm.tm_forward_batch(ctx, xs, ys)
            torch.cuda.synchronize()
            for k, y in enumerate(ys):
                assert torch.equal(y, refs[k % 7])
        assert _stages(ctx, lambda: tm.tm_forward_batch(ctx, xs, ys)) == {"batch"}
    finally:
        tm.tm_destroy(ctx)


def test_more_sizes_than_are_kept():
    """Eighty long sizes in turn, each measured anew once it has been replaced."""
    p = tm.make_params(17, [2, (30, 3)])
    xs = [synth.wdr_device(8 + k % 5, 200 + 3 * k, seed=k, device="cuda") for k in range(80)]
    refs = [_forward(x, p, 2) for x in xs]
    ctx = tm.tm_create(p)
    try:
        for _ in range(3):
            for x, r in zip(xs, refs):
                for _ in range(2):
                    y = torch.empty_like(x)
                    tm.tm_forward(ctx, x, y)
                    assert torch.equal(y, r)
    finally:
        tm.tm_destroy(ctx)


def test_short_memory_in_the_backward_passes_too():
    """The backward's recomputation of a 12 MP image without the memory for the
    compact histogram, and 256 calls later with it: the gradients of the sweep."""
    p = tm.make_params(64, [4])
    x, small = _images([(4000, 3000), (300, 200)], 9)
    g, gin, gp = torch.randn_like(x), torch.empty_like(x), torch.empty(5, device="cuda")
    gs, gsin = torch.randn_like(small), torch.empty_like(small)
    got = []
    for path in (1, 0):
        ctx = tm.tm_create(p)
        hold = None
        try:
            tm.tm_set_option(ctx, tm.TM_OPT_HIST_PATH, path)
            if path == 0:
                hold = _all_but(2000 << 20)  # (the backward's own workspace takes 0.8 GB)
            names = _stages(ctx, lambda: tm.tm_backward(ctx, x, g, gin, gp))
            torch.cuda.synchronize()
            assert "fused_sweep" in names
            got.append(gin.clone() if path else gin)
            if path == 0:
                assert torch.equal(*got)
                hold = None
                torch.cuda.empty_cache()
                assert "compact_histogram" in _stages(ctx, lambda: tm.tm_backward(ctx, small, gs, gsin, gp))
                for _ in range(256):
                    tm.tm_backward(ctx, small, gs, gsin, gp)
                assert "compact_histogram" in _stages(ctx, lambda: tm.tm_backward(ctx, x, g, gin, gp))
                torch.cuda.synchronize()
                assert torch.equal(*got)
        finally:
            tm.tm_destroy(ctx)
            hold = None
            torch.cuda.empty_cache()
