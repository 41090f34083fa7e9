"""Integral histogram planes whose segments are divided into parts (long rows
with few planes and segments): passes of 1024 columns, strips of 128, segments
of 64 rows, more and fewer than 32 segments, both kinds of planes."""
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


@pytest.mark.parametrize("H,W,n", [
    (1, 1025, 1), (1, 100000, 2), (63, 2048, 1), (64, 2049, 2), (65, 3000, 5), (64, 16384, 5), (200, 5121, 3),
    (2048, 2200, 2), (2112, 1153, 1), (2150, 4097, 2), (300, 1100, 200), (37, 9999, 256),
])
def test_parts_exact(H, W, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(H + W)
    bins = torch.randint(0, n, (H, W), generator=g, device="cuda", dtype=torch.int32).to(torch.uint8)
    bins[H // 2:, W // 3: W // 2] = n - 1  # a uniform part, over strip and segment edges
    hk = torch.full((n, H + 1, W + 1), -1, dtype=torch.int32, device="cuda")
    tm.tm_integral_histogram(bins, n, hk)
    for k in range(n):
        ref = torch.nn.functional.pad((bins == k).to(torch.int32).cumsum(0).cumsum(1), (1, 0, 1, 0))
        assert torch.equal(hk[k], ref.to(torch.int32)), k


@pytest.mark.parametrize("H,W,n", [(40, 5000, 3), (130, 3000, 2), (2100, 1030, 2), (64, 9000, 17)])
def test_cumulative_planes_in_parts(H, W, n):
    """The materialised path's planes: outputs equal to the sweep's."""
    x = synth.wdr_device(H, W, seed=H, device="cuda")
    p = tm.make_params(n, [3, (40, 9)])
    got = []
    for path in (1, 2):
        y = torch.empty_like(x)
        ctx = tm.tm_create(p)
        try:
            tm.tm_set_option(ctx, tm.TM_OPT_HIST_PATH, path)
            tm.tm_forward(ctx, x, y)
            torch.cuda.synchronize()
        finally:
            tm.tm_destroy(ctx)
        got.append(y)
    assert torch.equal(*got)


@pytest.mark.parametrize("H,W", [(1, 2 ** 31 - 1), (2 ** 31 - 1, 1), (2 ** 21, 1025)])
def test_sides_up_to_the_largest(H, W):
    """Maps of 2^31 pixels, one row, one column and two passes: two planes."""
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < 120 * 2 ** 30:
        pytest.skip("needs 120 GB of device memory")
    bins = torch.zeros((H, W), dtype=torch.uint8, device="cuda")
    bins.view(-1)[::3] = 1
    hk = torch.full((2, H + 1, W + 1), -1, dtype=torch.int32, device="cuda")
    tm.tm_integral_histogram(bins, 2, hk)
    assert int(hk[:, 0].abs().max()) == 0 and int(hk[:, :, 0].abs().max()) == 0
    row = min(H, 5)  # the first rows, and the last row: (entries are modulo 2^32)
    ones = (bins[:row] == 1).to(torch.int64).cumsum(1).cumsum(0)
    assert torch.equal(hk[1, 1:row + 1, 1:].to(torch.int64), ones)
    del ones
    cols = torch.zeros(W, dtype=torch.int64, device="cuda")
    for part in bins.split(1 << 18):
        cols += (part == 1).sum(0)
    assert torch.equal(hk[1, H, 1:].to(torch.int64) & 0xffffffff, cols.cumsum(0))
    area = torch.arange(1, W + 1, dtype=torch.int64, device="cuda") * H
    assert torch.equal((hk[0, H, 1:].to(torch.int64) + hk[1, H, 1:].to(torch.int64)) & 0xffffffff, area & 0xffffffff)


def test_long_rows_use_the_whole_chip():
    """Five planes of 16384 x 64 (1 Mi pixels) take less than four times as long
    as five planes of 1024 x 1024: one block per plane takes ten times as long."""
    times = {}
    for H, W in ((1024, 1024), (64, 16384)):
        bins = torch.randint(0, 5, (H, W), device="cuda", dtype=torch.uint8)
        hk = torch.empty((5, H + 1, W + 1), dtype=torch.int32, device="cuda")
        for _ in range(5):
            tm.tm_integral_histogram(bins, 5, hk)
        best = 1e9
        for _ in range(5):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                tm.tm_integral_histogram(bins, 5, hk)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) / 20)
        times[W] = best
    assert times[16384] < 4 * times[1024], times
