"""The checks of the forced paths (test_gpu_forward) and of the compact counts
(test_gpu_compact) on the automatic path: sizes, settings and group edges that
they leave out."""
import pytest

import synth  # noqa: F401

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2102_01289_gb300 as tm  # noqa: E402
import test_gpu_compact as compact  # noqa: E402
import test_gpu_forward as forward  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    tm.build()


@pytest.mark.parametrize("H,W,n,radii,seed", forward.CASES)
def test_forward_matches_oracle(orc, H, W, n, radii, seed):
    forward.test_forward_matches_oracle(orc, H, W, n, radii, seed, 0)


def test_degenerate_images(orc):
    forward.test_degenerate_images(orc, 0)


def test_full_size_12mp_every_count(orc):
    forward.test_full_size_12mp_every_count(orc, 0)


def test_paper_preset_matches_oracle(orc):
    forward.test_paper_preset_matches_oracle(orc, 0)


@pytest.mark.parametrize("flags", forward.FLAG_SETS)
def test_reading_variants_match_oracle(orc, flags):
    forward.test_reading_variants_match_oracle(orc, flags, 0)


def test_streaming_range_reuse(orc):
    forward.test_streaming_range_reuse(orc, 0)


@pytest.mark.parametrize("flags", [0, tm.TM_FLAG_CDF_INCLUSIVE | tm.TM_FLAG_AREA_LITERAL])
def test_eight_fields_and_maximum_radius(orc, flags):
    forward.test_eight_fields_and_maximum_radius(orc, flags, 0)


def test_large_image_64bit_offsets_sampled(orc):
    forward.test_large_image_64bit_offsets_sampled(orc, 0)


# n - 1 thresholds at the edges of the group sizes 4, 8, 16, 32 and 64: the
# last that fills a group, the first of the next size, and (past 64) one that
# leaves a single threshold in its group
@pytest.mark.parametrize("n", [5, 6, 9, 10, 17, 18, 33, 34, 65, 66, 67, 129, 130, 193, 194])
@pytest.mark.parametrize("H,W", [(40, 95), (33, 96), (97, 33)])
@pytest.mark.parametrize("flags", [0, tm.TM_FLAG_CDF_INCLUSIVE])
def test_threshold_groups_match_oracle(orc, H, W, n, flags):
    compact.test_counts_match_oracle(orc, H, W, n, [1, (12, 5), 40], "noise", flags)


def test_vectors_past_32_bit_indices():
    """8192 x 8192 of white noise with 96 bins: 200 M vector slots of 32 columns,
    6.4 G entries (12.8 GB); outputs equal to the sweep's."""
    if torch.cuda.mem_get_info()[0] < 60 * 2 ** 30:
        pytest.skip("needs 60 GB of device memory")
    g = torch.Generator(device="cuda")
    g.manual_seed(8)
    x = (10.0 ** (torch.rand((8192, 8192, 1), generator=g, device="cuda") * 6 - 2)).expand(8192, 8192, 3).contiguous()
    p = tm.make_params(96, [3, (70, 40)])
    got = []
    for path in (0, 1):  # (a first call is taken by the rules, whatever its content)
        y = torch.empty_like(x)
        ctx = tm.tm_create(p)
        try:
            tm.tm_set_option(ctx, tm.TM_OPT_HIST_PATH, path)
            tm.tm_set_option(ctx, tm.TM_OPT_STAGE_TIMING, 1)
            tm.tm_forward(ctx, x, y)
            assert ("compact_histogram" in tm.tm_stage_times(ctx)) == (path == 0)
        finally:
            tm.tm_destroy(ctx)
        got.append(y)
    assert torch.equal(*got)
