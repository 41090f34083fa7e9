"""Integral histogram planes (Eq. 7-8) at the edges of the kernel's strips (128
columns), passes (1024 columns), row batches (32) and segments (64 rows)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2102_01289_gb300 as tm  # noqa: E402


@pytest.fixture(scope="module", autouse=True)
def _built():
    tm.build()


@pytest.mark.parametrize("H,W,n", [(1, 1, 1), (33, 31, 5), (64, 128, 2), (65, 129, 7), (130, 1024, 3), (97, 1025, 6),
                                   (31, 2100, 256), (200, 3073, 4), (263000, 3, 2)])
def test_planes_exact(H, W, n):
    g = torch.Generator(device="cuda")
    g.manual_seed(H + W)
    bins = torch.randint(0, n, (H, W), generator=g, device="cuda", dtype=torch.int32).to(torch.uint8)
    bins[: H // 2, : W // 2] = n - 1  # a uniform part
    hk = torch.empty((n, H + 1, W + 1), dtype=torch.int32, device="cuda")
    hk.fill_(-1)
    tm.tm_integral_histogram(bins, n, hk)
    for k in range(n):
        ref = torch.nn.functional.pad((bins == k).to(torch.int32).cumsum(0).cumsum(1), (1, 0, 1, 0))
        assert torch.equal(hk[k], ref.to(torch.int32)), k


@pytest.mark.parametrize("H,W", [(1, 1), (37, 1025), (612, 700), (1220, 1000), (1300, 1000), (2500, 1100), (5000, 40)])
def test_integral_images_exact_at_every_segment_length(H, W):
    """Row segments of 4, 8 and 16 rows (few, some and many tiles), one and two
    column chunks: the integral images of q and q^2 against int64 sums."""
    g = torch.Generator(device="cuda")
    g.manual_seed(H)
    q = torch.randint(-(1 << 23), (1 << 23) + 1, (H, W), generator=g, device="cuda", dtype=torch.int32)
    q[: H // 3] = 1 << 23
    s1 = torch.full((H + 1, W + 1), -1, dtype=torch.int64, device="cuda")
    s2 = torch.full_like(s1, -1)
    tm.tm_integral_image(q, s1, s2)
    v = q.to(torch.int64)
    assert torch.equal(s1, torch.nn.functional.pad(v.cumsum(0).cumsum(1), (1, 0, 1, 0)))
    assert torch.equal(s2, torch.nn.functional.pad((v * v).cumsum(0).cumsum(1), (1, 0, 1, 0)))
