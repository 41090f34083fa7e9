"""Edges of tm_merge_exposures: infinite exposure times."""
import math

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


@pytest.mark.parametrize("n", [2, 4, 5])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float16])
def test_infinite_exposure_time(n, dtype):
    """An exposure time of +inf has ln E = -inf wherever it has a weight, so
    E = 0 there, four pixels at a time and one at a time alike."""
    rng = np.random.default_rng(n)
    H, W = 12, 40
    ldr = [torch.from_numpy(rng.integers(1, 255, size=(H, W, 3)).astype(np.uint8)).cuda() for _ in range(n)]
    times = [1.0 / (j + 1) for j in range(n - 1)] + [math.inf]
    out = torch.full((H, W, 3), 7.0, dtype=dtype, device="cuda")
    tm.tm_merge_exposures(ldr, times, synth.camera_log_response(), out)
    torch.cuda.synchronize()
    assert torch.equal(out, torch.zeros_like(out))
