"""Edges of tm_merge_exposures: infinite exposure times, and concurrent calls
with different numbers of exposures."""
import ctypes
import math
import threading

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


def test_concurrent_calls_with_different_counts():
    """Host threads that merge five and eight exposures at once, calling the
    library with prepared arguments so that the calls overlap: eight need more
    than the default 48 KB of shared memory, whatever the other calls need."""
    rng = np.random.default_rng(0)
    g = np.ascontiguousarray(synth.camera_log_response(), dtype=np.float32)
    ldr = [torch.from_numpy(rng.integers(0, 256, size=(8, 8, 3)).astype(np.uint8)).cuda() for _ in range(8)]
    ptrs = (ctypes.c_void_p * 8)(*[a.data_ptr() for a in ldr])
    times = (ctypes.c_float * 8)(*[2.0 ** -k for k in range(8)])
    merge = tm.lib().tm_merge_exposures
    counts = (5, 8, 6, 8, 5, 8)
    outs = [torch.empty((8, 8, 3), device="cuda") for _ in counts]
    torch.cuda.synchronize()
    failed = [0] * len(counts)

    def work(i):
        out = tm.image_of(outs[i])
        args = (counts[i], ctypes.cast(ptrs, ctypes.c_void_p), ctypes.cast(times, ctypes.c_void_p), 8, 8, 24,
                g.ctypes.data_as(ctypes.c_void_p), ctypes.byref(out), torch.cuda.Stream().cuda_stream)
        for _ in range(20000):
            failed[i] += merge(*args) != 0

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(counts))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert failed == [0] * len(counts)
