"""Contexts of their own in several host threads at once."""
import ctypes
import threading

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


@pytest.mark.parametrize("path", [0, 1, 2])
def test_contexts_with_different_bins(path):
    """Threads whose contexts need different amounts of shared memory in the
    same kernels, launched call by call (no graphs): every call succeeds and
    gives the output of its own context alone."""
    x = synth.wdr_device(96, 130, seed=2, device="cuda")
    bins = (4, 64, 9, 64, 256, 17)
    refs, ys, ctxs, streams = [], [], [], []
    for n in bins:
        ctx = tm.tm_create(tm.make_params(n, [3, 20]))
        tm.tm_set_option(ctx, tm.TM_OPT_HIST_PATH, path)
        tm.tm_set_debug(ctx, True)
        y = torch.empty_like(x)
        tm.tm_forward(ctx, x, y)
        torch.cuda.synchronize()
        refs.append(y.clone())
        ys.append(y.zero_())
        ctxs.append(ctx)
        streams.append(torch.cuda.Stream())
    torch.cuda.synchronize()
    failed = [0] * len(bins)
    forward = tm.lib().tm_forward

    def work(i):
        a, b = tm.image_of(x), tm.image_of(ys[i])
        args = (ctxs[i], ctypes.byref(a), ctypes.byref(b), streams[i].cuda_stream)
        for _ in range(1500):
            failed[i] += forward(*args) != 0

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(bins))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for c in ctxs:
        tm.tm_destroy(c)
    assert failed == [0] * len(bins)
    for y, r in zip(ys, refs):
        assert torch.equal(y, r)
