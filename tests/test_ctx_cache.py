"""The contexts that the autograd function keeps per parameter vector."""
import threading

import pytest

import paper_2102_01289_gb300 as tm

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module", autouse=True)
def _built():
    tm.build()


def _theta(p, **at):
    t = tm.params_tensor(p)
    for k, v in at.items():
        t[int(k[1:])] = v
    return t


def test_a_context_per_distinct_value():
    """Every float32 value of the parameters has its own context, however small
    the difference; the same values in another precision share one."""
    p = tm.make_params(8, [2, 5])
    cache = tm._CtxCache(p)
    try:
        a = cache.get(_theta(p, i3=1e-10, i4=1e-10))
        b = cache.get(_theta(p, i3=3e-10, i4=1e-10))
        assert a.value != b.value
        assert cache.get(_theta(p, i3=1e-10, i4=1e-10)).value == a.value
        assert cache.get(_theta(p, i3=3e-10, i4=1e-10).double()).value == b.value
        assert cache.get(_theta(p, i3=3e-10, i4=1e-10)[None].requires_grad_(True)).value == b.value  # any shape
        assert cache.get(_theta(p, i2=0.6)).value != cache.get(_theta(p, i2=0.6 + 2.0 ** -24)).value
    finally:
        cache.close()


def test_contexts_are_bounded(monkeypatch):
    """Parameters that change at every step leave `limit` contexts, the most
    recently used; the others are destroyed, one still referenced elsewhere
    with its last reference, and close destroys the rest."""
    destroyed = []
    real = tm.tm_destroy

    def record(ctx):
        destroyed.append(ctx.value)
        real(ctx)

    monkeypatch.setattr(tm, "tm_destroy", record)
    p = tm.make_params(8, [2, 5])
    cache = tm._CtxCache(p)
    first = cache.get(_theta(p, i2=0.5))
    handle = first.value
    held = cache.get(_theta(p, i2=0.25))
    for k in range(3 * cache.limit):
        cache.get(_theta(p, i3=0.1 + k))
        assert cache.get(_theta(p, i2=0.5)).value == handle  # used again: stays
        assert len(cache.ctxs) <= cache.limit
    assert len(destroyed) == 2 * cache.limit + 1 and handle not in destroyed and held.value not in destroyed
    old = held.value
    del held
    assert destroyed[-1] == old
    cache.close()
    assert handle in destroyed and first.value is None and not cache.ctxs
    del first
    assert len(destroyed) == 3 * cache.limit + 2  # each context once


def test_threads_get_their_own_contexts():
    """Threads with parameters of their own, more of them than the cache keeps:
    each context holds the values it was asked for while it is in use."""
    p = tm.make_params(8, [2, 5])
    cache = tm._CtxCache(p)
    bad = []

    def work(k):
        for i in range(50):
            c = cache.get(_theta(p, i3=0.1 * (k + 1)))
            if not c.value or tm.lib().tm_last_launch_count(c) != 0:
                bad.append(k)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(2 * cache.limit)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    cache.close()
    assert not bad


@pytest.mark.gpu
def test_small_parameters_reach_the_operator():
    """eps of 1e-10 and 3e-10 through the autograd function: each output and
    gradient is that of a context created with those values."""
    if not torch.cuda.is_available():  # pragma: no cover
        pytest.skip("no CUDA device")
    torch.manual_seed(0)
    x = (1.0 + 1e-4 * torch.randn(40, 60, 3)).cuda()
    x[0, 0], x[-1, -1] = 1e4, 1e-4  # both sides of the middle edge; variances of the normalised log near 1e-10
    g = torch.randn_like(x)
    p = tm.make_params(8, [1, 6])
    cache = tm._CtxCache(p)
    outs = []
    try:
        for eps in (1e-10, 3e-10):
            theta = _theta(p, i3=eps, i4=1e-10).requires_grad_(True)
            xi = x.clone().requires_grad_(True)
            y = tm.TMFunction.apply(xi, theta, cache)
            gx, gp = torch.autograd.grad(y, (xi, theta), g)
            ctx = tm.tm_create(tm.params_from_tensor(p, theta))
            ref, rgx, rgp = torch.empty_like(x), torch.empty_like(x), torch.empty(7, device="cuda")
            tm.tm_forward(ctx, x, ref)
            tm.tm_backward(ctx, x, g, rgx, rgp)
            torch.cuda.synchronize()
            tm.tm_destroy(ctx)
            assert torch.equal(y, ref) and torch.equal(gx, rgx)
            # (sums over the blocks in an order that varies from run to run)
            assert torch.allclose(gp, rgp.cpu(), rtol=1e-4, atol=1e-4 * float(rgp.abs().max()))
            outs.append(y.detach())
    finally:
        cache.close()
    assert not torch.equal(outs[0], outs[1])
