"""Two host threads with plans of their own, of very different shared-memory needs, each on its own stream:
every call succeeds and gives the results of a lone call."""
import threading

import numpy as np
import pytest

from gpuhelp import to_dev
from paper_1310_7114_gb300 import build, itc

pytestmark = pytest.mark.gpu
CALLS = 1500


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    itc.lib()


def _plan(n, shape, M, params, seed, ndim=2):
    rng = np.random.default_rng(seed)
    if ndim == 2:
        ims = [(rng.random(shape) < 0.4).astype(np.uint8) for _ in range(min(n, 2))]
        W = [np.floor(rng.random((M, 2)) * shape).astype(np.float32) for _ in range(n)]
    else:
        ims = [rng.integers(0, 8, shape).astype(np.uint8) for _ in range(min(n, 2))]
        W = [np.floor(rng.random((M, 3)) * [*shape, 8]).astype(np.float32) for _ in range(n)]
    ts = [to_dev(im) for im in ims]
    plan = itc.Plan([ts[b % len(ts)] for b in range(n)], [M] * n, params, ndims=[ndim] * n, Gs=[8 if ndim == 3 else 1] * n)
    return plan, plan.pack_W(W)


def _cases(kind):
    """(plan, codebooks) of the small and of the large thread, and one call's function of both."""
    p = itc.make_params(2.0, 3.0, 0)
    if kind == "recursive":
        rec = itc.make_params(12.0, 3.0, 0, flags=itc.ITC_RECURSIVE)
        return _plan(1, (40, 40), 4, rec, 1), _plan(1, (16, 2048), 4, rec, 2)
    if kind == "iterate":
        return _plan(160, (24, 24), 800, p, 1), _plan(160, (24, 24), 2048, p, 2)
    if kind == "fields_3d":
        return (_plan(1, (40, 40), 4, itc.make_params((1.0, 1.0, 1.0), 3.0, 0), 1, 3),
                _plan(1, (40, 40), 4, itc.make_params((7.0, 7.0, 1.0), 3.0, 0), 2, 3))
    if kind == "fields":
        return _plan(1, (40, 40), 4, itc.make_params(5.6, 3.0, 0), 1), _plan(1, (40, 40), 4, itc.make_params(10.0, 3.0, 0), 2)
    nd = 3 if kind == "backward_3d" else 2
    p = itc.make_params((2.0,) * nd, 3.0, 0)
    return _plan(1, (40, 40), 8, p, 1, nd), _plan(1, (40, 40), 2048, p, 2, nd)


def _caller(kind, plan, W, stream):
    import torch
    st = itc.new_stats(plan.B, W.device)
    gW = torch.zeros_like(W)
    gh = torch.zeros(plan.pixels, device=W.device)
    lab = torch.zeros(plan.pixels, dtype=torch.int16, device=W.device)
    itc.run_fields(plan)
    torch.cuda.synchronize()
    if kind in ("recursive", "fields", "fields_3d"):
        return (lambda: itc.run_fields(plan, stream=stream)), plan.ws[:4 * 40 * 40]
    if kind == "iterate":
        return (lambda: itc.run_iterate(plan, W, st, stream=stream)), st
    if kind == "segment":
        return (lambda: itc.segment(plan, W, lab, stream=stream)), lab
    return (lambda: itc.backward(plan, W, grad_W=gW, grad_h=gh, stream=stream)), gh


@pytest.mark.parametrize("kind", ["recursive", "iterate", "backward", "backward_3d", "segment", "fields", "fields_3d"])
def test_two_threads(kind):
    import torch
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    calls, outs = zip(*[_caller(kind, plan, W, s) for (plan, W), s in zip(_cases(kind), streams)])
    want = []
    for call, out in zip(calls, outs):
        call()
        torch.cuda.synchronize()
        want.append(out.clone())
    errors, start = [], threading.Barrier(2)

    def work(call):
        start.wait()
        try:
            for _ in range(CALLS):
                call()
        except itc.ItcError as e:
            errors.append(str(e))

    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for out, w in zip(outs, want):
        assert torch.equal(out, w)
