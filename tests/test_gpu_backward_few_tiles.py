"""The 2-D pixel pass with few tiles (16 x 16 per warp) and many (16 x 64): the same images alone and in a
batch give the same dD/dh bit for bit, at the edges of both tiles, on rows of every boundary, with codebooks on
and off the lattice; one against the oracle (the element-wise bound of gpuhelp)."""
import numpy as np
import pytest

import oracle
from gpuhelp import assert_grad_h_close, to_dev
from paper_1310_7114_gb300 import build, itc

pytestmark = pytest.mark.gpu
SHAPES = [(1, 1), (3, 15), (16, 16), (17, 17), (15, 33), (40, 47), (33, 64), (64, 65), (50, 130)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    itc.lib()


@pytest.mark.parametrize("M", [1, 15, 17, 33, 70])
@pytest.mark.parametrize("real", [False, True])
def test_few_and_many_tiles(M, real):
    import torch
    rng = np.random.default_rng(M)
    images = [(rng.random(s) * (rng.random(s) < 0.7)).astype(np.float32) for s in SHAPES]
    for im in images:
        im[0, 0] = 0.5
    ts = [to_dev(im) for im in images]
    books = [rng.uniform(0, 1, (M, 2)).astype(np.float32) * (np.array(s, np.float32) - 1) for s in SHAPES]
    if not real:
        books = [np.floor(b + 0.5).astype(np.float32) for b in books]
    for b in books:
        b[0] = 0.0                      # a vector on data
    p = itc.make_params(2.5, 3.0, 0, sigma_self=2.0)

    def grad(ids):
        plan = itc.Plan([ts[i] for i in ids], [M] * len(ids), p)
        W = plan.pack_W([books[i] for i in ids])
        itc.run_fields(plan)
        gh = torch.full((plan.pixels,), float("nan"), device=W.device)
        itc.backward(plan, W, grad_h=gh)
        return [g.copy() for g in plan.unpack_pixels(gh)]

    k = len(SHAPES)
    few = grad(range(k))
    many = grad([i % k for i in range(60 * k)])   # some 1700 strips
    for i, g in enumerate(many):
        assert np.array_equal(g, few[i % k]), SHAPES[i % k]
    for im, b, g in zip(images, books, few):
        h = im.astype(np.float64)
        _, ref, sums = oracle.dcs_grad2d_dense(h, 2.5, b.astype(np.float64), s=2.0)
        assert_grad_h_close(g, im, oracle.fields2d(h, 2.0)[0], sums, ref, what=str(im.shape))
