"""The pixel pass of the backward at the edges of its 16 x 64 warp tiles, with fewer and more codebook
vectors over a tile than are staged at once, rows on 16-byte boundaries and off them, one image and many:
dD/dh against the oracle's analytic gradient, every pixel within 3e-5 of the magnitudes of its two terms
(FP32 sums; gpuhelp.assert_grad_h_close).  A plan with 2-D and gray images gives each the gradients it has in
a plan of its own, bit for bit."""
import numpy as np
import pytest

import oracle
from gpuhelp import assert_grad_h_close, to_dev
from paper_1310_7114_gb300 import build, itc

pytestmark = pytest.mark.gpu
ODD = [(1, 1), (15, 63), (16, 64), (17, 65), (33, 130), (48, 191), (5, 300), (200, 17)]
ALIGNED = [(1, 4), (15, 60), (16, 64), (17, 68), (47, 132), (130, 260)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    itc.lib()


def _grads(images, books, sigma, ndims=None, Gs=None):
    import torch
    plan = itc.Plan([to_dev(im) for im in images], [len(w) for w in books], itc.make_params(sigma, 3.0, 0), ndims=ndims, Gs=Gs)
    W = plan.pack_W(books)
    itc.run(plan, W)
    gW = torch.empty_like(W)
    gh = torch.empty(plan.pixels, dtype=torch.float32, device=W.device)
    itc.backward(plan, W, grad_W=gW, grad_h=gh)
    torch.cuda.synchronize()
    return plan.unpack_W(gW), plan.unpack_pixels(gh)


@pytest.mark.parametrize("M", [1, 16, 17, 150])
@pytest.mark.parametrize("shapes", [ODD, ALIGNED, ODD[4:5], ALIGNED[-1:]], ids=["odd", "aligned", "odd1", "aligned1"])
def test_pixel_tiles(M, shapes):
    rng = np.random.default_rng(M)
    images = [rng.uniform(0.2, 1.0, s).astype(np.float32) for s in shapes]
    books = [(rng.random((M, 2)) * (np.array(s) - 1)).astype(np.float32) for s in shapes]
    _, gh = _grads(images, books, 2.3)
    for im, W, g in zip(images, books, gh):
        _, ref, sums = oracle.dcs_grad2d_dense(im.astype(np.float64), 2.3, W.astype(np.float64))
        assert_grad_h_close(g, im, oracle.fields2d(im.astype(np.float64), 2.3)[0], sums, ref, what=str(im.shape))


def test_mixed_dimensions():
    rng = np.random.default_rng(5)
    flat = [(rng.random(s) < 0.6).astype(np.uint8) for s in ((33, 70), (64, 64))]
    gray = [rng.integers(0, 8, s).astype(np.uint8) for s in ((20, 33), (40, 24))]
    images = [flat[0], gray[0], flat[1], gray[1]]
    ndims, Gs = [2, 3, 2, 3], [1, 8, 1, 8]
    books = [(rng.random((9, d)) * (np.array([*im.shape, 8][:d]) - 1)).astype(np.float32) for im, d in zip(images, ndims)]
    gW, gh = _grads(images, books, 2.0, ndims, Gs)
    for b in range(4):
        gW1, gh1 = _grads(images[b:b + 1], books[b:b + 1], 2.0, ndims[b:b + 1], Gs[b:b + 1])
        assert np.array_equal(gW[b], gW1[0]) and np.array_equal(gh[b], gh1[0]), b


@pytest.mark.parametrize("shape", [(260, 250), (257, 289)])
def test_gray_tiles(shape):
    """A batch that fills the GPU takes larger tiles than one image: the same gradients, bit for bit."""
    rng = np.random.default_rng(shape[1])
    images = [rng.integers(0, 12, shape).astype(np.uint8) for _ in range(8)]
    books = [(rng.random((70, 3)) * (np.array([*shape, 12]) - 1)).astype(np.float32) for _ in images]
    gW, gh = _grads(images, books, (2.0, 3.0, 2.0), [3] * 8, [12] * 8)
    for b in (0, 7):
        gW1, gh1 = _grads(images[b:b + 1], books[b:b + 1], (2.0, 3.0, 2.0), [3], [12])
        assert np.array_equal(gW[b], gW1[0]) and np.array_equal(gh[b], gh1[0]), b
