"""Segment labels at the edges of the 64 x 64 blocks and 8 x 32 tiles, with few and many codebook
vectors, images without data in whole blocks, weights, and gray images with and without weights: equal
to the oracle, which evaluates the same single-precision rule."""
import numpy as np
import pytest

import oracle
from gpuhelp import to_dev
from paper_1310_7114_gb300 import build, itc

pytestmark = pytest.mark.gpu
SHAPES = [(1, 1), (7, 31), (8, 32), (9, 33), (63, 65), (64, 64), (65, 63), (130, 129), (5, 300), (200, 17)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    itc.lib()


def _labels(images, W, sigma, ndim=2, G=1, weights=None):
    import torch
    n = len(images)
    ws = [None if weights is None else to_dev(w) for w in (weights or [None] * n)]
    plan = itc.Plan([to_dev(im) for im in images], [len(w) for w in W], itc.make_params(sigma, 3.0, 0), ndims=[ndim] * n,
                    Gs=[G] * n, weights=ws)
    lab = itc.segment(plan, plan.pack_W(W))
    torch.cuda.synchronize()
    return plan.unpack_pixels(lab)


@pytest.mark.parametrize("M", [1, 2, 31, 33, 150])
@pytest.mark.parametrize("dtype", [np.uint8, np.float32])
def test_blocks_2d(M, dtype):
    rng = np.random.default_rng(M)
    images, books = [], []
    for s in SHAPES:
        im = (rng.random(s) < 0.5).astype(dtype)
        im[: s[0] // 2, : s[1] // 2] = 0          # tiles and blocks without data
        images.append(im)
        w = np.stack([rng.uniform(-2, s[0] + 1, M), rng.uniform(-2, s[1] + 1, M)], 1)
        books.append(np.concatenate([w[: (M + 1) // 2], w[: M // 2]]).astype(np.float32))   # ties: equal sites
    for im, W, lab in zip(images, books, _labels(images, books, 2.7)):
        assert np.array_equal(lab.astype(np.int32), oracle.segment2d(im, 2.7, W)), im.shape


@pytest.mark.parametrize("weighted", [False, True])
def test_blocks_3d(weighted):
    rng = np.random.default_rng(5)
    sigma = (2.0, 3.0, 5.0)
    images = [rng.integers(0, 50, s).astype(np.uint8) for s in SHAPES]
    weights = [((rng.random(s) < 0.6) * rng.random(s)).astype(np.float32) for s in SHAPES] if weighted else None
    books = [rng.uniform(0, 1, (40, 3)).astype(np.float32) * np.array([s[0], s[1], 50], np.float32) for s in SHAPES]
    got = _labels(images, books, sigma, 3, 50, weights)
    for b, (im, W, lab) in enumerate(zip(images, books, got)):
        ref = oracle.segment3d(im, sigma, W, 50, weights[b] if weighted else None)
        assert np.array_equal(lab.astype(np.int32), ref), im.shape


@pytest.mark.parametrize("large", [(70, 520), (300, 280)])
def test_blocks_of_a_large_batch(large):
    """Enough images to fill the GPU: whole blocks for the large ones, strips of 16 rows for the small."""
    rng = np.random.default_rng(large[0])
    shapes = [(int(a), int(b)) for a, b in rng.integers(3, 40, (790, 2))] + [large] * 3 + [(64, 64), (65, 129)]
    images = [(rng.random(s) < 0.5).astype(np.uint8) for s in shapes]
    books = [np.stack([rng.uniform(-1, s[0], m), rng.uniform(-1, s[1], m)], 1).astype(np.float32)
             for s, m in zip(shapes, rng.integers(1, 40, len(shapes)))]
    got = _labels(images, books, 2.7)
    for b in [*range(0, 790, 40), *range(790, len(shapes))]:
        assert np.array_equal(got[b].astype(np.int32), oracle.segment2d(images[b], 2.7, books[b])), shapes[b]
