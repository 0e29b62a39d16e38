"""Segment labels at widths whose inverse square is infinite or nearly so, against the oracle, which
evaluates the same single-precision rule.  At tau = 1e-20 every metric is infinite or NaN: no comparison
holds and the first vector keeps every pixel; at 1e-19 sites up to one step away have finite metrics."""
import numpy as np
import pytest

import oracle
from gpuhelp import to_dev
from paper_1310_7114_gb300 import build, itc

pytestmark = pytest.mark.gpu
SHAPES = [(1, 1), (9, 33), (40, 40), (64, 65), (130, 129), (5, 300)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    itc.lib()


@pytest.mark.parametrize("sigma", [1e-20, 1e-19, (1e-20, 3.0)])
@pytest.mark.parametrize("M", [1, 3, 40])
def test_degenerate_widths(sigma, M):
    import torch
    rng = np.random.default_rng(M)
    images = [np.ones(s, np.uint8) for s in SHAPES]
    books = [np.stack([rng.uniform(0, s[0], M), rng.uniform(0, s[1], M)], 1).astype(np.float32) for s in SHAPES]
    plan = itc.Plan([to_dev(im) for im in images], [M] * len(images), itc.make_params(sigma, 3.0, 0))
    W = plan.pack_W(books)
    labels = torch.full((plan.pixels,), 9999, dtype=torch.int16, device=W.device)
    got = plan.unpack_pixels(itc.segment(plan, W, labels))
    with np.errstate(over="ignore"):
        for im, Wb, lab in zip(images, books, got):
            assert np.array_equal(lab.astype(np.int32), oracle.segment2d(im, sigma, Wb)), im.shape
