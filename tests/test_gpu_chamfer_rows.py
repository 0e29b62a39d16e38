"""Chamfer weights at the edges of the row layout: widths around each number of columns per lane,
heights around the rows loaded ahead, rows on 16-, 8- and 1-byte boundaries, foreground bytes of any
nonzero value.  Whole numbers: equal to the oracle's sequential passes."""
import numpy as np
import pytest

import oracle
from paper_1310_7114_gb300 import build, itc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    itc.lib()


@pytest.mark.parametrize("align", [16, 8, 1])
@pytest.mark.parametrize("width", [3, 4, 5, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024])
def test_row_layouts(width, align):
    import torch
    rng = np.random.default_rng(width * 31 + align)
    images = []
    for h in (1, 2, 3, 4, 5, 8, 9, 70):
        im = (rng.random((h, width)) < (0.97 if h > 4 else 0.7)).astype(np.uint8) * rng.integers(1, 256, (h, width))
        images.append(im.astype(np.uint8))
    _, views = itc.pack_images(images, "cuda", align=align)
    plan = itc.Plan(views, [1] * len(images), itc.make_params(2.0))
    _, T = itc.chamfer(plan)
    torch.cuda.synchronize()
    for im, t in zip(images, T):
        assert np.array_equal(t.cpu().numpy(), oracle.chamfer34((im != 0).astype(np.uint8)).astype(np.float32)), im.shape
