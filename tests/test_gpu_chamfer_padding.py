"""Chamfer weights of the narrowest images and of widths around the lane sizes: equal to the oracle, with
the padding columns of every row as they were (itc.h: the padding columns are not written)."""
import numpy as np
import pytest

import oracle
from gpuhelp import to_dev
from paper_1310_7114_gb300 import build, itc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H", [1, 2, 5, 33])
def test_padding_is_not_written(H):
    import torch
    build.build()
    rng = np.random.default_rng(H)
    images = [np.ones((H, w), np.uint8) if w < 4 else (rng.random((H, w)) < 0.8).astype(np.uint8)
              for w in (1, 2, 3, 5, 9, 127, 129, 130, 257, 258, 513, 515)]
    plan = itc.Plan([to_dev(im) for im in images], [1] * len(images), itc.make_params(2.0, 3.0, 0))
    out = torch.full((int(itc.lib().itc_plan_padded_offset(plan.host_ptr, plan.B)),), -7.0, device="cuda")
    itc.chamfer(plan, out)
    got = out.cpu().numpy()
    for b, im in enumerate(images):
        o, fp = int(itc.lib().itc_plan_padded_offset(plan.host_ptr, b)), itc.field_pitch(im.shape[1])
        rows = got[o:o + H * fp].reshape(H, fp)
        assert np.array_equal(rows[:, :im.shape[1]], oracle.chamfer34(im).astype(np.float32)), im.shape
        assert np.all(rows[:, im.shape[1]:] == -7.0), im.shape
