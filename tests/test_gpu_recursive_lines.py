"""Recursive fields at the edges of the line scan: lines shorter than a warp, one and two samples per
lane, odd row and column counts (a line pair with one line), the longest line the scan takes and the
first one it leaves to the sequential kernels, both data types, all in one batch.  Against the FP64
oracle with the rounding envelope of tests/test_gpu_recursive.py."""
import numpy as np
import pytest

import oracle
import test_gpu_recursive as rec
from gpuhelp import to_dev
from paper_1310_7114_gb300 import build, itc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    itc.lib()


SHAPES = [(1, 1), (1, 9), (31, 33), (32, 32), (33, 31), (65, 7), (8, 64), (9, 95), (97, 130), (2048, 5), (5, 2048),
          (2049, 9), (9, 2049)]


@pytest.mark.parametrize("dtype", [np.uint8, np.float32])
def test_lines_of_every_length(dtype):
    import torch
    rng = np.random.default_rng(11)
    images = [((rng.random(s) < 0.4) if dtype == np.uint8 else rng.random(s)).astype(dtype) for s in SHAPES]
    params = [itc.make_params(float(s), 3.0, 0, flags=itc.ITC_RECURSIVE, sigma_self=float(s) * 0.6)
              for s in np.linspace(4.0, 25.0, len(SHAPES))]
    plan = itc.Plan([to_dev(im) for im in images], [1] * len(images), params)
    st = itc.new_stats(len(images), plan.dev.device)
    itc.run(plan, plan.pack_W([np.zeros((1, 2), np.float32)] * len(images)), st)
    torch.cuda.synchronize()
    sxx = itc.stats_to_numpy(st)["sxx"]
    for b, (im, p) in enumerate(zip(images, params)):
        h = im.astype(np.float64)
        ref = oracle.fields2d_recursive(h, float(p.sigma[0]))
        got = plan.fields_of(b)[:, 0, :, :im.shape[1]].cpu().numpy().astype(np.float64)
        env = rec.rounding_envelope(h, float(p.sigma[0]))
        for f in range(3):
            err = np.abs(got[f] - ref[f])
            assert np.all(err <= env[f] + 1e-30), (im.shape, f, (err / np.maximum(env[f], 1e-300)).max())
        own = oracle.fields2d_recursive(h, float(p.sigma_self[0]))[0]
        assert abs(sxx[b] - float((h * own).sum())) <= 1e-5 * max(1e-6, float((h * np.abs(own)).sum())), im.shape
