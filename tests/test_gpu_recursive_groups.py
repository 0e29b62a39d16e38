"""Recursive fields of batches whose images are filtered differently: many small ones sequentially, longer
lines by scans in several launches, sides past the longest scanned line sequentially, ranges of the plan, and
the self-overlap pass.  One image of a kind against the FP64 oracle (the rounding envelope of
tests/test_gpu_recursive.py; S_XX 1e-5), the others of its kind and the ranges bit for bit like it."""
import numpy as np
import pytest

import oracle
import test_gpu_recursive as rec
from gpuhelp import to_dev
from paper_1310_7114_gb300 import build, itc

pytestmark = pytest.mark.gpu
#        shape, how many of it
MIXES = {
    "small beside long": [((64, 64), 400), ((30, 41), 150), ((10, 2048), 2), ((2048, 9), 1)],
    "small beside sequential": [((64, 64), 400), ((11, 2060), 1), ((3000, 5), 2)],
    "short lines beside long": [((200, 190), 300), ((9, 2048), 2), ((1030, 40), 3)],
    "few lines beside many": [((100, 230), 1200), ((100, 2040), 1), ((300, 20), 5)],
    "every length": [((40, 50), 300), ((24, 400), 260), ((500, 20), 200), ((16, 1000), 170), ((8, 1500), 3), ((9, 2100), 1)],
}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    itc.lib()


def _params(k):
    s = 6.0 + 2.0 * k
    return itc.make_params(s, 3.0, 0, flags=itc.ITC_RECURSIVE, sigma_self=0.7 * s)


@pytest.mark.parametrize("mix", sorted(MIXES))
@pytest.mark.parametrize("dtype", [np.uint8, np.float32])
def test_mixed_lengths(mix, dtype):
    import torch
    rng = np.random.default_rng(3)
    kinds = [s for s, _ in MIXES[mix]]
    images = [((rng.random(s) < 0.4) if dtype == np.uint8 else rng.random(s)).astype(dtype) for s in kinds]
    ts = [to_dev(im) for im in images]
    W1 = [np.array([[h // 2, w // 2], [h // 3, w // 4]], np.float32) for h, w in kinds]
    ids = rng.permutation(np.repeat(np.arange(len(kinds)), [n for _, n in MIXES[mix]]))
    n = len(ids)
    plan = itc.Plan([ts[k] for k in ids], [2] * n, [_params(k) for k in ids])
    W = plan.pack_W([W1[k] for k in ids])
    st = itc.new_stats(n, W.device)
    itc.run(plan, W, st)
    torch.cuda.synchronize()
    s = itc.stats_to_numpy(st)
    first = {}
    for b in range(n):
        k = ids[b]
        F = plan.fields_of(b)[:, 0, :, :kinds[k][1]]
        if k not in first:
            first[k] = (F.clone(), s[b])
        assert torch.equal(F, first[k][0]) and s[b]["sxx"] == first[k][1]["sxx"] and s[b]["dcs"] == first[k][1]["dcs"], (b, kinds[k])
    for k, im in enumerate(images):
        h, p = im.astype(np.float64), _params(k)
        ref, env = oracle.fields2d_recursive(h, float(p.sigma[0])), rec.rounding_envelope(h, float(p.sigma[0]))
        for f in range(3):
            err = np.abs(first[k][0][f].cpu().numpy().astype(np.float64) - ref[f])
            assert np.all(err <= env[f] + 1e-30), (im.shape, f, (err / np.maximum(env[f], 1e-300)).max())
        own = oracle.fields2d_recursive(h, float(p.sigma_self[0]))[0]
        assert abs(first[k][1]["sxx"] - float((h * own).sum())) <= 1e-5 * max(1e-6, float((h * np.abs(own)).sum())), im.shape
    plan.ws.zero_()
    st = itc.new_stats(n, W.device)
    cur = torch.cuda.current_stream().cuda_stream
    cuts = [0, n // 3, n // 3 + 1, n - 7]   # the last images stay undone
    for b0, b1 in zip(cuts, cuts[1:]):
        assert itc.lib().itc_run_fields_range(plan.host_ptr, plan.dev.data_ptr(), b0, b1, plan.ws.data_ptr(),
                                              plan.ws.numel(), cur) == itc.ITC_OK
        assert itc.lib().itc_run_iterate_range(plan.host_ptr, plan.dev.data_ptr(), b0, b1, W.data_ptr(), st.data_ptr(),
                                               plan.ws.data_ptr(), plan.ws.numel(), cur) == itc.ITC_OK
    torch.cuda.synchronize()
    s = itc.stats_to_numpy(st)
    for b in range(cuts[-1]):
        k = ids[b]
        assert torch.equal(plan.fields_of(b)[:, 0, :, :kinds[k][1]], first[k][0]) and s[b]["sxx"] == first[k][1]["sxx"], (b, kinds[k])
    assert not any(plan.fields_of(b).any() for b in range(cuts[-1], n))
