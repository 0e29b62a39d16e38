"""The iteration kernels' variants against the FP64 oracle and one another: a lone image (two
threads per vector, or a cluster of CTAs above 128 vectors), a batch of 160 (threads and CTAs
shared, one CTA per large image, in the common launch or one of its own) and images one at a time
in range calls.  Every variant adds its sums in the same order, so they agree bit for bit; the
oracle comparison is that of tests/test_gpu_run.py (equal codebooks but for rounding ties)."""
import numpy as np
import pytest

import oracle
from gpuhelp import DCS_ATOL, plan_lockstep, to_dev
from paper_1310_7114_gb300 import build, itc, synth

pytestmark = pytest.mark.gpu
ITERS = 6


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    itc.lib()


def _image(ndim, seed):
    rng = np.random.default_rng(seed)
    if ndim == 2:
        return (rng.random((61, 77)) < 0.4).astype(np.uint8), 1
    return rng.integers(0, 40, (40, 45)).astype(np.uint8), 40


def _run(ts, n, M, W0s, params, ndim, G):
    import torch
    k = len(ts)
    plan = itc.Plan([ts[b % k] for b in range(n)], [M] * n, params, ndims=[ndim] * n, Gs=[G] * n)
    W = plan.pack_W([W0s[b % k] for b in range(n)])
    st = itc.new_stats(n, W.device)
    itc.run(plan, W, st)
    torch.cuda.synchronize()
    return plan, plan.unpack_W(W), itc.stats_to_numpy(st)


@pytest.mark.parametrize("M", [31, 33, 63, 64, 65, 127, 128, 129, 144, 257, 700])
@pytest.mark.parametrize("ndim,flags", [(2, 0), (2, itc.ITC_CONTINUOUS), (2, itc.ITC_STOP_ON_FIXED), (3, 0)])
def test_variants_agree_with_the_oracle_and_bit_for_bit(M, ndim, flags):
    import torch
    sigma = 2.0 if ndim == 2 else (2.0, 2.5, 3.0)
    images = [_image(ndim, s)[0] for s in (1, 2, 3)]
    G = _image(ndim, 1)[1]
    init = synth.init_codebook if ndim == 2 else synth.init_codebook_gray
    W0s = [init(synth.rng_for(7, M + i), im.astype(np.float32) if ndim == 2 else im, M) for i, im in enumerate(images)]
    params = itc.make_params(sigma, 3.0, ITERS, flags=flags)
    ts = [to_dev(im) for im in images]
    plan, Wb, sb = _run(ts, 160, M, W0s, params, ndim, G)
    # one image at a time, as ranges of the same plan
    Wr, sr = plan.pack_W([W0s[b % 3] for b in range(160)]), itc.new_stats(160, plan.dev.device)
    s = torch.cuda.current_stream().cuda_stream
    for b in (0, 1, 159):
        rc = itc.lib().itc_run_iterate_range(plan.host_ptr, plan.dev.data_ptr(), b, b + 1, Wr.data_ptr(), sr.data_ptr(),
                                             plan.ws.data_ptr(), plan.ws.numel(), s)
        assert rc == itc.ITC_OK
    torch.cuda.synchronize()
    Wr, sr = plan.unpack_W(Wr), itc.stats_to_numpy(sr)
    for i in range(3):
        _, (W1,), (s1,) = _run([ts[i]], 1, M, [W0s[i]], params, ndim, G)
        assert np.array_equal(Wb[i], W1) and np.array_equal(Wb[156 + i], W1), (i, "batch and lone image")
        for f in ("sxw", "sww", "empty", "moved", "iters_done"):
            assert sb[i][f] == s1[f], (i, f)
        assert abs(sb[i]["dcs"] - s1["dcs"]) <= 1e-12 * max(1.0, abs(s1["dcs"]))
    for b in (0, 1, 159):
        assert np.array_equal(Wb[b], Wr[b]) and sb[b]["sxw"] == sr[b]["sxw"] and sb[b]["sww"] == sr[b]["sww"], b
    if flags:
        return
    im = images[0]
    if ndim == 2:
        A, *F = oracle.fields2d(im.astype(np.float64), sigma)
        sxx = oracle.sxx(im.astype(np.float64), A)
    else:
        A, *F = oracle.fields3d(im, G, sigma)
        uu, vv = np.meshgrid(np.arange(im.shape[0]), np.arange(im.shape[1]), indexing="ij")
        sxx = float(A[im, uu, vv].sum())
    Wo, dcs, tie, _ = oracle.lattice_run(A, F, sxx, sigma, W0s[0], ITERS)
    if tie.min() > 1e-4:
        assert np.array_equal(Wb[0], Wo)
        assert abs(sb[0]["dcs"] - dcs[-1]) <= DCS_ATOL
    else:
        plan_lockstep([im], [M], params, [W0s[0]], ITERS, lambda b, W: oracle.lattice_step(A, F, sigma, W)[:2],
                      ndims=[ndim], Gs=[G])
