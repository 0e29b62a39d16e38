"""S_XX and D_cs of gray images do not depend on how a batch is cut: one image, a range of a plan, a batch
that shares CTAs between images, and the backward's statistics give the same bits."""
import numpy as np
import pytest

from gpuhelp import to_dev
from paper_1310_7114_gb300 import build, itc

pytestmark = pytest.mark.gpu
N, G = 163, 90   # more images than one CTA each; 3 to a CTA's last group at M <= 32


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    itc.lib()


@pytest.mark.parametrize("M", [5, 30, 50, 100, 150])
def test_gray_sums_of_every_grouping(M):
    import torch
    rng = np.random.default_rng(M)
    shapes = [(33, 40), (70, 45), (40, 130), (97, 66)]
    ts = [to_dev(rng.integers(0, G, s).astype(np.uint8)) for s in shapes]
    # weights over 14 orders of magnitude, so that FP64 sums of the tiles' shares round
    hs = [to_dev((10.0 ** rng.uniform(-7, 7, s)).astype(np.float32)) for s in shapes]
    Ws = [np.floor(rng.random((M, 3)) * [*s, G]).astype(np.float32) for s in shapes]
    p = itc.make_params((2.0, 2.0, 3.0), 3.0, 1)

    def plan_of(ids):
        plan = itc.Plan([ts[i] for i in ids], [M] * len(ids), p, ndims=[3] * len(ids), Gs=[G] * len(ids),
                        weights=[hs[i] for i in ids])
        return plan, plan.pack_W([Ws[i] for i in ids]), itc.new_stats(len(ids), plan.dev.device)

    lone = []
    for i in range(4):
        plan, W, st = plan_of([i])
        itc.run(plan, W, st)
        b = itc.new_stats(1, plan.dev.device)
        itc.backward(plan, W, grad_W=torch.empty_like(W), stats=b)
        torch.cuda.synchronize()
        lone.append(itc.stats_to_numpy(st)[0])
        assert itc.stats_to_numpy(b)[0]["sxx"] == lone[i]["sxx"], i
    ids = [b % 4 for b in range(N)]
    plan, W, st = plan_of(ids)
    itc.run(plan, W, st)
    torch.cuda.synchronize()
    s = itc.stats_to_numpy(st)
    for b in range(N):
        for f in ("sxx", "sxw", "sww", "dcs"):
            assert s[b][f] == lone[ids[b]][f], (b, f, s[b][f], lone[ids[b]][f])
