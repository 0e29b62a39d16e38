"""The 2-D fields kernel with many tiles per launch (chunks of tiles, and the table of one-run windows of
byte images at radii 9 to 13): 0/1 silhouettes at radii 7 to 13, rows on 16-byte boundaries (tensor
copies) and on any boundary (copies by the threads), with the self-overlap pass at another radius.
Images repeat in the batch: each one's fields against the FP64 oracle (bounds of gpuhelp), every
repetition bit for bit the first.  S_XX: sums of products within the fields bound, 1e-5 relative."""
import numpy as np
import pytest

import oracle
from gpuhelp import assert_fields_close, radii, to_dev
from paper_1310_7114_gb300 import build, itc

pytestmark = pytest.mark.gpu
H, W = 121, 123          # 4 tiles; odd rows land on every boundary
KINDS = 4


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    itc.lib()


def _silhouette(k):
    """Discs, bars and rings whose edges fall on every column phase, and single pixels."""
    rng = np.random.default_rng(k)
    uu, vv = np.mgrid[0:H, 0:W]
    im = np.zeros((H, W), bool)
    for _ in range(6):
        cu, cv, r = rng.uniform(0, H), rng.uniform(0, W), rng.uniform(4, 40)
        d = np.hypot(uu - cu, vv - cv)
        im |= (d < r) & (d > r - rng.uniform(2, 60))
    im[:, 10 * k: 10 * k + 3 + k] ^= True
    im[rng.integers(0, H, 20), rng.integers(0, W, 20)] ^= True
    return im.astype(np.uint8)


@pytest.mark.parametrize("R", range(7, 14))
@pytest.mark.parametrize("align", [16, 1])
@pytest.mark.parametrize("tiles", [2000, 10000])
def test_many_tiles(R, align, tiles):
    import torch
    own_R = 13 if R < 10 else R - 1
    sigma, own = (R - 0.3) / 3.0, (own_R - 0.4) / 3.0
    images = [_silhouette(k) for k in range(KINDS)]
    _, views = itc.pack_images(images, "cuda", align=align)
    n = tiles // 4
    plan = itc.Plan([views[b % KINDS] for b in range(n)], [1] * n, itc.make_params(sigma, 3.0, 0, sigma_self=own))
    st = itc.new_stats(n, plan.dev.device)
    itc.run(plan, plan.pack_W([np.array([[60.0, 60.0]], np.float32)] * n), st)
    torch.cuda.synchronize()
    sxx = itc.stats_to_numpy(st)["sxx"]
    for k in range(KINDS):
        F = plan.fields_of(k)[:, 0, :, :W].clone()
        for b in range(k, n, KINDS):
            assert torch.equal(plan.fields_of(b)[:, 0, :, :W], F), (k, b)
            assert sxx[b] == sxx[k], (k, b)
        h = images[k].astype(np.float64)
        ref = oracle.fields2d(h, sigma)
        assert_fields_close([F[i].cpu().numpy().astype(np.float64) for i in range(3)], ref, radii(sigma), False, f"R={R}")
        want = oracle.sxx(h, oracle.fields2d(h, own)[0])
        assert abs(sxx[k] - want) <= 1e-5 * want
