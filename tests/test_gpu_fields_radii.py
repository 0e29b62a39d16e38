"""Every compiled radius of the tensor-tile fields kernel and the radii around them, both data types,
with the self-overlap pass at another width: against the FP64 oracle (bounds of gpuhelp) and bit for
bit against the plain kernel (a plan whose class is pinned to plain staging), S_XX included."""
import numpy as np
import pytest

import oracle
from gpuhelp import assert_fields_close, radii
from paper_1310_7114_gb300 import build, itc

pytestmark = pytest.mark.gpu
H, W = 197, 203


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    itc.lib()


def _image(dtype, seed):
    rng = np.random.default_rng(seed)
    uu, vv = np.mgrid[0:H, 0:W]
    solid = ((uu - 90) ** 2 + (vv - 110) ** 2 < 60 ** 2) | (vv >= 185) | (uu < 15)
    h = np.where(solid, 1.0, rng.random((H, W)) * (rng.random((H, W)) < 0.1))
    if dtype == np.uint8:
        h = np.where(h == 1.0, 1, (rng.random((H, W)) < 0.1) * rng.integers(1, 256, (H, W)))
        h[60:64] = 0
    return h.astype(dtype)


@pytest.mark.parametrize("R", range(2, 18))
@pytest.mark.parametrize("dtype", [np.uint8, np.float32])
@pytest.mark.parametrize("align", [16, 1])
def test_radius(R, dtype, align):
    import torch
    sigma, own = (R - 0.3) / 3.0, (max(R - 1, 1) - 0.4) / 3.0
    h = _image(dtype, R)
    _, (t,) = itc.pack_images([h], "cuda", align=align)
    p = itc.make_params(sigma, 3.0, 0, sigma_self=own)
    out = []
    for staging in ("default", "plain"):
        plan = itc.Plan([t], [1], p)
        if staging == "plain":
            plan.configure(0, 64, 0, "plain")
        st = itc.new_stats(1, t.device)
        itc.run(plan, plan.pack_W([np.array([[90.0, 110.0]], np.float32)]), st)
        gh = torch.empty(plan.pixels, device=t.device)
        itc.backward(plan, plan.pack_W([np.array([[90.0, 110.0]], np.float32)]), grad_h=gh)
        torch.cuda.synchronize()
        out.append((plan.fields_of(0)[:, 0, :, :W].clone(), itc.stats_to_numpy(st)[0], gh))
    (Fa, sa, ga), (Fb, sb, gb) = out
    assert torch.equal(Fa, Fb) and torch.equal(ga, gb) and sa["sxx"] == sb["sxx"]
    F1, s1 = itc.fields(t, sigma, sigma_self=own)
    assert torch.equal(F1[:, 0, :, :W], Fa) and s1.item() == sa["sxx"]
    hd = h.astype(np.float64)
    ref = oracle.fields2d(hd, sigma)
    assert_fields_close([Fa[i].cpu().numpy().astype(np.float64) for i in range(3)], ref, radii(sigma), False, f"R={R}")
    A_own = oracle.fields2d(hd, own)[0]
    sxx = oracle.sxx(hd, A_own)
    assert abs(sa["sxx"] - sxx) <= 1e-5 * sxx
