"""The tiled 2-D fields kernel against the plain one: absolute moments on rows off 16-byte boundaries go
through the plain kernel at every radius, and its A plane and S_XX are the same sums in the same order as
those of centred moments, which the tiled kernel computes at radii 3 to 16 (weights: 12) from thread copies
(the same rows) and tensor copies (rows on 16-byte boundaries).  Bit for bit, with few, many and very many
tiles per launch, so that byte images of 0/1 also meet the table of one-run windows (radii 9 to 13)."""
import numpy as np
import pytest

from paper_1310_7114_gb300 import build, itc

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    itc.lib()


def _image(side, dtype, binary):
    """Rings and bars with edges on every column phase; off binary, noise in a tenth of the pixels."""
    import torch
    g = torch.Generator(device="cuda").manual_seed(side)
    H, W = side, side + 3
    u = torch.arange(H, device="cuda")[:, None].float()
    v = torch.arange(W, device="cuda")[None].float()
    r = torch.hypot((u % 173) - 80, (v % 211) - 100)
    x = ((r < 70) & (r > 31)) | ((u + 2 * v) % 157 < 23)
    x[: H // 3, : W // 4] = False
    x = x.to(dtype)
    if not binary:
        noise = torch.rand((H, W), generator=g, device="cuda")
        vals = torch.randint(1, 256, (H, W), generator=g, device="cuda").to(dtype) if dtype == torch.uint8 else torch.rand((H, W), generator=g, device="cuda")
        x = torch.where(noise < 0.1, vals, x)
    return x.contiguous()


@pytest.mark.parametrize("R", range(3, 17))
@pytest.mark.parametrize("kind", ["few bytes", "few 0/1", "few weights", "many bytes", "many 0/1", "many weights", "very many 0/1"])
def test_same_bits(R, kind):
    import torch
    size, what = kind.rsplit(" ", 1)
    dtype = torch.float32 if what == "weights" else torch.uint8
    if dtype == torch.float32 and R > 12:
        pytest.skip("weights at radii above 12 have the plain kernel alone")
    if size == "very many" and R not in (9, 10, 11, 12, 13, 14):
        pytest.skip("the table's radii")
    side = {"few": 200, "many": 3100, "very many": 8200}[size]   # 16, 2401 and 16641 tiles
    x = _image(side, dtype, what != "bytes")
    H, W = x.shape
    sigma = (R - 0.3) / 3.0
    plain, s0 = itc.fields(x, sigma, absolute=True)
    want = plain[0, 0, :, :W].clone()
    del plain
    wide = torch.zeros((H, (W + 15) // 16 * 16), dtype=dtype, device="cuda")
    wide[:, :W] = x
    for t in (x, wide[:, :W]):
        F, s = itc.fields(t, sigma)
        assert torch.equal(F[0, 0, :, :W], want), (t.stride(), (F[0, 0, :, :W] != want).sum().item())
        assert s.item() == s0.item()
