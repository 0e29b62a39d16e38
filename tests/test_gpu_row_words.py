"""Byte images whose rows start on every boundary of a word, down to one column, as views into a buffer of
other bytes: fields against the FP64 oracle, chamfer weights equal to it, and recursive fields with odd
widths in padded rows bit for bit those of contiguous ones.  The neighbours are 255 in one buffer and 0 in
the other, and no result depends on them."""
import numpy as np
import pytest

import oracle
from gpuhelp import assert_fields_close, radii
from paper_1310_7114_gb300 import build, itc

pytestmark = pytest.mark.gpu
SHAPES = [(1, 1), (1, 70), (2, 9), (5, 1), (3, 2), (4, 3), (7, 4), (6, 5), (40, 37), (70, 63), (66, 131), (9, 300)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    itc.lib()


def _views(images, pitches, shift, fill):
    """Every image at byte `shift` of a word of one buffer that holds `fill` elsewhere."""
    import torch
    offs, total = [], 64
    for im, p in zip(images, pitches):
        offs.append(total + shift)
        total += (im.shape[0] * p + 64 + 15) // 16 * 16
    buf = torch.full((total + 64,), fill, dtype=torch.uint8, device="cuda")
    out = []
    for im, p, o in zip(images, pitches, offs):
        v = buf[o:o + im.shape[0] * p].view(im.shape[0], p)[:, :im.shape[1]]
        v.copy_(torch.from_numpy(im))
        out.append(v)
    return out


def _images(seed):
    rng = np.random.default_rng(seed)
    return [(rng.random(s) < 0.6).astype(np.uint8) for s in SHAPES]


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("pad", [0, 1, 16])
def test_fields_and_chamfer(shift, pad):
    images = _images(shift)
    pitches = [(s[1] + 15) // 16 * 16 if pad == 16 else s[1] + pad for s in SHAPES]
    got = []
    for fill in (255, 0):
        ts = _views(images, pitches, shift, fill)
        plan = itc.Plan(ts, [1] * len(ts), itc.make_params(2.0, 3.0, 0))
        itc.run_fields(plan)
        T = [t.cpu().numpy() for t in itc.chamfer(plan)[1]]
        got.append(([plan.fields_of(b)[:, 0, :, :s[1]].cpu().numpy() for b, s in enumerate(SHAPES)], T))
    for b, im in enumerate(images):
        (Fa, Ta), (Fb, Tb) = [(g[0][b], g[1][b]) for g in got]
        assert np.array_equal(Fa, Fb) and np.array_equal(Ta, Tb), im.shape
        assert np.array_equal(Ta, oracle.chamfer34(im).astype(np.float32)), im.shape
        assert_fields_close(list(Fa.astype(np.float64)), oracle.fields2d(im.astype(np.float64), 2.0), radii(2.0), False, str(im.shape))


@pytest.mark.parametrize("fill", [0, 255])
def test_recursive_pairs_of_odd_widths(fill):
    import torch
    images = _images(9)
    params = itc.make_params(7.0, 3.0, 0, flags=itc.ITC_RECURSIVE, sigma_self=5.0)
    out = []
    for pitches in ([s[1] for s in SHAPES], [(s[1] + 2) // 2 * 2 for s in SHAPES]):
        plan = itc.Plan(_views(images, pitches, 0, fill), [1] * len(images), params)
        st = itc.new_stats(len(images), plan.dev.device)
        itc.run(plan, plan.pack_W([np.zeros((1, 2), np.float32)] * len(images)), st)
        torch.cuda.synchronize()
        out.append(([plan.fields_of(b)[:, 0, :, :s[1]].clone() for b, s in enumerate(SHAPES)], itc.stats_to_numpy(st)["sxx"]))
    for b, s in enumerate(SHAPES):
        assert torch.equal(out[0][0][b], out[1][0][b]) and out[0][1][b] == out[1][1][b], s
