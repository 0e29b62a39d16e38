"""What the library is measured on: calls that its users' programs make, through the public binding
(``paper_1310_7114_gb300.itc`` and ``.autograd``), from one 64 x 64 icon to a batch of 4096 ragged
silhouettes.

A case is a dict of plain values.  Image sides, codebook counts and widths follow from the case
alone; pixels, weights and codebooks from the seed.  Inputs are drawn on the GPU: silhouettes as
unions of ellipses, weights and gray images as smoothed noise, the distributions that
``paper_1310_7114_gb300.synth`` draws on the host.  ``exact`` restates the method in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1310_7114_gb300 import autograd, itc

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # one small shape, clustered and differentiated: the latency of the smallest calls
        dict(name="icon", kind="run", n=1, lo=64, hi=64, m_lo=8, m_hi=8, sigma="2", iters=50, aligned=True, f32=False),
        # one large scene, 100 iterations of one codebook
        dict(name="scene", kind="run", n=1, lo=1024, hi=1024, m_lo=64, m_hi=64, sigma="4", iters=100, aligned=True,
             f32=False),
        # the benchmark's batch: thousands of ragged silhouettes in one plan, forward and backward
        dict(name="shapes_4096", kind="run", n=4096, lo=64, hi=512, m_lo=16, m_hi=128, sigma="2,3,4", iters=50,
             aligned=True, f32=False),
        # weighted images, divergence and its gradient (no iterations): a training set's step on a kept plan
        dict(name="weights_256", kind="run", n=256, lo=512, hi=512, m_lo=32, m_hi=32, sigma="3", iters=0, aligned=True,
             f32=True),
        # a gray image as a 3-D lattice, forward and backward
        dict(name="gray_lattice", kind="gray", n=1, lo=256, hi=256, m=64, sigma="3,3,8", iters=100, levels=256,
             weighted=False),
        # the paper's two Parzen widths (V(X) at a width of its own), images as plain contiguous tensors
        dict(name="parzen_shapes", kind="parzen", n=512, lo=64, hi=512, m_lo=16, m_hi=128, xi=1.2, omega=1.7, iters=30,
             aligned=False),
        # fields and D_cs at the widths of the paper's schedule (recursive filters)
        dict(name="large_widths", kind="recursive", n=48, lo=128, hi=1024, m_lo=16, m_hi=128),
        # chamfer weights of a batch, the input of weighted clustering
        dict(name="chamfer_1024", kind="chamfer", n=1024, lo=64, hi=512),
        # segments of a batch by its codebooks
        dict(name="segment_1024", kind="segment", n=1024, lo=64, hi=512, m_lo=16, m_hi=128, sigma="2,3,4"),
        # fields and one update of a single weighted image of odd size, an ordinary contiguous tensor
        dict(name="odd_fields", kind="fields", rows=517, cols=771, m=48, sigma=2.5, absolute=False, aligned=False,
             f32=True),
        # the iterations of one large codebook on stored fields
        dict(name="big_codebook", kind="iterate", n=1, lo=768, hi=768, m_lo=1024, m_hi=1024, sigma="3", iters=20),
        # one training step through autograd, the plan built by the call as the function does
        dict(name="training_step", kind="autograd", n=8, lo=256, hi=256, m=32, sigma=3.0, budget=0),
    ]


def draw(rng):
    def log(lo, hi):
        return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))

    def sides(most):   # (lo, hi) of the sides
        hi = log(40, most)
        return max(24, int(hi * rng.uniform(0.15, 1.0))), hi

    def widths():
        if rng.random() < 0.5:
            return ",".join(rng.sample(["2", "3", "4"], rng.randint(1, 3)))
        return ",".join("%.2f" % rng.uniform(1.0, 6.0) for _ in range(rng.randint(1, 2)))

    def books(lo, most):   # (m_lo, m_hi), the smallest image large enough for the largest codebook
        cap = max(4, min(most, lo * lo // 64))
        m = log(2, cap)
        return m, m * 2 ** rng.randint(0, int(math.log2(max(1, cap // m))))

    kind = rng.choice(["run", "run", "gray", "parzen", "recursive", "chamfer", "segment", "fields", "iterate", "autograd"])
    if kind == "run":
        n = log(1, 2048)
        lo, hi = sides(1536 if n < 8 else 700 if n < 512 else 512)
        m_lo, m_hi = books(lo, 256)
        return dict(kind=kind, n=n, lo=lo, hi=hi, m_lo=m_lo, m_hi=m_hi, sigma=widths(),
                    iters=rng.choice([0, rng.randint(1, 100)]), aligned=rng.random() < 0.6, f32=rng.random() < 0.4)
    if kind == "gray":
        side = log(48, 288)
        return dict(kind=kind, n=rng.randint(1, 2), lo=int(side * rng.uniform(0.5, 1.0)), hi=side, m=log(2, 96),
                    sigma="%s,%.1f" % (rng.choice(["3,3", "2,2", "2.5,3.5"]), rng.uniform(2, 10)),
                    iters=rng.randint(1, 100), levels=rng.choice([256, 64, rng.randint(30, 256)]),
                    weighted=rng.random() < 0.3)
    if kind == "parzen":
        n = log(4, 768)
        lo, hi = sides(512)
        m_lo, m_hi = books(lo, 192)
        return dict(kind=kind, n=n, lo=lo, hi=hi, m_lo=m_lo, m_hi=m_hi, xi=round(rng.uniform(0.7, 2.5), 2),
                    omega=round(rng.uniform(1.0, 3.0), 2), iters=rng.randint(0, 50), aligned=rng.random() < 0.5)
    if kind == "recursive":
        lo, hi = sides(1024)
        m_lo, m_hi = books(lo, 128)
        return dict(kind=kind, n=log(1, 60), lo=lo, hi=hi, m_lo=m_lo, m_hi=m_hi)
    if kind == "chamfer":
        lo, hi = sides(1024)
        return dict(kind=kind, n=log(1, 2048 if hi <= 512 else 256), lo=lo, hi=hi)
    if kind == "segment":
        lo, hi = sides(1024)
        m_lo, m_hi = books(lo, 512)
        return dict(kind=kind, n=log(1, 2048 if hi <= 512 else 256), lo=lo, hi=hi, m_lo=m_lo, m_hi=m_hi, sigma=widths())
    if kind == "fields":
        return dict(kind=kind, rows=log(17, 2048), cols=log(17, 2048), m=log(1, 128),
                    sigma=round(rng.choice([rng.uniform(0.8, 8.0), 2.0, 3.0, 4.0]), 2), absolute=rng.random() < 0.3,
                    aligned=rng.random() < 0.5, f32=rng.random() < 0.5)
    if kind == "iterate":
        side = log(384, 1024)
        m = log(24, 2048)
        return dict(kind=kind, n=rng.choice([1, 1, rng.randint(2, 24)]), lo=side, hi=side, m_lo=m, m_hi=m,
                    sigma="%.1f" % rng.uniform(2.0, 4.0), iters=rng.randint(5, 60 if m < 512 else 20))
    side = log(48, 512)
    return dict(kind=kind, n=rng.randint(1, 24), lo=max(32, int(side * rng.uniform(0.5, 1.0))), hi=side, m=log(4, 96),
                sigma=round(rng.choice([rng.uniform(1.0, 5.0), 3.0]), 2), budget=rng.choice([0, 0, 16 << 20]))


# ------------------------------------------------------------------------- what a case fixes
def _shapes(c):
    """(rows, columns) of every image."""
    if "rows" in c:
        return [(c["rows"], c["cols"])]
    rng = np.random.default_rng([c["n"], c["lo"], c["hi"]])
    return [tuple(int(x) for x in p) for p in rng.integers(c["lo"], c["hi"] + 1, (c["n"], 2))]


def _counts(c):
    """Codebook vectors of every image: m_lo times a power of two, up to m_hi."""
    n = c.get("n", 1)
    if "m" in c:
        return [c["m"]] * n
    steps = int(math.log2(c["m_hi"] // c["m_lo"])) if "m_lo" in c else 0
    rng = np.random.default_rng([n, steps])
    return [c.get("m_lo", 1) << int(k) for k in rng.integers(0, steps + 1, n)]


def _widths(c):
    """Kernel width of every image of a 2-D batch."""
    s = [float(x) for x in str(c.get("sigma", 2.0)).split(",")]
    rng = np.random.default_rng([len(s), 7])
    return [s[int(k)] for k in rng.integers(0, len(s), c.get("n", 1))]


def _radius(sigma):
    return math.ceil(3.0 * float(np.float32(sigma)))


# ------------------------------------------------------------------------------- inputs
def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 64 + salt)
    return g


def _uniform(g, shape, lo, hi):
    return lo + (hi - lo) * torch.rand(shape, generator=g, device=DEV)


def _silhouettes(shapes, seed):
    """Unions of ellipses (semi-axes 4-16 % of the shorter side), 5-40 % on; yields padded
    uint8 chunks [m, H, W] of consecutive images."""
    g = _gen(seed, 1)
    host = np.random.default_rng([int(seed), 1])
    frac = host.uniform(0.05, 0.40, len(shapes))
    count = [int(min(96, max(2, math.ceil(-math.log1p(-f) * h * w / (0.0314 * min(h, w) ** 2)))))
             for f, (h, w) in zip(frac, shapes)]
    b = 0
    while b < len(shapes):
        e = b + 1
        while e < len(shapes) and e - b < 64:
            m = e + 1 - b
            hm, wm = (max(s[i] for s in shapes[b:e + 1]) for i in (0, 1))
            if m * max(count[b:e + 1]) * hm * wm > 1 << 28:
                break
            e += 1
        hm, wm = (max(s[i] for s in shapes[b:e]) for i in (0, 1))
        m, k = e - b, max(count[b:e])
        hw = torch.tensor(shapes[b:e], dtype=torch.float32, device=DEV)
        side = hw.amin(1, keepdim=True)
        cu, cv = (_uniform(g, (m, k), 0.0, 1.0) * hw[:, i:i + 1] for i in (0, 1))
        ra, rb = ((_uniform(g, (m, k), 0.04, 0.16) * side).clamp_min(1.5) for _ in range(2))
        th = _uniform(g, (m, k), 0.0, math.pi)
        co, si = th.cos(), th.sin()
        quu = (co / ra) ** 2 + (si / rb) ** 2
        qvv = (si / ra) ** 2 + (co / rb) ** 2
        quv = 2 * co * si * (1 / ra ** 2 - 1 / rb ** 2)
        cst = quu * cu ** 2 + quv * cu * cv + qvv * cv ** 2
        off = torch.arange(k, device=DEV)[None, :] >= torch.tensor(count[b:e], device=DEV)[:, None]
        cst = torch.where(off, torch.full_like(cst, 1e9), cst)
        coef = torch.stack([quu, quv, qvv, -2 * quu * cu - quv * cv, -2 * qvv * cv - quv * cu, cst], -1)
        u = torch.arange(hm, device=DEV, dtype=torch.float32)[:, None].expand(hm, wm)
        v = torch.arange(wm, device=DEV, dtype=torch.float32)[None, :].expand(hm, wm)
        basis = torch.stack([u * u, u * v, v * v, u, v, torch.ones_like(u)]).reshape(6, -1)
        inside = (coef.reshape(m * k, 6) @ basis).view(m, k, hm, wm).amin(1) <= 1.0
        yield b, e, inside.to(torch.uint8)
        b = e


def _noise(shapes, seed, width):
    """Smoothed white noise of unit variance, padded chunks [m, H, W] as _silhouettes yields."""
    g = _gen(seed, 2)
    r = int(4 * width)
    x = torch.arange(-r, r + 1, device=DEV, dtype=torch.float32)
    k = torch.exp(-x * x / (2 * width * width))
    k = k / k.sum()
    for b in range(0, len(shapes), 32):
        e = min(len(shapes), b + 32)
        hm, wm = (max(s[i] for s in shapes[b:e]) for i in (0, 1))
        z = torch.randn((e - b, 1, hm + 2 * r, wm + 2 * r), generator=g, device=DEV)
        z = torch.nn.functional.conv2d(z, k.view(1, 1, -1, 1))
        z = torch.nn.functional.conv2d(z, k.view(1, 1, 1, -1))[:, 0]
        yield b, e, z / z.std()


def _pixels(c, seed):
    """Padded chunks of the case's images, as prepare() lays them out and exact() reads them."""
    shapes = _shapes(c)
    if c["kind"] == "gray":
        g = _gen(seed, 3)
        for b, e, z in _noise(shapes, seed, 6.0):
            lo, hi = z.amin((1, 2), keepdim=True), z.amax((1, 2), keepdim=True)
            top = c["levels"] - 1
            q = torch.round(top * (z - lo) / (hi - lo))
            flip = torch.rand(q.shape, generator=g, device=DEV)
            q = torch.where(flip < 0.025, torch.zeros_like(q), torch.where(flip > 0.975, torch.full_like(q, top), q))
            yield b, e, q.to(torch.uint8)
    elif c.get("f32", c["kind"] == "autograd"):
        for b, e, z in _noise(shapes, seed, 8.0):
            yield b, e, (0.5 + 0.25 * z).clamp(0.0, 1.0)
    else:
        yield from _silhouettes(shapes, seed)


def _sites(x, shapes, counts, g, thresh):
    """Distinct lattice sites with data of each image of a padded chunk, drawn at random."""
    m, hm, wm = x.shape
    score = torch.rand((m, hm * wm), generator=g, device=DEV)
    score = torch.where(x.reshape(m, -1) > thresh, score + 1.0, score)
    size = torch.tensor(shapes, device=DEV)
    inside = (torch.arange(hm, device=DEV)[None, :, None] < size[:, 0, None, None]) & \
             (torch.arange(wm, device=DEV)[None, None, :] < size[:, 1, None, None])
    score = torch.where(inside.reshape(m, -1), score, torch.full_like(score, -1.0))
    top = score.topk(max(counts), dim=1).indices
    uv = torch.stack([top // wm, top % wm], -1).float()
    return [uv[i, :counts[i]] for i in range(m)]


def _make(c, seed):
    """(images as 2-D tensors, codebooks, gray weights or None) on the GPU."""
    shapes, counts = _shapes(c), _counts(c)
    g = _gen(seed, 4)
    images, books = [], []
    aligned = c.get("aligned", c["kind"] != "autograd")
    for b, e, x in _pixels(c, seed):
        es = x.element_size()
        pitch = [(w + 15) // 16 * 16 if aligned else w for _, w in shapes[b:e]]
        start, total = [], 0
        for (h, _), p in zip(shapes[b:e], pitch):   # every image on a 256-byte boundary
            start.append(total)
            total += (h * p * es + 255) // 256 * 256 // es
        buf = torch.zeros(total, dtype=x.dtype, device=DEV)
        for i, (h, w) in enumerate(shapes[b:e]):
            im = buf[start[i]:start[i] + h * pitch[i]].view(h, pitch[i])[:, :w]
            im.copy_(x[i, :h, :w])
            images.append(im)
        if c["kind"] != "chamfer":
            thresh = -1.0 if c["kind"] == "gray" else 0.5
            books += _sites(x, shapes[b:e], counts[b:e], g, thresh)
    weights = None
    if c["kind"] == "gray":
        books = [torch.cat([w, im[w[:, 0].long(), w[:, 1].long()].float()[:, None]], 1) for w, im in zip(books, images)]
        if c["weighted"]:
            weights = []
            for im in images:
                wt = torch.empty((im.shape[0], im.stride(0)), device=DEV)[:, :im.shape[1]]
                weights.append(wt.copy_(_uniform(g, im.shape, 0.2, 1.0)))
    if c["kind"] == "autograd":   # codebooks that gradient steps have moved off the lattice
        books = [w + _uniform(g, w.shape, -0.45, 0.45) for w in books]
        books = [torch.minimum(w.clamp_min(0.0), torch.tensor([h - 1.0, v - 1.0], device=DEV))
                 for w, (h, v) in zip(books, shapes)]
    return images, books, weights


def _params(c, images, counts):
    if c["kind"] == "gray":
        return itc.make_params([float(x) for x in c["sigma"].split(",")], 3.0, c["iters"])
    if c["kind"] == "parzen":
        return itc.params_parzen(2, xi=c["xi"], omega=c["omega"], iters=c["iters"])
    if c["kind"] == "recursive":   # the schedule of Sec. 4: widths from each image's mass and codebook size
        return [itc.params_parzen(2, mass=float(im.sum()), M=m, flags=itc.ITC_RECURSIVE)
                for im, m in zip(images, counts)]
    made = {s: itc.make_params(s, 3.0, c.get("iters", 0)) for s in set(_widths(c))}
    return [made[s] for s in _widths(c)]


def prepare(case, seed):
    c = dict(case)
    kind = c["kind"]
    counts = _counts(c)
    images, books, weights = _make(c, seed)
    if kind == "autograd":
        return dict(c=c, hs=[im.contiguous().requires_grad_() for im in images],
                    Ws=[w.clone().requires_grad_() for w in books])
    if kind == "fields":
        return dict(c=c, image=images[0], W=books[0])
    n = len(images)
    dims = [3] * n if kind == "gray" else None
    plan = itc.Plan(images, counts, _params(c, images, counts), ndims=dims, Gs=[c["levels"]] * n if dims else None,
                    weights=weights)
    st = dict(c=c, plan=plan, images=images)
    if kind == "chamfer":
        st["out"] = torch.zeros(sum(h * itc.field_pitch(w) for h, w in plan.shapes), device=DEV)
        return st
    st["W0"] = torch.cat([w.reshape(-1) for w in books]).contiguous()
    if kind == "segment":
        st["labels"] = torch.empty(plan.pixels, dtype=torch.int16, device=DEV)
        return st
    st["stats"] = itc.new_stats(n, DEV)
    if kind == "recursive":
        st["fields"] = [plan.fields_of(b)[:, 0, :, :plan.shapes[b][1]] for b in range(n)]
        return st
    if kind == "iterate":
        itc.run_fields(plan)
        return st
    st["grad_W"] = torch.empty_like(st["W0"])
    st["grad_h"] = torch.empty(plan.pixels, device=DEV)
    return st


def _stats(buf, n):
    """D_cs per image in the type the autograd function gives it, and the counts of itc_stats."""
    return buf.view(torch.float64).view(n, 7)[:, 0].float(), buf.view(torch.int32).view(n, 14)[:, 10:]


def run(state):
    c = state["c"]
    kind = c["kind"]
    if kind == "autograd":
        hs, Ws = state["hs"], state["Ws"]
        d = autograd.itc_divergence(hs, Ws, c["sigma"], fields_budget_bytes=c["budget"] or None)
        grads = torch.autograd.grad(d.sum(), hs + Ws)
        return dict(dcs=d.detach(), grad_h=list(grads[:len(hs)]), grad_W=list(grads[len(hs):]))
    if kind == "fields":
        im = state["image"]
        flags = itc.ITC_FIELDS_ABSOLUTE if c["absolute"] else 0
        F, sxx = itc.fields(im, c["sigma"], absolute=c["absolute"])
        W, site, st = itc.step(im, F, sxx, state["W"], c["sigma"], flags=flags | itc.ITC_CONTINUOUS)
        return dict(fields=F[:, 0, :, :im.shape[1]], W=W, dcs=_stats(st, 1)[0])
    plan = state["plan"]
    if kind == "chamfer":
        return itc.chamfer(plan, state["out"], views=False)[0]
    if kind == "segment":
        return itc.segment(plan, state["W0"], state["labels"])
    W = state["W0"].clone()
    if kind == "recursive":
        itc.run(plan, W, state["stats"])
        return dict(dcs=_stats(state["stats"], plan.B)[0], fields=state["fields"])
    if kind == "iterate":
        itc.run_iterate(plan, W, state["stats"])
    else:
        itc.run(plan, W, state["stats"])
        itc.backward(plan, W, grad_W=state["grad_W"], grad_h=state["grad_h"])
    d, counts = _stats(state["stats"], plan.B)
    out = dict(W=W, dcs=d, counts=counts)
    if kind != "iterate":
        out.update(grad_W=state["grad_W"], grad_h=state["grad_h"])
    return out


# ------------------------------------------------------------------------------------- work
def work(case):
    c = dict(case)
    kind = c["kind"]
    shapes, counts = _shapes(c), _counts(c)
    px = sum(h * w for h, w in shapes)
    es = 4 if c.get("f32", kind == "autograd") else 1
    d = 3 if kind == "gray" else 2
    book = 4.0 * d * sum(counts)
    if kind == "chamfer":
        return dict(bytes=5.0 * px, flops=16.0 * px)
    if kind == "segment":
        return dict(bytes=3.0 * px + book, flops=0.2 * px * 5 * 8)
    if kind == "recursive":
        return dict(bytes=13.0 * px, flops=2 * 60.0 * px)
    if kind == "iterate":
        return dict(bytes=2 * book + 12.0 * sum(counts) * c["iters"], flops=10.0 * (c["iters"] + 1) * sum(m * m for m in counts))
    if kind == "gray":
        s = [float(x) for x in c["sigma"].split(",")]
        fma = px * c["levels"] * 7 * (2 * _radius(s[0]) + 1)
        window = (2 * _radius(s[0]) + 1) * (2 * _radius(s[1]) + 1)
    else:
        tau = [math.hypot(c["xi"], c["omega"])] * len(shapes) if kind == "parzen" else _widths(c)
        taps = [2 * _radius(s) + 1 for s in tau]
        fma = sum(5 * t * h * w for t, (h, w) in zip(taps, shapes))
        if kind == "parzen":
            fma += 2 * (2 * _radius(math.sqrt(2) * c["xi"]) + 1) * px
        window = taps[0] ** 2
    if kind == "fields":   # the fields are the result
        return dict(bytes=(es + 12.0) * px + 2 * book, flops=2.0 * fma)
    pairs = (c.get("iters", 0) + 1) * sum(m * m for m in counts)
    # the images and codebooks in, the codebooks and both gradients out
    return dict(bytes=(es + 4.0) * px + 3 * book, flops=2.0 * fma + 10.0 * pairs + 2.0 * sum(counts) * window)


# ------------------------------------------------------------------- the method in 64 bits
def _conv(x, dim, sigma):
    """(sum_d g(d) x(y + d), sum_d d g(d) x(y + d)) along dim, |d| <= ceil(3 sigma), zero outside."""
    sigma = float(np.float32(sigma))
    r, n = _radius(sigma), x.shape[dim]
    val, mom = torch.zeros_like(x), torch.zeros_like(x)
    for d in range(-min(r, n - 1), min(r, n - 1) + 1):
        g = math.exp(-d * d / (2 * sigma * sigma))
        src = x.narrow(dim, max(d, 0), n - abs(d))
        val.narrow(dim, max(-d, 0), n - abs(d)).add_(src, alpha=g)
        if d:
            mom.narrow(dim, max(-d, 0), n - abs(d)).add_(src, alpha=g * d)
    return val, mom


def _fields64(h, sigma):
    """[A, F_u, F_v] of a padded chunk [m, H, W] (zero outside each image)."""
    t, tv = _conv(h, 2, sigma)
    a, fu = _conv(t, 1, sigma)
    return [a, fu, _conv(tv, 1, sigma)[0]]


def _gather(planes, r):
    """planes[i][b, r...] for sites r [m, M, d]."""
    m = r.shape[0]
    idx = r[..., 0]
    for i in range(1, r.shape[2]):
        idx = idx * planes[0].shape[i + 1] + r[..., i]
    return [p.reshape(m, -1).gather(1, idx) for p in planes]


def _round(w, top):
    return torch.minimum((w + 0.5).floor().clamp_min(0.0), top)


def _evaluate(w, on, top, planes, rho):
    """(a, D, s, E) of every codebook vector: the gathered data terms and the pair sums."""
    r = _round(w, top)
    got = _gather(planes, r.long())
    a = got[0] * on
    D = torch.stack(got[1:], -1) * on[..., None] + (r - w) * a[..., None]
    d = w[:, None, :, :] - w[:, :, None, :]
    g = torch.exp(-(d * d / (2 * rho * rho)).sum(-1)) * on[:, None, :] * on[:, :, None]
    return a, D, g.sum(2), (g[..., None] * d).sum(2)


def _cluster(w, on, top, planes, sxx, tau, rho, s, iters):
    """(W, D_cs, a, D, S_XW, S_WW, E) after the snapped iterations."""
    kappa = tau * tau / (rho * rho)
    for t in range(iters + 1):
        a, D, ss, E = _evaluate(w, on, top, planes, rho)
        sxw, sww = a.sum(1), ss.sum(1)
        if t == iters:
            break
        step = (D - (sxw / sww)[:, None, None] * kappa * E) / a.clamp_min(1e-300)[..., None]
        w = torch.where((a > 0)[..., None], _round(w + step, top), w)
    const = 0.5 * torch.log(tau ** 4 / (rho ** 2 * s ** 2)).sum()
    return w, sww.log() + sxx.log() - 2 * sxw.log() + const, a, D, sxw, sww, E


def _stamp(w, on, top, hm, wm, tau):
    """sum_k g(x - w_k) over the box around round(w_k), [m, H, W]."""
    r = _round(w, top)
    f = []
    for i, n in ((0, hm), (1, wm)):
        x = torch.arange(n, device=DEV, dtype=F64)[None, None, :]
        d = x - w[..., i:i + 1]
        f.append(torch.exp(-d * d / (2 * tau[i] ** 2)) * ((x - r[..., i:i + 1]).abs() <= _radius(tau[i])))
    return torch.einsum("bkh,bkw->bhw", f[0] * on[..., None], f[1])


def _window_terms(h, w, on, top, tau):
    """a_k and D_k summed over the box around round(w_k) with the kernel at the real w_k."""
    m, hm, wm = h.shape
    r = _round(w, top)
    R = _radius(tau[0])
    o = torch.arange(-R, R + 1, device=DEV)
    u, v = (r[..., i].long()[..., None] + o for i in (0, 1))
    ok = ((u >= 0) & (u < hm))[..., :, None] & ((v >= 0) & (v < wm))[..., None, :]
    idx = u.clamp(0, hm - 1)[..., :, None] * wm + v.clamp(0, wm - 1)[..., None, :]
    x = h.reshape(m, -1).gather(1, idx.reshape(m, -1)).view(idx.shape) * ok * on[..., None, None]
    du, dv = u.to(F64) - w[..., :1], v.to(F64) - w[..., 1:]
    gu, gv = (torch.exp(-d * d / (2 * tau[0] ** 2)) for d in (du, dv))
    return (torch.einsum("bkuv,bku,bkv->bk", x, gu, gv),
            torch.stack([torch.einsum("bkuv,bku,bkv->bk", x, gu * du, gv), torch.einsum("bkuv,bku,bkv->bk", x, gu, gv * dv)], -1))


def _per_sigma(members, widths):
    """Members grouped by width, in pieces that keep the 64-bit planes within a few GB."""
    for s in sorted(set(widths)):
        same = [b for b in members if widths[b] == s]
        for i in range(0, len(same), 32):
            yield s, same[i:i + 32]


def _exact_2d(c, seed):
    kind = c["kind"]
    shapes, counts = _shapes(c), _counts(c)
    images, books, _ = _make(c, seed)
    n = len(images)
    widths = [math.hypot(np.float32(c["xi"]), np.float32(c["omega"]))] * n if kind == "parzen" else _widths(c)
    rho_s = [math.sqrt(2) * c["omega"], math.sqrt(2) * c["xi"]] if kind == "parzen" else None
    got = [None] * n
    for s, part in _per_sigma(range(n), widths):
        hm, wm = (max(shapes[b][i] for b in part) for i in (0, 1))
        mk = max(counts[b] for b in part)
        h = torch.zeros((len(part), hm, wm), dtype=F64, device=DEV)
        w = torch.zeros((len(part), mk, 2), dtype=F64, device=DEV)
        on = torch.zeros((len(part), mk), dtype=F64, device=DEV)
        for i, b in enumerate(part):
            h[i, :shapes[b][0], :shapes[b][1]] = images[b]
            w[i, :counts[b]] = books[b]
            on[i, :counts[b]] = 1.0
        tau = torch.tensor([float(np.float32(s))] * 2, dtype=F64, device=DEV)
        rho, slf = [torch.full_like(tau, float(np.float32(x))) for x in rho_s] if rho_s else (tau, tau)
        planes = _fields64(h, s)
        own = planes[0] if rho_s is None else _conv(_conv(h, 2, rho_s[1])[0], 1, rho_s[1])[0]
        sxx = (h * own).sum((1, 2))
        top = torch.tensor([[x - 1 for x in shapes[b]] for b in part], dtype=F64, device=DEV)[:, None, :]
        w, dcs, a, D, sxw, sww, E = _cluster(w, on, top, planes, sxx, tau, rho, slf, c.get("iters", 0))
        if kind == "autograd":   # the gradient takes its data terms at the real codebooks
            a, D = _window_terms(h, w, on, top, tau.tolist())
            sxw = a.sum(1)
        gw = gh = None
        if kind != "iterate":
            gw = 2 * (E / (rho * rho * sww[:, None, None]) - D / (tau * tau * sxw[:, None, None]))
            gh = 2 * own / sxx[:, None, None] - 2 / sxw[:, None, None] * _stamp(w, on, top, hm, wm, tau.tolist())
        for i, b in enumerate(part):
            k, (rows, cols) = counts[b], shapes[b]
            got[b] = (w[i, :k], dcs[i], None if gw is None else gw[i, :k], None if gh is None else gh[i, :rows, :cols].contiguous())
    flat = lambda j: torch.cat([g[j].reshape(-1) for g in got])  # noqa: E731
    if kind == "autograd":
        return dict(dcs=flat(1), grad_h=[g[3] for g in got], grad_W=[g[2] for g in got])
    out = dict(W=flat(0), dcs=flat(1), counts=None)
    if kind != "iterate":
        out.update(grad_W=flat(2), grad_h=flat(3))
    return out


def _exact_gray(c, seed):
    images, books, weights = _make(c, seed)
    s = [float(x) for x in c["sigma"].split(",")]
    tau = torch.tensor([float(np.float32(x)) for x in s], dtype=F64, device=DEV)
    G = c["levels"]
    Ws, ds, gws, ghs = [], [], [], []
    for b, im in enumerate(images):
        H, W = im.shape
        hw = weights[b].to(F64) if weights is not None else torch.ones((H, W), dtype=F64, device=DEV)
        vox = torch.zeros((H, W, G), dtype=F64, device=DEV)
        vox.scatter_(2, im.long()[..., None], hw[..., None])
        a0, ag = _conv(vox, 2, s[2])
        t, tv = _conv(a0, 1, s[1])
        A, Fu = _conv(t, 0, s[0])
        Fv, Fg = _conv(tv, 0, s[0])[0], _conv(_conv(ag, 1, s[1])[0], 0, s[0])[0]
        sxx = (vox * A).sum().reshape(1)
        planes = [p[None] for p in (A, Fu, Fv, Fg)]
        top = torch.tensor([[[H - 1.0, W - 1.0, G - 1.0]]], dtype=F64, device=DEV)
        on = torch.ones((1, c["m"]), dtype=F64, device=DEV)
        w, d, a, D, sxw, sww, E = _cluster(books[b].to(F64)[None], on, top, planes, sxx, tau, tau, tau, c["iters"])
        gw = 2 * (E / (tau * tau * sww[:, None, None]) - D / (tau * tau * sxw[:, None, None]))
        own = A.gather(2, im.long()[..., None])[..., 0]
        f = []
        for i, x in enumerate((torch.arange(H, device=DEV).view(1, H, 1), torch.arange(W, device=DEV).view(1, 1, W), im.long()[None])):
            e = x.to(F64) - w[0, :, i].view(-1, 1, 1)
            f.append(torch.exp(-e * e / (2 * tau[i] ** 2)) * (e.abs() <= _radius(s[i])))
        Ws.append(w.reshape(-1)), ds.append(d), gws.append(gw.reshape(-1))
        ghs.append((2 * own / sxx - 2 / sxw * (f[0] * f[1] * f[2]).sum(0)).reshape(-1))
    return dict(W=torch.cat(Ws), dcs=torch.cat(ds), counts=None, grad_W=torch.cat(gws), grad_h=torch.cat(ghs))


def _exact_fields(c, seed):
    images, books, _ = _make(c, seed)
    h = images[0].to(F64)[None]
    H, W = h.shape[1:]
    planes = _fields64(h, c["sigma"])
    sxx = (h * planes[0]).sum((1, 2))
    tau = torch.tensor([float(np.float32(c["sigma"]))] * 2, dtype=F64, device=DEV)
    top = torch.tensor([[[H - 1.0, W - 1.0]]], dtype=F64, device=DEV)
    w = books[0].to(F64)[None]
    on = torch.ones(w.shape[:2], dtype=F64, device=DEV)
    a, D, ss, E = _evaluate(w, on, top, planes, tau)
    sxw, sww = a.sum(1), ss.sum(1)
    step = (D - (sxw / sww)[:, None, None] * E) / a.clamp_min(1e-300)[..., None]
    w = torch.where((a > 0)[..., None], torch.minimum((w + step).clamp_min(0.0), top), w)
    if c["absolute"]:
        planes[1] = planes[1] + planes[0] * torch.arange(H, device=DEV)[:, None]
        planes[2] = planes[2] + planes[0] * torch.arange(W, device=DEV)[None, :]
    return dict(fields=torch.cat(planes), W=w[0], dcs=sww.log() + sxx.log() - 2 * sxw.log())


def _exact_recursive(c, seed):
    """The convolution with Deriche's two damped sinusoids (his fit of exp(-x^2 / 2)), untruncated."""
    images, books, _ = _make(c, seed)
    fit = [(1.680, 3.735, 0.6318, 1.783), (-0.6803, -0.2598, 1.997, 1.723)]   # alpha, beta, omega, b
    out, dcs = [], []

    def filters(n, sigma):   # the sampled fit and its first moment as matrices [site, source]
        d = torch.arange(n, device=DEV, dtype=F64)
        d = d[None, :] - d[:, None]
        x = d.abs() / float(np.float32(sigma))
        g = sum(torch.exp(-b * x) * (al * torch.cos(o * x) + be * torch.sin(o * x)) for al, be, o, b in fit)
        return g, g * d

    for im, m, w in zip(images, _counts(c), books):
        omega = math.sqrt(float(im.sum()) / m) / 2
        tau, rho, slf = math.hypot(omega, omega / 2), math.sqrt(2) * omega, math.sqrt(2) * omega / 2
        h = im.to(F64)
        (gu, mu), (gv, mv) = (filters(n, tau) for n in im.shape)
        t = h @ gv.T
        planes = [gu @ t, mu @ t, gu @ (h @ mv.T)]
        sxx = (h * (filters(im.shape[0], slf)[0] @ h @ filters(im.shape[1], slf)[0].T)).sum()
        wide = [torch.full((2,), float(np.float32(x)), dtype=F64, device=DEV) for x in (tau, rho, slf)]
        top = torch.tensor([[[n - 1.0 for n in im.shape]]], dtype=F64, device=DEV)
        on = torch.ones((1, m), dtype=F64, device=DEV)
        dcs.append(_cluster(w.to(F64)[None], on, top, [p[None] for p in planes], sxx.reshape(1), *wide, 0)[1])
        out.append(torch.stack(planes))
    return dict(dcs=torch.cat(dcs), fields=out)


def _exact_chamfer(c, seed):
    """The 3-4 distance to the background by relaxation; the plan's padded per-pixel layout."""
    shapes = _shapes(c)
    out = []
    for b, e, x in _pixels(c, seed):
        m, hm, wm = x.shape
        for i, (h, w) in enumerate(shapes[b:e]):
            x[i, h:] = 0
            x[i, :, w:] = 0
        T = torch.nn.functional.pad(torch.where(x != 0, 1e6, 0.0), (1, 1, 1, 1))
        mid = T[:, 1:-1, 1:-1]
        while True:
            best = mid
            for du in (0, 1, 2):
                for dv in (0, 1, 2):
                    if (du, dv) != (1, 1):
                        best = torch.minimum(best, T[:, du:du + hm, dv:dv + wm] + (3.0 if 1 in (du, dv) else 4.0))
            if torch.equal(best, mid):
                break
            mid.copy_(best)
        for i, (h, w) in enumerate(shapes[b:e]):
            out.append(torch.nn.functional.pad(mid[i, :h, :w], (0, -w % 4)).reshape(-1).to(F64))
    return torch.cat(out)


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "segment":
        return None   # labels: whole numbers
    if kind in ("run", "parzen", "iterate", "autograd"):
        return _exact_2d(c, seed)
    return {"gray": _exact_gray, "fields": _exact_fields, "recursive": _exact_recursive, "chamfer": _exact_chamfer}[kind](c, seed)
