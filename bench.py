#!/usr/bin/env python3
"""Benchmark of batched lattice ITC on one GB300 (or N, one process per GPU, weak scaling).

A step is one pass of the whole method over one batch of synthetic input, all in libitc.so:
  fields   (Algorithm 1 step 2: truncated separable Gaussian fields + S_XX of every image),
  iterate  (Algorithm 1 steps 3-11: 50 fixed-point updates per image, Eq. (origupdate)),
  backward (gradient of Eq. (1) with respect to every codebook and every pixel weight).
Default workload: 4096 binary blob silhouettes with sides U{64..512}, per-image M in
{16, 32, 64, 128} and sigma in {2, 3, 4} (synthetic stand-ins for the paper's MPEG-7 shapes).

Printed: one JSON line (rank 0).  `value` is images/s with the inputs resident in HBM, timed with
CUDA events on the launching stream; `e2e` is the same metric through the C ABI with the inputs
copied from pinned host memory and the results read back inside the timed region; `roofline`
is the fields pass (bytes per launch / its event-timed duration vs the measured HBM copy
bandwidth); `per_image_launch` is the same work launched image by image; `cpu_baseline` is the
FP64 oracle on this host.  `--impl reference` times the oracle alone on the same workload.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "batched ITC images/s vs per-image launch at ≤1e-5 rel err; conv GB/s % HBM peak"
FALLBACK_HBM_GBS = 6800.0

# DRAM bytes (read + write) per lattice site of the fields pass, from one ncu capture of the workload
# (C3: 1024 of its images, profiles/fields_tma_kernel_c3_1024.md; C5: its one launch,
# profiles/fields3d_kernel_c5_gray3d.md), valid only for the kernel source it was taken on
# (sha256 prefix below); scaled to a launch by its site count (pixels, or voxels of the 3-D lattice).
FIELDS_TRAFFIC = {
    "c3": {"bytes_per_site": 969.22e6 / 86358723, "source_sha256": "b4e07329e6363145",
           "source": "paper_1310_7114_gb300/csrc/itc_fields_tma.cuh",
           "note": "ncu dram bytes of the 1024-image capture scaled by pixels (profiles/fields_tma_kernel_c3_1024.md)"},
    "c5": {"bytes_per_site": (0.21e6 + 206.58e6) / 16777216, "source_sha256": "2e6cf066545e002d",
           "source": "paper_1310_7114_gb300/csrc/itc_fields3d.cu",
           "note": "ncu dram bytes of one launch (profiles/fields3d_kernel_c5_gray3d.md)"},
}


def fields_traffic(name, sites):
    """(DRAM bytes of one fields pass, note), or (None, why) when no capture covers this source."""
    import hashlib
    t = FIELDS_TRAFFIC.get(name)
    if t is None:
        return None, "no ncu capture of this workload's fields pass"
    with open(os.path.join(ROOT, t["source"]), "rb") as f:
        if hashlib.sha256(f.read()).hexdigest()[:16] != t["source_sha256"]:
            return None, "the kernel changed since its ncu capture"
    return t["bytes_per_site"] * sites, t["note"]


def fields_kernel_name(ndims, tuning):
    """The kernel that runs the fields pass of this plan."""
    if all(d == 3 for d in ndims):
        return "fields3d_kernel (persistent CTAs over runs of one-slice tiles, one launch)"
    kinds = sorted({c["staging"] for c in tuning})
    names = {"tma": "fields_tma_kernel", "plain": "fields_tma_kernel (thread staging) or fields_kernel"}
    return " + ".join(names.get(k, k) for k in kinds) + " (persistent, one launch per sigma class)"

WORKLOADS = {
    "c3": dict(desc="4096 binary blob silhouettes, sides U{64..512}, M in {16,32,64,128}, sigma in {2,3,4}, "
                    "50 iterations, fwd+bwd", n=4096, iters=50),
    "c4": dict(desc="256 weighted 512x512 images (smoothed noise, sigma 8), M=32, sigma=3, D_cs fwd+bwd",
               n=256, iters=0),
    "c2": dict(desc="one 1024x1024 binary image (ellipses + polylines), M=64, sigma=4, 100 iterations, fwd+bwd",
               n=1, iters=100),
    "c5": dict(desc="one 256x256 gray image as a 256^3 [u,v,g] lattice, sigma=(3,3,8), M=64, 100 iterations, "
                    "fwd+bwd", n=1, iters=100),
    "c1": dict(desc="one 64x64 binary image (5 ellipses), M=8, sigma=2, 50 iterations, fwd+bwd", n=1, iters=50),
}


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            return json.load(f), "measured"
    return {"hbm_gbs": FALLBACK_HBM_GBS}, "fallback"


# ------------------------------------------------------------------------------------ workload
def make_workload(name, rank, n=None):
    """Host inputs of one rank: (images, Ms, params kwargs per image, W0s, ndims, Gs, weights)."""
    from paper_1310_7114_gb300 import synth
    w = WORKLOADS[name]
    n = n or w["n"]
    if name == "c3":
        images, Ms, sig = synth.c3_batch(n, start=rank * n)
        W0s = [synth.c3_codebook(rank * n + i, im, m) for i, (im, m) in enumerate(zip(images, Ms))]
        params = [dict(sigma=float(s), iters=w["iters"]) for s in sig]
        return images, [int(m) for m in Ms], params, W0s, [2] * n, [1] * n
    if name == "c4":
        images = [synth.c4_weights(rank * n + i) for i in range(n)]
        W0s = [synth.init_codebook(synth.rng_for(4, 500_000 + rank * n + i), im, 32, 0.5) for i, im in enumerate(images)]
        return images, [32] * n, [dict(sigma=3.0, iters=0)] * n, W0s, [2] * n, [1] * n
    if name == "c2":
        images = [synth.c2_image(rank)]
        W0s = [synth.init_codebook(synth.rng_for(2, rank), images[0].astype(np.float32), 64)]
        return images, [64], [dict(sigma=4.0, iters=100)], W0s, [2], [1]
    if name == "c1":
        images = [synth.c1_image(rank)]
        W0s = [synth.init_codebook(synth.rng_for(1, rank), images[0].astype(np.float32), 8)]
        return images, [8], [dict(sigma=2.0, iters=50)], W0s, [2], [1]
    if name == "c5":
        images = [synth.c5_gray(rank)]
        W0s = [synth.init_codebook_gray(synth.rng_for(5, rank), images[0], 64)]
        return images, [64], [dict(sigma=(3.0, 3.0, 8.0), iters=100)], W0s, [3], [256]
    raise ValueError(name)


def algorithmic_field_fmas(images, params, ndims):
    """FMAs the fields pass must do: five 1-D passes of 2R+1 taps per pixel in 2-D (T, T_v; A,
    F_u, F_v); in 3-D the g pass is read off the gray value, then T, T_v, T_g along v and A, F_u,
    F_v, F_g along u: seven passes per voxel of the lattice (R from the in-plane sigma)."""
    import math
    tot = 0
    for im, p, nd in zip(images, params, ndims):
        s = p["sigma"] if np.isscalar(p["sigma"]) else p["sigma"][0]
        taps = 2 * math.ceil(3.0 * s) + 1
        if nd == 2:
            tot += 5 * taps * im.size
        else:
            tot += 7 * taps * im.size * 256
    return tot


# FP32 FMA lanes per SM per clock (4 SM sub-partitions x 32 lanes); the ALU roofline uses it with
# the SM clock sampled during the timed region.
FMA_LANES_PER_SM = 128


def algorithmic_field_bytes(images, ndims, Gs):
    """Bytes the fields pass must move: read the input once, write its fields once.
    2-D: input bytes + 3 FP32 planes per pixel; 3-D: input bytes + 4 FP32 planes per voxel."""
    tot = 0
    for im, d, G in zip(images, ndims, Gs):
        px = im.shape[0] * im.shape[1]
        tot += px * im.dtype.itemsize + (12 * px if d == 2 else 16 * px * G)
    return tot


# ---------------------------------------------------------------------------------- clocks
class ClockSampler:
    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
        time.sleep(0.3)
        return self

    def __exit__(self, *a):
        self.out = ""
        if self.proc is not None:
            time.sleep(0.25)
            self.proc.terminate()
            try:
                self.out, _ = self.proc.communicate(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
                self.out, _ = self.proc.communicate()

    def summary(self):
        rows = [r.split(", ") for r in self.out.strip().splitlines() if r.count(",") >= 7]
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"], "samples": 0}
        sm = [float(r[0]) for r in rows if r[0].replace(".", "").isdigit()]
        mx = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[4 + i].strip() == "Active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


# ------------------------------------------------------------------------------ CPU baseline
def oracle_image(im, M, p, W0, ndim, G):
    """The FP64 oracle on one image: fields, the fixed-point iterations, and the gradient."""
    import oracle
    sigma, iters = p["sigma"], p["iters"]
    if ndim == 2:
        h = im.astype(np.float64)
        A, Fu, Fv = oracle.fields2d(h, sigma)
        sxx = oracle.sxx(h, A)
        W, dcs, _, _ = oracle.lattice_run(A, [Fu, Fv], sxx, sigma, W0, iters)
        oracle.dcs_grad2d_dense(h, sigma, W, A=A)
    else:
        A, Fu, Fv, Fg = oracle.fields3d(im, G, sigma)
        occ = np.zeros((G,) + im.shape)
        uu, vv = np.meshgrid(np.arange(im.shape[0]), np.arange(im.shape[1]), indexing="ij")
        occ[im, uu, vv] = 1.0
        W, dcs, _, _ = oracle.lattice_run(A, [Fu, Fv, Fg], float((occ * A).sum()), sigma, W0, iters)
    return W


def host_cpu():
    """(cores, model) of this host: os.cpu_count() and lscpu's model name."""
    model = None
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.strip().lower().startswith("model name"):
                model = line.split(":", 1)[1].strip()
                break
    except (OSError, subprocess.SubprocessError):
        pass
    return os.cpu_count() or 1, model


def oracle_images_per_s(images, Ms, params, W0s, ndims, Gs, seconds, threads):
    """The oracle on images taken in order until about `seconds` have passed, on `threads` host
    threads (one image per thread at a time; the C oracle releases the interpreter lock, so the
    threads run on separate cores).  Returns (images done, seconds, pixels)."""
    import concurrent.futures as cf
    t0 = time.perf_counter()
    done = 0
    with cf.ThreadPoolExecutor(max_workers=threads) as ex:
        futs, nxt = set(), 0
        while nxt < len(images) and len(futs) < threads:
            futs.add(ex.submit(oracle_image, images[nxt], Ms[nxt], params[nxt], W0s[nxt], ndims[nxt], Gs[nxt]))
            nxt += 1
        while futs:
            fin, futs = cf.wait(futs, return_when=cf.FIRST_COMPLETED)
            for f in fin:
                f.result()
                done += 1
            if nxt < len(images) and time.perf_counter() - t0 < seconds:
                while nxt < len(images) and len(futs) < threads:
                    futs.add(ex.submit(oracle_image, images[nxt], Ms[nxt], params[nxt], W0s[nxt], ndims[nxt],
                                       Gs[nxt]))
                    nxt += 1
    dt = time.perf_counter() - t0
    return done, dt, sum(images[i].size for i in range(done))


def cpu_baseline(name, seconds):
    """Oracle images/s on the first images of this workload: on one thread and on every host core
    (one image per core), each for about `seconds` of work."""
    import oracle
    oracle.build()
    oracle.lib()   # loaded once before the threads start
    cores, model = host_cpu()
    images, Ms, params, W0s, ndims, Gs = make_workload(name, 0, n=min(WORKLOADS[name]["n"], 1200))
    d1, t1, px1 = oracle_images_per_s(images, Ms, params, W0s, ndims, Gs, seconds, 1)
    dn, tn, pxn = oracle_images_per_s(images, Ms, params, W0s, ndims, Gs, seconds, cores)
    return {"value": dn / tn, "unit": "images/s", "cores": cores, "kind": "oracle", "cpu_model": model,
            "sample": f"first {dn} images of the workload ({pxn} pixels), fields + iterations + gradient, FP64 C "
                      f"oracle, one image per thread on {cores} threads, {tn:.1f} s",
            "single_thread": {"value": d1 / t1, "unit": "images/s", "cores": 1,
                              "sample": f"first {d1} images ({px1} pixels), one thread, {t1:.1f} s"}}


def original_vs_lattice(name, seconds=8.0, max_images=4):
    """Context for the paper's per-iteration speed-up of lattice ITC over original ITC (Sec. 4):
    both updates in the FP64 oracle on one thread, on the first 2-D images of this workload.
    The original update (Eq. origupdate) sums over every data point for every codebook vector;
    the lattice step gathers the fields, computed once per image, and sums over codebook pairs."""
    import oracle
    images, Ms, params, W0s, ndims, Gs = make_workload(name, 0, n=min(WORKLOADS[name]["n"], max_images))
    rows, t_start = [], time.perf_counter()
    for im, M, p, W0, nd in zip(images, Ms, params, W0s, ndims):
        if nd != 2 or time.perf_counter() - t_start > seconds:
            continue
        sigma = p["sigma"]
        h = im.astype(np.float64)
        X, hx = oracle.image_points(h)
        t0 = time.perf_counter()
        A, Fu, Fv = oracle.fields2d(h, sigma)
        sxx = oracle.sxx(h, A)
        t_fields = time.perf_counter() - t0
        it = 20
        t0 = time.perf_counter()
        oracle.lattice_run(A, [Fu, Fv], sxx, sigma, W0, it)
        t_lat = (time.perf_counter() - t0) / it
        reps, t0 = 0, time.perf_counter()
        while reps < 3 and (reps == 0 or time.perf_counter() - t0 < 1.0):
            oracle.original_step(X, sigma, W0, hx)
            reps += 1
        t_orig = (time.perf_counter() - t0) / reps
        rows.append({"shape": list(im.shape), "data_points": int(X.shape[0]), "M": int(M), "sigma": float(sigma),
                     "original_ms_per_iter": 1e3 * t_orig, "lattice_ms_per_iter": 1e3 * t_lat,
                     "fields_ms_once": 1e3 * t_fields, "speedup_per_iter": t_orig / t_lat,
                     "speedup_run": p["iters"] * t_orig / (t_fields + p["iters"] * t_lat)})
    if not rows:
        return None
    return {"images": rows, "iters": int(params[0]["iters"]), "cores": 1,
            "note": "FP64 oracle, one thread; speedup_run includes the fields, computed once per image. "
                    "The paper reports about 100x per iteration (Sec. 4) on its own machine: context only"}


# ------------------------------------------------------------------------------- parity sample
def parity_sample(images, Ms, pk, n=16):
    """Indices of the timed batch checked against the oracle: its largest image, its costliest
    image (most pair work, then most pixels), and evenly spaced others."""
    B = len(images)
    size = [im.size for im in images]
    cost = [(Ms[b] * Ms[b], size[b]) for b in range(B)]
    pick = [int(np.argmax(size)), max(range(B), key=lambda b: cost[b])]
    for b in np.linspace(0, B - 1, n, dtype=int):
        if int(b) not in pick and len(pick) < n:
            pick.append(int(b))
    return sorted(set(pick))


def parity_report(images, Ms, pk, W0s, ndims, Gs, snap, idx):
    """The timed batch's results on the sampled images against the FP64 oracle, with the tests'
    bars: fields element-wise (A within 1e-5 relative, centred moments within 1e-5 R A); final
    codebooks equal where the oracle trajectory has no rounding tie (within 1e-4 of a half-integer);
    D_cs within 4e-5; the gradient at the returned codebooks normwise (1e-4), and dD/dh
    element-wise within 3e-5 of its two terms.  2-D images only (3-D: codebooks and D_cs)."""
    import concurrent.futures as cf

    import oracle
    oracle.lib()

    def one(b):
        p, nd = pk[b], ndims[b]
        sigma, iters = p["sigma"], p["iters"]
        Wg = snap["W"][b]
        r = {}
        if nd == 2:
            h = images[b].astype(np.float64)
            A, Fu, Fv = oracle.fields2d(h, sigma)
            R = oracle.radius(sigma)
            F = snap["fields"][b]
            pos = A > 0
            r["zeros_equal"] = bool(np.array_equal(F[0] == 0, A == 0))
            r["A_rel"] = float(np.max(np.abs(F[0][pos] - A[pos]) / A[pos])) if pos.any() else 0.0
            r["F_ratio"] = float(max(np.max(np.abs(F[1 + i][pos] - f[pos]) / (1e-5 * R * A[pos])) if pos.any() else 0.0
                                     for i, f in enumerate((Fu, Fv))))
            sxx = oracle.sxx(h, A)
            Wo, dcs, tie, _ = oracle.lattice_run(A, [Fu, Fv], sxx, sigma, W0s[b], iters)
            gref, ghref, sums = oracle.dcs_grad2d_dense(h, sigma, Wg.astype(np.float64), A=A)
            r["gW_rel"] = float(np.linalg.norm(snap["gW"][b] - gref) / max(np.linalg.norm(gref), 1e-300))
            gh = snap["gh"][b].astype(np.float64)
            r["gh_rel"] = float(np.linalg.norm(gh - ghref) / max(np.linalg.norm(ghref), 1e-300))
            t1 = 2.0 * A / sums[2]
            tol = 3e-5 * (np.abs(t1) + np.abs(t1 - ghref))
            err = np.abs(gh - ghref)
            r["gh_ratio"] = float(np.max(np.where(tol > 0, err / np.where(tol > 0, tol, 1.0), np.where(err > 0, np.inf, 0.0))))
        else:
            A, Fu, Fv, Fg = oracle.fields3d(images[b], Gs[b], sigma)
            occ = np.zeros((Gs[b],) + images[b].shape)
            uu, vv = np.meshgrid(np.arange(images[b].shape[0]), np.arange(images[b].shape[1]), indexing="ij")
            occ[images[b], uu, vv] = 1.0
            Wo, dcs, tie, _ = oracle.lattice_run(A, [Fu, Fv, Fg], float((occ * A).sum()), sigma, W0s[b], iters)
        r["tied"] = bool(len(tie) and tie.min() <= 1e-4)
        r["equal"] = bool(np.array_equal(Wg, Wo))
        r["dcs_err"] = None if r["tied"] else float(abs(snap["stats"][b]["dcs"] - dcs[-1]))
        return r

    with cf.ThreadPoolExecutor(max_workers=os.cpu_count() or 1) as ex:
        rows = list(ex.map(one, idx))
    two = [r for r in rows if "A_rel" in r]
    untied = [r for r in rows if not r["tied"]]
    out = {"images": len(idx), "indices": idx,
           "codebooks_equal": sum(r["equal"] for r in rows),
           "codebooks_tied": sum(r["tied"] for r in rows),
           "codebooks_differ_untied": sum((not r["equal"]) for r in untied),
           "dcs_max_abs_err": max([r["dcs_err"] for r in untied], default=None)}
    if two:
        out.update({"fields_A_max_rel_err": max(r["A_rel"] for r in two),
                    "fields_moment_max_over_bound": max(r["F_ratio"] for r in two),
                    "fields_zero_pattern_equal": all(r["zeros_equal"] for r in two),
                    "grad_W_max_rel": max(r["gW_rel"] for r in two),
                    "grad_h_max_rel": max(r["gh_rel"] for r in two),
                    "grad_h_max_over_elementwise_bound": max(r["gh_ratio"] for r in two)})
    out["bars"] = ("A 1e-5 relative; moments 1e-5 R A (ratio <= 1); codebooks equal unless the oracle "
                   "trajectory has a tie within 1e-4 of a half-integer; D_cs 4e-5; gradients normwise 1e-4, "
                   "dD/dh element-wise 3e-5 of its two terms (ratio <= 1)")
    out["note"] = ("results of the timed step on a sample of the timed batch (its largest and costliest "
                   "images and evenly spaced others), checked after the timed region")
    return out


# ----------------------------------------------------------------------------------- our arm
def segment_report(images, seg_ms, world, B, peaks, peak_src):
    """itc_segment over the batch: images/s and its bytes (input once, one int16 label per pixel)
    against the HBM copy bandwidth."""
    nbytes = sum(im.size * (im.itemsize + 2) for im in images)
    hbm = float(peaks.get("hbm_gbs", FALLBACK_HBM_GBS))
    ach = nbytes / (seg_ms / 1000.0) / 1e9
    return {"value": world * B / (seg_ms / 1000.0), "unit": "images/s", "ms": seg_ms,
            "roofline": {"bound": "hbm", "achieved": ach, "peak": hbm, "unit": "GB/s", "frac": ach / hbm,
                         "algorithmic_bytes_per_launch": nbytes, "peak_source": f"{peak_src} hbm_gbs"},
            "note": "labels by the final codebook after the timed steps; timed on its own, not part of the step"}


def chamfer_report(images, ms, world, B, peaks, peak_src):
    """itc_chamfer over the batch: images/s and its bytes (input once, one float weight per pixel)
    against the HBM copy bandwidth."""
    if ms is None:
        return None
    nbytes = sum(im.size * 5 for im in images)
    hbm = float(peaks.get("hbm_gbs", FALLBACK_HBM_GBS))
    ach = nbytes / (ms / 1000.0) / 1e9
    return {"value": world * B / (ms / 1000.0), "unit": "images/s", "ms": ms,
            "roofline": {"bound": "hbm", "achieved": ach, "peak": hbm, "unit": "GB/s", "frac": ach / hbm,
                         "algorithmic_bytes_per_launch": nbytes, "peak_source": f"{peak_src} hbm_gbs"},
            "note": "Sec. 5 weights T(X) of every binary image; one warp per image walks its rows twice; "
                    "timed on its own, not part of the step"}


def alu_roofline(images, pk, ndims, fields_ms, clocks, dev):
    """The fields pass against the FP32 FMA rate of the SMs at the clock seen under load."""
    import torch
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    mhz = clocks.get("sm_mhz") or clocks.get("sm_max_mhz") or 0.0
    fmas = algorithmic_field_fmas(images, pk, ndims)
    peak = 2.0 * FMA_LANES_PER_SM * sms * mhz * 1e6 / 1e12
    ach = 2.0 * fmas / (fields_ms / 1000.0) / 1e12
    return {"bound": "alu", "achieved": ach, "peak": peak, "unit": "TFLOP/s", "frac": ach / peak if peak else None,
            "algorithmic_fma_per_launch": fmas,
            "peak_source": f"{FMA_LANES_PER_SM} FP32 FMA lanes/SM x {sms} SMs x {mhz:.0f} MHz (median SM clock "
                           "sampled in the timed region), 2 flop/FMA",
            "note": "secondary: 5 (2-D) or 7 (3-D) x (2R+1) FMA per lattice site, the ideal count without "
                    "halo recompute; tiles and windows that hold no data are skipped, so this may exceed what "
                    "executes"}


def max_over_ranks(x, world, device):
    """The largest value of x over the ranks (the slowest rank's time); x itself on one rank."""
    if world <= 1:
        return float(x)
    import torch
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    torch.distributed.all_reduce(t, op=torch.distributed.ReduceOp.MAX)
    return float(t.item())


def run_ours(args, rank, world, local_rank):
    import torch
    from paper_1310_7114_gb300 import build, itc

    build.build()
    itc.lib()
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    name = args.workload
    images, Ms, pk, W0s, ndims, Gs = make_workload(name, rank, args.images)
    B = len(images)
    stream = torch.cuda.current_stream()

    # resident inputs: every image in one device buffer (rows padded to 16 elements)
    buf, views = itc.pack_images(images, dev)
    params = [itc.make_params(p["sigma"], 3.0, p["iters"]) for p in pk]
    plan = itc.Plan(views, Ms, params, ndims=ndims, Gs=Gs)
    # per sigma class: fields tile height, persistent CTAs per SM, staging -- timed on this batch
    tuning = plan.classes() if args.no_tune else plan.autotune(reps=3)
    if args.fields_ctas is not None:
        # leave room on every SM for the iteration CTAs of the pipelined step
        for c, info in enumerate(tuning):
            if info["staging"] == "tma":
                plan.configure(c, info["tile_h"], args.fields_ctas, "tma")
        tuning = plan.classes()
    W0 = plan.pack_W(W0s)
    W = W0.clone()
    stats = itc.new_stats(B, dev)
    gW = torch.empty_like(W)
    gh = torch.empty(plan.pixels, dtype=torch.float32, device=dev)
    ncls = len({(p["sigma"] if np.isscalar(p["sigma"]) else tuple(p["sigma"])) for p in pk})
    launches_per_step = args.chunks * (ncls + 1) + 2   # per image range: fields per class + iterations

    ev = [[torch.cuda.Event(enable_timing=True) for _ in range(4)] for _ in range(args.steps)]
    stream2 = torch.cuda.Stream(device=dev)

    def step_phases(e=None):
        """The step with its phases in sequence (events between them time each phase)."""
        W.copy_(W0)
        if e: e[0].record(stream)
        itc.run_fields(plan)
        if e: e[1].record(stream)
        itc.run_iterate(plan, W, stats)
        if e: e[2].record(stream)
        itc.backward(plan, W, grad_W=gW, grad_h=gh)
        if e: e[3].record(stream)

    def step():
        """The step as timed: fields and iterations pipelined over image ranges, then backward."""
        W.copy_(W0)
        itc.run_pipelined(plan, W, stats, stream2=stream2, chunks=args.chunks)
        itc.backward(plan, W, grad_W=gW, grad_h=gh)

    def barrier():
        if world > 1:
            torch.distributed.barrier()

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    barrier()
    t_start, t_end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(local_rank) as clk:
        torch.cuda.synchronize()
        t_start.record(stream)
        for k in range(args.steps):
            step()
        t_end.record(stream)
        torch.cuda.synchronize()
    barrier()
    # per-phase durations (same work, phases in sequence), for the roofline of the fields pass
    for _ in range(args.warmup):
        step_phases()
    torch.cuda.synchronize()
    for k in range(args.steps):
        step_phases(ev[k])
    torch.cuda.synchronize()
    ms = max_over_ranks(t_start.elapsed_time(t_end), world, dev)
    ms_step = ms / args.steps

    # the timed batch's results on a sample of its images, for the parity report (checked against
    # the oracle after every timing is done)
    snap = None
    if rank == 0 and not args.no_parity:
        pidx = parity_sample(images, Ms, pk)
        Wn, gWn, ghn = plan.unpack_W(W), plan.unpack_W(gW), plan.unpack_pixels(gh)
        snap = {"idx": pidx, "W": {b: Wn[b].copy() for b in pidx}, "gW": {b: gWn[b].copy() for b in pidx},
                "gh": {b: ghn[b].copy() for b in pidx}, "stats": itc.stats_to_numpy(stats),
                "fields": {b: plan.fields_of(b)[:, 0, :, :images[b].shape[1]].cpu().numpy().copy()
                           for b in pidx if ndims[b] == 2}}

    # the same step with the fields recomputed under a memory budget (itc_run_budget +
    # itc_backward_budget in a workspace of an eighth of the stored fields), results compared
    # with the stored-fields step bit for bit
    budget = None
    if not args.no_budget:
        ref = (W.clone(), gW.clone(), gh.clone())
        bws = itc.budget_workspace(plan, plan.ws_bytes // 8)
        bW, bgW, bgh = torch.empty_like(W), torch.empty_like(gW), torch.empty_like(gh)
        bst = itc.new_stats(B, dev)

        def budget_step():
            bW.copy_(W0)
            itc.run_budget(plan, bW, bws, bst)
            itc.backward_budget(plan, bW, bws, grad_W=bgW, grad_h=bgh)

        for _ in range(args.warmup):
            budget_step()
        torch.cuda.synchronize()
        q0, q1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        q0.record(stream)
        for _ in range(args.steps):
            budget_step()
        q1.record(stream)
        torch.cuda.synchronize()
        bms = q0.elapsed_time(q1) / args.steps
        same = bool(torch.equal(bW, ref[0]) and torch.equal(bgW, ref[1]) and torch.equal(bgh, ref[2]))
        budget = {"value": world * B / (bms / 1000.0), "unit": "images/s", "ms_per_step": bms,
                  "workspace_bytes": int(bws.numel()), "stored_workspace_bytes": int(plan.ws_bytes),
                  "time_over_stored_step": bms / ms_step, "equal_to_stored_fields_bit_for_bit": same,
                  "note": "itc_run_budget + itc_backward_budget: the fields of each image range recomputed in "
                          "a window (an eighth of the batch's fields) in the forward and again in the backward; "
                          "iterations one image per CTA per range"}
        del bws, bW, bgW, bgh, bst, ref
    f_ms = [e[0].elapsed_time(e[1]) for e in ev]
    i_ms = [e[1].elapsed_time(e[2]) for e in ev]
    b_ms = [e[2].elapsed_time(e[3]) for e in ev]

    # the same step captured once as a CUDA graph and replayed (one launch per step from the host)
    graph_ms = None
    try:
        g = torch.cuda.CUDAGraph()
        side = torch.cuda.Stream()
        side.wait_stream(stream)
        with torch.cuda.stream(side):
            step()   # warm the capture stream
        stream.wait_stream(side)
        torch.cuda.synchronize()
        with torch.cuda.graph(g):
            step()
        for _ in range(args.warmup):
            g.replay()
        torch.cuda.synchronize()
        g0, g1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        g0.record(stream)
        for _ in range(args.steps):
            g.replay()
        g1.record(stream)
        torch.cuda.synchronize()
        graph_ms = g0.elapsed_time(g1) / args.steps
        del g
    except Exception as exc:  # report, never fall back silently
        graph_ms = f"capture failed: {type(exc).__name__}: {exc}"

    # e2e through the C ABI: host inputs -> device, itc_run + itc_backward, results -> host
    host_buf = buf.cpu().pin_memory()
    host_W0 = W0.cpu().pin_memory()
    out_W = torch.empty(W.shape, dtype=W.dtype).pin_memory()
    out_gW = torch.empty(W.shape, dtype=W.dtype).pin_memory()
    out_st = torch.empty(stats.shape, dtype=stats.dtype).pin_memory()

    copy_stream = torch.cuda.Stream(device=dev)

    def e2e_step():
        # inputs from pinned host memory: the codebooks, then the images range by range on a copy
        # stream while the ranges already copied run (itc_run_staged)
        W.copy_(host_W0, non_blocking=True)
        itc.run_staged(plan, host_buf, buf, W, stats, chunks=args.e2e_chunks, copy_stream=copy_stream)
        itc.backward(plan, W, grad_W=gW, grad_h=gh)
        out_W.copy_(W, non_blocking=True)
        out_gW.copy_(gW, non_blocking=True)
        out_st.copy_(stats, non_blocking=True)

    for _ in range(args.warmup):
        e2e_step()
    torch.cuda.synchronize()
    barrier()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        e2e_step()
    e1.record(stream)
    torch.cuda.synchronize()
    e2e_single_ms = max_over_ranks(e0.elapsed_time(e1) / args.steps, world, dev)
    h2d = buf.numel() * buf.element_size() + W0.numel() * 4
    d2h = 2 * W.numel() * 4 + stats.numel()

    # the same per step, as a stream of batches would run it: two image buffers and two plans, the
    # copies of step k+1 (copy stream) overlapping the work of step k; every step still copies its
    # inputs from pinned host memory and reads its results back
    buf2, views2 = itc.pack_images(images, dev)
    plan2 = itc.Plan(views2, Ms, params, ndims=ndims, Gs=Gs)
    for c, info in enumerate(tuning):
        if info["staging"] in ("tma", "plain") and plan2.classes()[c]["staging"] in ("tma", "plain"):
            plan2.configure(c, info["tile_h"], info["ctas_per_sm"], info["staging"])
    sets = [(plan, buf, W, stats, gW, gh), (plan2, buf2, torch.empty_like(W), itc.new_stats(B, dev),
                                            torch.empty_like(gW), torch.empty_like(gh))]
    host_out = [(out_W, out_gW, out_st),
                (torch.empty_like(out_W).pin_memory(), torch.empty_like(out_gW).pin_memory(),
                 torch.empty_like(out_st).pin_memory())]
    copied = [torch.cuda.Event(), torch.cuda.Event()]
    released = [torch.cuda.Event(), torch.cuda.Event()]

    def stage(k):   # the image copy of step k, on the copy stream, once step k-2 has released the buffer
        _, bk, Wk, _, _, _ = sets[k % 2]
        copy_stream.wait_event(released[k % 2])
        with torch.cuda.stream(copy_stream):
            bk.copy_(host_buf, non_blocking=True)
            Wk.copy_(host_W0, non_blocking=True)
        copied[k % 2].record(copy_stream)

    def compute(k):
        pk_, _, Wk, stk, gWk, ghk = sets[k % 2]
        stream.wait_event(copied[k % 2])
        itc.run(pk_, Wk, stk)
        itc.backward(pk_, Wk, grad_W=gWk, grad_h=ghk)
        oW, ogW, ost = host_out[k % 2]
        oW.copy_(Wk, non_blocking=True)
        ogW.copy_(gWk, non_blocking=True)
        ost.copy_(stk, non_blocking=True)
        released[k % 2].record(stream)   # the buffers of this step may be refilled after the read-back

    def first_step():   # step 0 has no step before it to hide its copy under: its image ranges
        # are copied on the copy stream and each range's fields start as soon as it has landed
        pk_, bk, Wk, stk, gWk, ghk = sets[0]
        stream.wait_event(released[0])
        Wk.copy_(host_W0, non_blocking=True)
        itc.run_staged(pk_, host_buf, bk, Wk, stk, chunks=args.e2e_chunks, copy_stream=copy_stream)
        itc.backward(pk_, Wk, grad_W=gWk, grad_h=ghk)
        oW, ogW, ost = host_out[0]
        oW.copy_(Wk, non_blocking=True)
        ogW.copy_(gWk, non_blocking=True)
        ost.copy_(stk, non_blocking=True)
        released[0].record(stream)

    def stream_steps(n):
        first_step()
        for k in range(1, n):
            stage(k)   # on the copy stream behind the copies of step k - 1: under step k - 1's work
            compute(k)

    for b_ in range(2):
        released[b_].record(stream)
    stream_steps(args.warmup)
    torch.cuda.synchronize()
    barrier()
    e0.record(stream)
    stream_steps(args.steps)
    e1.record(stream)
    torch.cuda.synchronize()
    e2e_ms = max_over_ranks(e0.elapsed_time(e1) / args.steps, world, dev)
    same = bool(torch.equal(sets[0][2], sets[1][2]))
    del plan2, buf2, sets

    # the same work launched image by image (one plan per image), on a prefix of the batch
    # segmentation of every image by its final codebook (outside the step), its own timing
    labels = torch.empty(plan.pixels, dtype=torch.int16, device=dev)
    for _ in range(args.warmup):
        itc.segment(plan, W, labels)
    torch.cuda.synchronize()
    s0, s1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    s0.record(stream)
    for _ in range(args.steps):
        itc.segment(plan, W, labels)
    s1.record(stream)
    torch.cuda.synchronize()
    seg_ms = s0.elapsed_time(s1) / args.steps

    # Sec. 5 chamfer weights of every binary image (outside the step), its own timing
    cham = None
    if all(im.dtype == np.uint8 for im in images) and all(n == 2 for n in ndims) and max(im.shape[1] for im in images) <= 1024:
        cbuf = torch.zeros(max(int(itc.lib().itc_plan_padded_offset(plan.host_ptr, B)), 4), dtype=torch.float32,
                           device=dev)
        for _ in range(args.warmup):
            itc.chamfer(plan, cbuf, views=False)
        torch.cuda.synchronize()
        c0, c1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        c0.record(stream)
        for _ in range(args.steps):
            itc.chamfer(plan, cbuf, views=False)
        c1.record(stream)
        torch.cuda.synchronize()
        cham = c0.elapsed_time(c1) / args.steps
        del cbuf

    # Algorithm 1's own stopping test (step 11, theta = 0: stop once no codebook moves), same
    # images and step otherwise; the codebooks equal those of the full iteration count
    stop = None
    if WORKLOADS[name]["iters"] > 0:
        pparams = [itc.make_params(p["sigma"], 3.0, p["iters"], flags=itc.ITC_STOP_ON_FIXED) for p in pk]
        pplan = itc.Plan(views, Ms, pparams, ndims=ndims, Gs=Gs)
        for c, info in enumerate(tuning):   # the tuned fields configuration of the main plan
            if info["staging"] in ("tma", "plain") and pplan.classes()[c]["staging"] in ("tma", "plain"):
                pplan.configure(c, info["tile_h"], info["ctas_per_sm"], info["staging"])
        pW = pplan.pack_W(W0s)
        pst = itc.new_stats(B, dev)
        pgW = torch.empty_like(pW)

        def stop_step():
            pW.copy_(W0)
            itc.run(pplan, pW, pst)
            itc.backward(pplan, pW, grad_W=pgW, grad_h=gh)

        for _ in range(args.warmup):
            stop_step()
        torch.cuda.synchronize()
        p0, p1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        p0.record(stream)
        for _ in range(args.steps):
            stop_step()
        p1.record(stream)
        torch.cuda.synchronize()
        pms = p0.elapsed_time(p1) / args.steps
        done = itc.stats_to_numpy(pst)["iters_done"]
        same = bool(torch.equal(pW, W))
        stop = {"value": world * B / (pms / 1000.0), "unit": "images/s", "ms_per_step": pms,
                "iters_done_mean": float(np.mean(done)), "iters_done_max": int(np.max(done)),
                "codebooks_equal_full_run": same,
                "note": "ITC_STOP_ON_FIXED: Algorithm 1 step 11 with theta = 0; not the headline (the workload "
                        "fixes the iteration count)"}
        del pplan, pW, pst, pgW

    # the paper's width schedule of Sec. 4 (omega = sqrt(N/M)/2, xi = omega/2 per image) on the
    # same images: its widths are far beyond the masks, so the fields come from the recursive
    # filters; fields + iterations (the adjoint needs mask fields), timed on their own
    sched = None
    if name == "c3" and not args.no_schedule:
        sparams = [itc.params_parzen(2, mass=float(im.sum()), M=int(m), iters=WORKLOADS[name]["iters"],
                                     flags=itc.ITC_RECURSIVE) for im, m in zip(images, Ms)]
        splan = itc.Plan(views, Ms, sparams)
        sW0 = splan.pack_W(W0s)
        sW = sW0.clone()
        sst = itc.new_stats(B, dev)
        for _ in range(args.warmup):
            sW.copy_(sW0)
            itc.run(splan, sW, sst)
        torch.cuda.synchronize()
        q0, q1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        q0.record(stream)
        for _ in range(args.steps):
            sW.copy_(sW0)
            itc.run(splan, sW, sst)
        q1.record(stream)
        torch.cuda.synchronize()
        sms = q0.elapsed_time(q1) / args.steps
        taus = [p.sigma[0] for p in sparams]
        sched = {"value": world * B / (sms / 1000.0), "unit": "images/s", "ms": sms,
                 "tau_px": {"min": float(min(taus)), "median": float(np.median(taus)), "max": float(max(taus))},
                 "note": "Sec. 4 schedule (omega = sqrt(N/M)/2, xi = omega/2), fields by recursive filtering "
                         "(ITC_RECURSIVE) + 50 iterations per image; no adjoint"}
        del splan, sW0, sW, sst

    per_image = None
    if not args.no_per_image and rank == 0:
        n_pi = min(B, args.per_image_n)
        plans = [itc.Plan([views[b]], [Ms[b]], params[b], ndims=[ndims[b]], Gs=[Gs[b]]) for b in range(n_pi)]
        Ws = [p.pack_W([W0s[b]]) for b, p in enumerate(plans)]
        sts = [itc.new_stats(1, dev) for _ in plans]
        gWs = [torch.empty_like(w) for w in Ws]
        ghs = [torch.empty(p.pixels, dtype=torch.float32, device=dev) for p in plans]

        def pi_pass():
            for b in range(n_pi):
                itc.run(plans[b], Ws[b], sts[b])
                itc.backward(plans[b], Ws[b], grad_W=gWs[b], grad_h=ghs[b])

        pi_pass()
        torch.cuda.synchronize()
        p0, p1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        p0.record(stream)
        pi_pass()
        p1.record(stream)
        torch.cuda.synchronize()
        pms = p0.elapsed_time(p1)
        per_image = {"value": n_pi / (pms / 1000.0), "unit": "images/s", "images": n_pi,
                     "launches_per_image": 4,
                     "note": "one plan per image, itc_run + itc_backward per image, same stream"}
        del plans, Ws, sts, gWs, ghs

    if rank != 0:
        return None

    peaks, peak_src = measured_peaks()
    fbytes = algorithmic_field_bytes(images, ndims, Gs)
    traffic, traffic_note = fields_traffic(name, sum(im.size * (G if d == 3 else 1)
                                                     for im, d, G in zip(images, ndims, Gs)))
    f_avg = statistics.mean(f_ms)
    achieved = fbytes / (f_avg / 1000.0) / 1e9
    hbm = float(peaks.get("hbm_gbs", FALLBACK_HBM_GBS))
    value = world * B / (ms_step / 1000.0)
    res = {
        "metric": METRIC,
        "value": value,
        "unit": "images/s",
        "n_gpus": world,
        "steps": args.steps,
        "warmup": args.warmup,
        "ms_per_step": ms_step,
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "f32",
        "data": "synthetic (seeded stand-ins for the paper's MPEG-7 shapes, which are not available)",
        "config": {"workload": f"{name}: {WORKLOADS[name]['desc']}", "images_per_gpu": B,
                   "pixels_per_gpu": int(sum(im.size for im in images)),
                   "l2": "inputs larger than L2 (packed images %.0f MB, fields %.0f MB per step)"
                         % (buf.numel() * buf.element_size() / 1e6, plan.ws_bytes / 1e6),
                   "parallelism": f"replicas x{world} (independent images per GPU, no collective)",
                   "fields_tuning": [{k: c[k] for k in ("sigma", "images", "tile_h", "ctas_per_sm", "staging",
                                                        "tuned_ms")} for c in tuning]},
        "segment": segment_report(images, seg_ms, world, B, peaks, peak_src),
        "chamfer": chamfer_report(images, cham, world, B, peaks, peak_src),
        "schedule": sched,
        "stop_on_fixed": stop,
        "phases_ms": {"fields": f_avg, "iterate": statistics.mean(i_ms), "backward": statistics.mean(b_ms),
                      "note": "phases run in sequence in a separate timed loop; the headline step overlaps "
                              f"fields and iterations over {args.chunks} image ranges on two streams"},
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": hbm, "unit": "GB/s",
                     "frac": achieved / hbm, "traffic": traffic, "traffic_note": traffic_note,
                     "kernel": "fields pass: " + fields_kernel_name(ndims, tuning),
                     "algorithmic_bytes_per_launch": fbytes, "peak_source": f"{peak_src} hbm_gbs"},
        "roofline_alu": alu_roofline(images, pk, ndims, f_avg, clk.summary(), dev),
        "e2e": {"value": world * B / (e2e_ms / 1000.0), "unit": "images/s", "h2d_bytes_per_step": int(h2d),
                "d2h_bytes_per_step": int(d2h), "ms_per_step": e2e_ms,
                "pipeline": "two image buffers and plans: the host-to-device copy of step k+1 runs on a copy "
                            "stream while step k computes (itc_run + itc_backward); the first step copies its "
                            "images range by range under its own fields (itc_run_staged); both buffers give "
                            f"the same codebooks: {same}",
                "single_buffer": {"value": world * B / (e2e_single_ms / 1000.0), "ms_per_step": e2e_single_ms,
                                  "path": "itc_run_staged: the copy overlaps only this step's fields"},
                "path": "inputs from pinned host memory every step (images and codebooks), results (W, grad_W, "
                        "stats) back to pinned host memory every step, through the C ABI"},
        "graph": ({"value": world * B / (graph_ms / 1000.0), "unit": "images/s", "ms_per_step": graph_ms,
                   "note": "the same step captured in one CUDA graph and replayed"}
                  if isinstance(graph_ms, float) else {"error": graph_ms}),
        "gpu_launches": launches_per_step * args.steps,
        "clocks": clk.summary(),
    }
    if per_image:
        res["per_image_launch"] = per_image
        res["batched_over_per_image"] = value / world / per_image["value"]
    if budget:
        res["budget"] = budget
    if snap is not None:
        res["parity"] = parity_report(images, Ms, pk, W0s, ndims, Gs, snap, snap["idx"])
    if not args.no_cpu_baseline and world == 1:
        res["cpu_baseline"] = cpu_baseline(name, args.cpu_seconds)
        ovl = original_vs_lattice(name)
        if ovl:
            res["cpu_baseline"]["original_vs_lattice"] = ovl
    return res


# ------------------------------------------------------------------------------ reference arm
def run_reference(args, rank):
    """The FP64 oracle, as it stands, on this host's cores: each step runs a bounded sample of the
    workload (the first --ref-images images)."""
    if rank != 0:
        return None
    import concurrent.futures as cf

    import oracle
    oracle.build()
    oracle.lib()
    name = args.workload
    cores, model = host_cpu()
    n = min(args.ref_images or 2 * cores, WORKLOADS[name]["n"])
    images, Ms, pk, W0s, ndims, Gs = make_workload(name, 0, n=max(n, 1))
    pool = cf.ThreadPoolExecutor(max_workers=cores)

    def step():   # one image per host thread at a time (the C oracle releases the interpreter lock)
        list(pool.map(lambda b: oracle_image(images[b], Ms[b], pk[b], W0s[b], ndims[b], Gs[b]), range(n)))

    for _ in range(args.warmup):
        step()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        step()
    dt = (time.perf_counter() - t0) / args.steps
    pool.shutdown()
    v = n / dt
    return {
        "impl": "reference", "metric": METRIC, "value": v, "unit": "images/s", "n_gpus": 1,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt * 1000.0, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": f"{name}: {WORKLOADS[name]['desc']}", "images_per_step": n},
        "cpu_baseline": {"value": v, "unit": "images/s", "cores": cores, "kind": "oracle", "cpu_model": model,
                         "sample": f"first {n} images of the workload per step, FP64 C oracle, one image per "
                                   f"thread on {cores} threads"},
        "e2e": {"value": v, "unit": "images/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", choices=sorted(WORKLOADS), default="c3")
    ap.add_argument("--images", type=int, default=None)
    ap.add_argument("--per-image-n", type=int, default=512)
    ap.add_argument("--no-per-image", action="store_true")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-seconds", type=float, default=8.0)
    ap.add_argument("--ref-images", type=int, default=None, help="images per reference step (default 2 x cores)")
    ap.add_argument("--no-tune", action="store_true", help="keep the default fields configuration")
    ap.add_argument("--e2e-chunks", type=int, default=4, help="image ranges of the staged end-to-end step")
    ap.add_argument("--no-schedule", action="store_true", help="skip the Sec. 4 width-schedule timing")
    ap.add_argument("--fields-ctas", type=int, default=None,
                    help="persistent fields CTAs per SM after tuning (room for overlapping iterations)")
    ap.add_argument("--chunks", type=int, default=1, help="image ranges of the pipelined fields/iterations")
    ap.add_argument("--no-parity", action="store_true", help="skip the oracle check of a sample of the timed batch")
    ap.add_argument("--no-budget", action="store_true", help="skip the step with the fields recomputed under a budget")
    args = ap.parse_args()
    args.warmup = max(args.warmup, 3) if args.impl == "ours" else max(args.warmup, 1)

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        res = run_reference(args, rank)
    else:
        if world > 1:
            import torch
            torch.cuda.set_device(local_rank)
            torch.distributed.init_process_group("nccl")
        res = run_ours(args, rank, world, local_rank)
        if world > 1:
            import torch
            torch.distributed.destroy_process_group()
    if res is not None:
        print(json.dumps(res), flush=True)


if __name__ == "__main__":
    main()
