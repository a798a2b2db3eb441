"""The work that users of the framework have it do, as cases to measure.

Each case is one call (or one short sequence of calls) through the public
entry points (the Python classes, or the C ABI as bound for a program that
keeps its own buffers), on inputs made from a seed:

path      process_batch: correction, integration, clipping, kept lists, peaks
mixed     sep_process_mixed: the same on a stream of several detectors' frames
host      process_host: the same from pinned host memory to host memory
clip      integrate_clip alone (profiles without sparsification)
correct   corrected frames
compress  sparsify, then densify: the stored form of a batch and back
densify   dense frames from stored profiles and kept lists
grad      loss and gradient of the surrogate network on recorded rows

The detectors are those of the benchmark and the tests (a 256 x 256 frame and
the Jungfrau 1M, 4M and 16M layouts) and plain rectangles of any size; the
frames follow the same recipe (a ring background of 0.05 to 5 photons, Poisson
counts, Bragg spots on some frames, raw words with three gain levels).
`exact` states every step again in binary64 with torch alone.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2411_09515_gb300 import (SEP_CUTOFF_CHAUVENET, SEP_DTYPE_F32, SEP_ERROR_AZIMUTHAL, SEP_ERROR_HYBRID,
                                    SEP_ERROR_POISSON, SEP_PREC_DWORD, SEP_PREC_FP64MERGE, SEP_PREC_KAHAN,
                                    SEP_PREC_PLAIN, SEP_UNIT_Q_NM, Context, Separator, Surrogate)
from paper_2411_09515_gb300 import _binding as C_ABI

DEV = "cuda"
PRECISIONS = {"plain": SEP_PREC_PLAIN, "kahan": SEP_PREC_KAHAN, "fp64merge": SEP_PREC_FP64MERGE,
              "dword": SEP_PREC_DWORD}
MODELS = {"azimuthal": SEP_ERROR_AZIMUTHAL, "poisson": SEP_ERROR_POISSON, "hybrid": SEP_ERROR_HYBRID}
DARK_VAR = 0.04          # dark variance of the Poisson and hybrid models, photons^2
N_ITER, K_CLIP, K_PICK = 5, 3.0, 3.0
PIXEL_M, DIST_M, LAMBDA_M = 75e-6, 0.150, 1.0e-10
PED, PED_STD, GAIN = (1500.0, 14000.0, 15000.0), (50.0, 200.0, 200.0), (40.0, -1.5, -0.1)

# name: rows, columns, module grid (rows x columns of 514 x 1030 modules; 0: no mask), bins
LAYOUTS = {"256": (256, 256, 0, 0, 64), "1M": (1064, 1030, 2, 1, 600), "4M": (2164, 2068, 4, 2, 1000),
           "16M": (4362, 4148, 8, 4, 2000)}
MIXED = ("1M", "4M", "16M")   # detectors of the mixed stream, frames 3 : 2 : 1


def _detector(kind, layout, **kw):
    rows, cols, mr, mc, nbins = LAYOUTS[layout]
    c = {"kind": kind, "rows": rows, "cols": cols, "modules_y": mr, "modules_x": mc, "nbins": nbins, "split": 1,
         "raw": False, "norm": False, "precision": "dword", "model": "azimuthal", "chauvenet": False,
         "smooth": False, "side_stream": False}
    c.update(kw)
    return c


def listed():
    return [
        # one small photon-counting frame, as a viewer or a beam-centre scan asks for it: launches and latency
        dict(_detector("path", "256", frames=1, side_stream=True), name="path_256_f32_1"),
        # online analysis of a running detector: a few raw Jungfrau 4M frames as they arrive
        dict(_detector("path", "4M", frames=4, split=2, raw=True, side_stream=True), name="path_4M_raw_4"),
        # the benchmark's workload: a large batch of raw Jungfrau 4M frames, throughput
        dict(_detector("path", "4M", frames=512, split=2, raw=True), name="path_4M_raw_512"),
        # an odd-sized photon-counting detector, cut-off by set size, thresholds from the smooth background
        dict(_detector("path", "256", rows=1031, cols=1065, nbins=401, frames=29, chauvenet=True, smooth=True),
             name="path_odd_f32_smooth_29"),
        # profiles with a flat-field and solid-angle norm in compensated arithmetic
        dict(_detector("clip", "1M", frames=67, split=2, raw=True, norm=True, precision="kahan"),
             name="clip_1M_norm_kahan_67"),
        # profiles with exact pixel areas and the hybrid error model, ragged size
        dict(_detector("clip", "256", rows=619, cols=487, nbins=211, frames=131, split=0, model="hybrid"),
             name="clip_ragged_area_hybrid_131"),
        # frames of three detectors in one call
        {"kind": "mixed", "frames": 18, "name": "mixed_f32_18"},
        # end to end from an acquisition's pinned buffers
        dict(_detector("host", "4M", frames=16, split=2, raw=True), name="host_4M_raw_16"),
        # corrected frames for another program (an indexer, a viewer)
        dict(_detector("correct", "4M", frames=64, split=2, raw=True), name="correct_4M_raw_64"),
        # compression with given profiles and the dense frames back, to check the loss
        dict(_detector("compress", "4M", frames=48, split=2, raw=True), name="compress_4M_raw_48"),
        # decompression of stored frames with a smooth and noisy background
        dict(_detector("densify", "4M", frames=64, split=2, smooth=True, noise=True), name="densify_4M_smooth_noise_64"),
        # one training step's gradient of the surrogate
        {"kind": "grad", "rows": 16384, "name": "grad_16384"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["path", "path", "path", "clip", "clip", "mixed", "host", "correct", "compress", "densify",
                       "grad"])
    if kind == "grad":
        return {"kind": kind, "rows": _log(rng, 500, 300000)}
    if kind == "mixed":
        return {"kind": kind, "frames": rng.randint(3, 19)}
    layout = rng.choice(["256", "1M", "4M", "", ""])
    raw = rng.random() < 0.5
    c = _detector(kind, layout or "256", raw=raw, split=rng.choice([1, 2, 2, 0]))
    if not layout:
        c["rows"], c["cols"] = _log(rng, 120, 2200), _log(rng, 120, 2200)
    npix = c["rows"] * c["cols"]
    if layout != "4M" or c["split"] == 0:
        # any number of bins whose longest row stays well inside the library's limit
        fewest = max(24, int(npix * (4e-4 if c["split"] == 0 else 1.3e-4)))
        c["nbins"] = max(fewest, _log(rng, 30, 1200))
    most = {"host": 24, "clip": 160}.get(kind, 96)
    c["frames"] = max(1, min(_log(rng, 1, 400), int(most * 4.5e6 / npix)))
    if kind in ("path", "clip", "host"):
        c["precision"] = rng.choice(["dword", "dword", "plain", "kahan", "fp64merge"])
        c["chauvenet"] = rng.random() < 0.25
        c["norm"] = rng.random() < 0.25
        if not c["norm"]:
            c["model"] = rng.choice(["azimuthal", "azimuthal", "poisson", "hybrid"])
    if kind in ("correct", "compress"):
        c["norm"] = rng.random() < 0.25
    if kind in ("path", "compress", "densify"):
        c["smooth"] = rng.random() < 0.3
    if kind == "path":
        c["side_stream"] = rng.random() < 0.5
    if kind == "densify":
        c["noise"], c["raw"] = rng.random() < 0.6, False
    return c


# ---- what a user's program has in hand ------------------------------------

def _generator(*seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(np.random.SeedSequence([int(x) & 0xFFFFFFFF for x in seed]).generate_state(2, np.uint64)[0] >> 1))
    return g


def _center(c):
    """Beam centre (x = column, y = row), a little off the middle."""
    if (c["rows"], c["cols"]) == (2164, 2068):
        return 1040.3, 1090.7
    return c["cols"] / 2 + 0.3, c["rows"] / 2 + 0.7


def _mask(rows, cols, mr, mc):
    """1 where there is no pixel: the gaps between modules of 514 x 1030 and between their 2 x 4 chips."""
    m = np.zeros((rows, cols), np.uint8)
    if mr == 0:
        return m.reshape(-1)
    m[:] = 1
    gap_y = (rows - mr * 514) // (mr - 1) if mr > 1 else 0
    gap_x = (cols - mc * 1030) // (mc - 1) if mc > 1 else 0
    ys = [y for y in range(514) if y not in (256, 257)]
    xs = [x for x in range(1030) if x not in (256, 257, 514, 515, 772, 773)]
    for i in range(mr):
        for j in range(mc):
            m[np.ix_([i * (514 + gap_y) + y for y in ys], [j * (1030 + gap_x) + x for x in xs])] = 0
    return m.reshape(-1)


DET_KEYS = ("rows", "cols", "modules_y", "modules_x")


@functools.lru_cache(maxsize=8)
def _planes(rows, cols, mr, mc):
    """The detector's mask (host), pedestals, gains and norm (device), the same for every seed of frames."""
    g = _generator(rows, cols, 7)
    n = rows * cols
    ped = torch.stack([m + s * torch.randn(n, generator=g, device=DEV) for m, s in zip(PED, PED_STD)])
    gain = torch.stack([m * (1 + 0.02 * (2 * torch.rand(n, generator=g, device=DEV) - 1)) for m in GAIN])
    norm = 0.5 + torch.rand(n, generator=g, device=DEV)
    return _mask(rows, cols, mr, mc), ped, gain, norm


def _key(c):
    return tuple(sorted((k, v) for k, v in c.items() if k not in ("name", "kind", "frames", "side_stream", "noise")))


@functools.lru_cache(maxsize=4)
def _separator(key, context=None):
    """A program's handle: one per detector and set of parameters, kept from batch to batch."""
    c = dict(key)
    mask, ped, gain, norm = _planes(*(c[k] for k in DET_KEYS))
    geometry = dict(rows=c["rows"], cols=c["cols"], pixel_m=(PIXEL_M, PIXEL_M), dist_m=DIST_M, center_px=_center(c),
                    wavelength_m=LAMBDA_M, unit=SEP_UNIT_Q_NM, nbins=c["nbins"], split=c["split"],
                    range=(math.nan, math.nan))
    sep = Separator(geometry, mask=mask, norm=norm.cpu().numpy() if c["norm"] else None,
                    calib=(ped.cpu().numpy(), gain.cpu().numpy()) if c["raw"] else None, n_iter=N_ITER,
                    k_clip=K_CLIP, k_pick=K_PICK, precision=PRECISIONS[c["precision"]], context=context)
    sep.set_params(error_model=MODELS[c["model"]], interpolate=int(c["smooth"]))
    if c["model"] != "azimuthal":
        sep.set_params(dark_var=DARK_VAR)
    if c["chauvenet"]:
        sep.set_params(cutoff=SEP_CUTOFF_CHAUVENET)
    return sep


@functools.lru_cache(maxsize=1)
def _mixed_separators():
    context = Context(0)
    return [_separator.__wrapped__(_key(_detector("mixed", name)), context) for name in MIXED]


@functools.lru_cache(maxsize=1)
def _side_stream():
    return torch.cuda.Stream()


def _profile(c):
    """The solvent background at every pixel: an exponential fall-off and three rings."""
    cx, cy = _center(c)
    y = torch.arange(c["rows"], device=DEV, dtype=torch.float32) + 0.5
    x = torch.arange(c["cols"], device=DEV, dtype=torch.float32) + 0.5
    r = torch.sqrt((y[:, None] - cy) ** 2 + (x[None, :] - cx) ** 2).reshape(-1) / (0.25 * (c["rows"] + c["cols"]))
    rings = ((0.8, 0.35, 0.05), (1.0, 0.6, 0.08), (0.5, 0.9, 0.12))
    return torch.exp(-r / 0.4) + sum(a * torch.exp(-0.5 * ((r - m) / s) ** 2) for a, m, s in rings)


def _scales(c, seed, n):
    """Each frame's background level."""
    g = _generator(seed, c["rows"], c["cols"], 5)
    return torch.exp(torch.rand(n, generator=g, device=DEV) * math.log(6.0) + math.log(0.5))


def _photons(c, seed, n):
    """n frames' photon counts (float32 [n][pixels], 0 where masked), a few frames at a time."""
    rows, cols = c["rows"], c["cols"]
    g = _generator(seed, rows, cols, 1)
    profile, scales = _profile(c), _scales(c, seed, n)
    valid = torch.from_numpy(_mask(*(c[k] for k in DET_KEYS)) == 0).to(DEV)
    dy, dx = torch.meshgrid(torch.arange(-4, 5, device=DEV), torch.arange(-4, 5, device=DEV), indexing="ij")
    step = max(1, min(n, int(3e8) // (rows * cols)))
    for f0 in range(0, n, step):
        m = min(step, n - f0)
        rate = (scales[f0:f0 + m, None] * profile[None]).clamp_(0.05, 5.0)
        # spots on three frames of ten: 10 to 1e4 photons, 0.8 to 1.5 px wide, the number by the detector's size
        u = torch.rand(m, generator=g, device=DEV)
        ns = int(min(300, max(12, rows * cols / 15000)))
        sy = torch.rand((m, ns), generator=g, device=DEV) * (rows - 10) + 5
        sx = torch.rand((m, ns), generator=g, device=DEV) * (cols - 10) + 5
        amp = torch.exp(torch.rand((m, ns), generator=g, device=DEV) * math.log(1e3) + math.log(10.0))
        sig = 0.8 + 0.7 * torch.rand((m, ns), generator=g, device=DEV)
        amp = amp * (u < 0.3)[:, None] / (2 * math.pi * sig ** 2)
        py, px = sy.long()[..., None, None] + dy, sx.long()[..., None, None] + dx
        d2 = (py + 0.5 - sy[..., None, None]) ** 2 + (px + 0.5 - sx[..., None, None]) ** 2
        spot = amp[..., None, None] * torch.exp(-0.5 * d2 / sig[..., None, None] ** 2)
        at = torch.arange(m, device=DEV)[:, None, None, None] * (rows * cols) + py * cols + px
        extra = torch.zeros_like(rate)   # (where spots overlap, the brighter one)
        extra.view(-1).scatter_reduce_(0, at.reshape(-1), spot.reshape(-1), "amax")
        rate += extra
        yield f0, m, torch.poisson(rate, generator=g) * valid, g


def _frames(c, seed, n):
    """n frames as the detector delivers them: float32 photons, or raw words (int16 bits) with gain levels."""
    npix = c["rows"] * c["cols"]
    out = torch.empty((n, npix), dtype=torch.int16 if c["raw"] else torch.float32, device=DEV)
    if c["raw"]:
        mask, ped, gain, _ = _planes(*(c[k] for k in DET_KEYS))
        valid = torch.from_numpy(mask == 0).to(DEV)
    for f0, m, q, g in _photons(c, seed, n):
        if not c["raw"]:
            out[f0:f0 + m] = q
            continue
        low, high = ped[0] + GAIN[0] * q > 16000.0, q > 9000.0
        word = torch.where(low, ped[1] + gain[1] * q, ped[0] + gain[0] * q)
        word = torch.where(high, ped[2] + gain[2] * q, word)
        word += 10.0 * torch.randn(q.shape, generator=g, device=DEV)
        word = word.round_().clamp_(0, 16383).int()
        word += torch.where(high, 3 << 14, torch.where(low, 1 << 14, 0)).int()
        out[f0:f0 + m] = torch.where(valid, word, 0).short()
    return out


def _capacities(c):
    """Room for the kept pixels (the Poisson deviation keeps several times more) and the peaks of a frame."""
    npix = c["rows"] * c["cols"]
    few = c.get("model", "azimuthal") == "azimuthal"
    return max(4096, npix // (24 if few else 2)), max(1024, npix // (512 if few else 64))


def _levels(c, seed, n):
    """Stored background profiles of the frames: mean and deviation by bin."""
    q = _radial(c, 0.5, 0.5)
    bins = ((q - q.min()) / (q.max() - q.min()) * c["nbins"]).long().clamp_(0, c["nbins"] - 1)
    level = torch.bincount(bins, weights=_profile(c).double(), minlength=c["nbins"])
    level = (level / torch.bincount(bins, minlength=c["nbins"]).clamp(min=1)).float()
    g = _generator(seed, c["rows"], c["cols"], 2)
    mean = (_scales(c, seed, n)[:, None] * level[None]).clamp_(0.05, 5.0)
    mean *= 1 + 0.005 * torch.randn(mean.shape, generator=g, device=DEV)
    sigma = (mean + 0.0625).sqrt() * (1 + 0.01 * torch.randn(mean.shape, generator=g, device=DEV))
    return mean, sigma


def prepare(case, seed):
    c = dict(case)
    s = {"case": c}
    kind, n = c["kind"], c.get("frames", 0)
    if kind == "grad":
        g = _generator(seed, c["rows"], 3)
        s["x"] = torch.randn((c["rows"], 20), generator=g, device=DEV)
        s["t"] = 0.3 * torch.randn((c["rows"], 2), generator=g, device=DEV) + 0.2 * s["x"][:, :2]
        s["model"] = Surrogate(Context(0), seed=1)
        s["model"].params(_weights(seed))
    elif kind == "mixed":
        s["seps"] = _mixed_separators()
        s["frames"] = []
        for d, m in enumerate(_mixed_counts(n)):
            x = _frames(_detector("mixed", MIXED[d]), seed, m)
            s["frames"] += [(d, SEP_DTYPE_F32, x[i]) for i in range(m)]
        s["kept"], s["peaks"] = 1 << 20, 1 << 15
        o = s["seps"][0].alloc_outputs(len(s["frames"]), s["kept"], s["peaks"])
        for k in ("mean", "sigma", "count"):   # rows of all frames, one after another
            o[k] = o[k].new_empty(sum(s["seps"][d].nbins for d, _, _ in s["frames"]))
        s["out"] = {k: v.zero_() for k, v in o.items()}
    else:
        s["sep"] = sep = _separator(_key(c))
        kept, peaks = s["kept"], s["peaks"] = _capacities(c)
        if kind != "densify":
            s["frames"] = _frames(c, seed, n)
        if kind in ("path", "host"):
            out = sep.alloc_outputs(n, kept, peaks) if kind == "path" else sep.alloc_host_outputs(n, kept, peaks)
            s["out"] = {k: v.zero_() for k, v in out.items()}
            s["stream"] = _side_stream() if c["side_stream"] else None
        if kind == "host":
            s["frames"] = s["frames"].cpu().pin_memory()
        if kind in ("compress", "densify"):
            s["mean"], s["sigma"] = _levels(c, seed, n)
            s["dense"] = torch.zeros((n, sep.npix), dtype=torch.float32, device=DEV)
        if kind == "densify":
            g = _generator(seed, c["rows"], c["cols"], 4)
            valid = torch.from_numpy(_planes(*(c[k] for k in DET_KEYS))[0] == 0).to(DEV)
            s["idx"] = torch.zeros((n, kept), dtype=torch.int32, device=DEV)
            s["n_kept"] = torch.zeros(n, dtype=torch.int32, device=DEV)
            for f in range(n):
                i = ((torch.rand(sep.npix, generator=g, device=DEV) < 0.024) & valid).nonzero()[:kept, 0]
                s["idx"][f, :i.numel()], s["n_kept"][f] = i.int(), i.numel()
            s["val"] = 5 + 20 * torch.rand(s["idx"].shape, generator=g, device=DEV)
            s["noise"] = torch.randn((n, sep.npix), generator=g, device=DEV) if c["noise"] else None
    torch.cuda.synchronize()
    return s


def _mixed_counts(n):
    a, b = max(1, n // 2), max(1, n // 3)
    return a, b, max(1, n - a - b)


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "grad":
        loss, grad = s["model"].loss_grad(s["x"], s["t"])
        return {"loss": loss, "grad": grad}
    if kind == "mixed":
        o, seps = s["out"], s["seps"]
        row_off = C_ABI.sep_process_mixed(seps[0].ctx, [p.csr for p in seps], [p.calib for p in seps], s["frames"],
                                          seps[0].params, o["mean"], o["sigma"], o["count"], o["idx"], o["val"],
                                          s["kept"], o["n_kept"], o["peaks"], s["peaks"], o["n_peaks"])
        return dict(_lists(o), row_off=row_off)
    sep, frames = s["sep"], s.get("frames")
    if kind == "path":
        o = sep.process_batch(frames, s["kept"], s["peaks"], out=s["out"], stream=s["stream"])
        return _lists(o)
    if kind == "host":
        o = sep.process_host(frames, s["out"], s["kept"], s["peaks"])
        torch.cuda.current_stream().synchronize()
        # fixed-size records for the store: what lies behind a list's end is cleared
        for f, (k, p) in enumerate(zip(o["n_kept"].tolist(), o["n_peaks"].tolist())):
            o["idx"][f, k:], o["val"][f, k:], o["peaks"][f, p:] = 0, 0, 0
        return _lists(o)
    if kind == "clip":
        return sep.integrate_clip(frames)
    if kind == "correct":
        return {"frames": sep.correct(frames)}
    if kind == "compress":
        o = sep.sparsify(frames, s["mean"], s["sigma"], s["kept"])
        dense = sep.densify(s["mean"], s["sigma"], o["idx"], o["val"], o["n_kept"], out=s["dense"],
                            interpolate=c["smooth"])
        return {"n_kept": o["n_kept"], "dense": dense}
    dense = sep.densify(s["mean"], s["sigma"], s["idx"], s["val"], s["n_kept"], noise=s["noise"], out=s["dense"],
                        interpolate=c["smooth"])
    return {"dense": dense}


def _lists(o):
    """The outputs with the peak records (index, y, x, I, sigma, pixel count) split by type."""
    p = o["peaks"]
    return {k: v for k, v in o.items() if k != "peaks"} | {
        "peak_idx": p[..., 0], "peak_values": p.view(torch.float32)[..., 1:5], "peak_npix": p[..., 5]}


def work(case):
    c = case
    if c["kind"] == "grad":
        per = 20 * 64 + 64 * 64 + 64 * 2
        return {"bytes": c["rows"] * 88 + 2 * 5634 + 4 * 5635, "flops": 6 * per * c["rows"]}
    if c["kind"] == "mixed":
        total = {"bytes": 0, "flops": 0}
        for name, m in zip(MIXED, _mixed_counts(c["frames"])):
            w = work(dict(_detector("path", name), frames=m))
            total = {k: total[k] + w[k] for k in total}
        return total
    n, npix, b = c["frames"], c["rows"] * c["cols"], c["nbins"]
    word = 2 if c["raw"] else 4
    planes = npix * ((24 if c["raw"] else 0) + (4 if c["norm"] else 0))
    entries = npix * {0: 2.0, 1: 1.0, 2: 1.34}[c["split"]]
    kept = 0.024 * npix
    if c["kind"] == "correct":
        return {"bytes": n * npix * (word + 4) + planes, "flops": 2 * n * npix}
    if c["kind"] == "densify":
        return {"bytes": n * (npix * (8 if c["noise"] else 4) + 8 * kept + 8 * b) + npix * (12 if c["smooth"] else 4),
                "flops": (4 if c["noise"] else 1) * n * npix}
    if c["kind"] == "compress":
        return {"bytes": n * (npix * (word + 4) + 8 * b) + planes + npix * (12 if c["smooth"] else 4),
                "flops": 4 * n * npix}
    # a frame's words and a bin's sums once; 2 operations a pixel to correct, 5 an entry for the moments of each step
    lists = 8 * kept if c["kind"] in ("path", "host") else 0
    return {"bytes": n * (npix * word + 12 * b + lists) + planes + 4 * entries + 4 * npix,
            "flops": n * (2 * npix + 5 * (N_ITER + 1) * entries)}


# ---- the same in binary64 ---------------------------------------------------

def _weights(seed):
    """Network parameters (float32 [5634]): W1, b1, W2, b2, W3, b3."""
    r = np.random.default_rng(int(seed))
    parts = [r.normal(0, 20 ** -0.5, 1280), r.normal(0, 0.1, 64), r.normal(0, 0.125, 4096), r.normal(0, 0.1, 64),
             r.normal(0, 0.125, 128), r.normal(0, 0.1, 2)]
    return np.concatenate(parts).astype(np.float32)


def _radial(c, fy, fx):
    """q (nm^-1) at the offset (fy, fx) of every pixel."""
    cx, cy = _center(c)
    y = ((torch.arange(c["rows"], device=DEV, dtype=torch.float64) + fy) - cy) * PIXEL_M
    x = ((torch.arange(c["cols"], device=DEV, dtype=torch.float64) + fx) - cx) * PIXEL_M
    r = torch.sqrt(x[None, :] * x[None, :] + y[:, None] * y[:, None]).reshape(-1)
    return _q(r)


def _q(r):
    return 4.0 * math.pi * torch.sin(0.5 * torch.atan2(r, torch.full_like(r, DIST_M))) / (LAMBDA_M * 1e9)


def _area_entries(c, valid):
    """(pixel, bin, area fraction) of every pixel, and the range, by the closed form of a rectangle and a disc."""
    B = c["nbins"]
    cx, cy = _center(c)
    x0 = ((torch.arange(c["cols"], device=DEV, dtype=torch.float64) - cx) * PIXEL_M).repeat(c["rows"])[valid]
    y0 = ((torch.arange(c["rows"], device=DEV, dtype=torch.float64) - cy) * PIXEL_M).repeat_interleave(c["cols"])[valid]
    x1, y1, zero = x0 + PIXEL_M, y0 + PIXEL_M, torch.zeros_like(x0)
    near = torch.sqrt(torch.where(x0 > 0, x0, torch.where(x1 < 0, x1, zero)) ** 2 +
                      torch.where(y0 > 0, y0, torch.where(y1 < 0, y1, zero)) ** 2)
    far = torch.sqrt(torch.maximum(x0.abs(), x1.abs()) ** 2 + torch.maximum(y0.abs(), y1.abs()) ** 2)
    a, b = _q(near), _q(far)
    lo, hi = a.min(), b.max()
    first = ((a - lo) / (hi - lo) * B).floor().long().clamp_(0, B - 1)
    last = ((b - lo) / (hi - lo) * B).floor().long().clamp_(0, B - 1)

    def quadrant(x, y, R):   # of the disc of radius R inside [0, x] x [0, y]
        G = lambda t: 0.5 * (t * (R * R - t * t).clamp(min=0).sqrt() + R * R * torch.asin((t / R).clamp(max=1)))
        top = (R * R - y * y).clamp(min=0).sqrt()
        xc = torch.minimum(x, R)
        cut = torch.where(xc <= top, xc * y, top * y + G(xc) - G(top))
        return torch.where((R <= 0) | (x <= 0) | (y <= 0), zero, torch.where(y >= R, G(xc), cut))

    def corner(x, y, R):
        return quadrant(x.abs(), y.abs(), R) * torch.where((x < 0) != (y < 0), -1.0, 1.0)

    def inside(edge):        # area of the pixel inside the circle of radial value `edge`
        tth = 2 * torch.asin(edge * (LAMBDA_M * 1e9) / (4 * math.pi))
        R = (DIST_M * torch.tan(tth)).clamp(min=0)
        return corner(x1, y1, R) - corner(x0, y1, R) - corner(x1, y0, R) + corner(x0, y0, R)

    pix, at, out = valid.nonzero()[:, 0], [], []
    for k in range(int((last - first).max()) + 1):
        bin_ = first + k
        w = (inside(lo + (hi - lo) * (bin_ + 1).double() / B) - inside(lo + (hi - lo) * bin_.double() / B)) / PIXEL_M ** 2
        use = (bin_ <= last) & (w > 1e-12)
        at.append((pix[use], bin_[use]))
        out.append(w[use].clamp(max=1))
    return torch.cat([p for p, _ in at]), torch.cat([b for _, b in at]), torch.cat(out), lo, hi


@functools.lru_cache(maxsize=3)
def _matrix(key):
    """The rows of the integration matrix, padded: pixels, coefficients [bins][longest]; the range of q."""
    c = dict(key)
    B, s = c["nbins"], c["split"]
    valid = torch.from_numpy(_planes(*(c[k] for k in DET_KEYS))[0] == 0).to(DEV)
    if s == 0:
        pix, bins, w, lo, hi = _area_entries(c, valid)
    else:
        sub = [_radial(c, (a + 0.5) / s, (b + 0.5) / s)[valid] for a in range(s) for b in range(s)]
        lo, hi = torch.stack([x.min() for x in sub]).min(), torch.stack([x.max() for x in sub]).max()
        pix = valid.nonzero()[:, 0]
        codes = torch.cat([pix * B + ((x - lo) / (hi - lo) * B).floor().long().clamp_(0, B - 1) for x in sub])
        codes, k = torch.unique(codes, return_counts=True)
        pix, bins, w = codes // B, codes % B, k.double() / (s * s)
    order = torch.argsort(bins, stable=True)
    pix, bins, w = pix[order], bins[order], w[order]
    n = torch.bincount(bins, minlength=B)
    at = torch.arange(bins.numel(), device=DEV) - (torch.cumsum(n, 0) - n)[bins]
    P = torch.zeros((B, int(n.max())), dtype=torch.int64, device=DEV)
    C = torch.zeros(P.shape, dtype=torch.float64, device=DEV)
    P[bins, at], C[bins, at] = pix, w
    return P, C, lo, hi


def _values(c, frame):
    """Corrected pixels of one frame, divided by the norm."""
    _, ped, gain, norm = _planes(*(c[k] for k in DET_KEYS))
    v = frame.double()
    if c["raw"]:
        word = frame.int() & 0xFFFF
        level = (word >> 14).clamp(max=2).long()[None]
        v = ((word & 0x3FFF).double() - ped.gather(0, level)[0].double()) / gain.gather(0, level)[0].double()
    return v / norm.double() if c["norm"] else v


def _clip(c, frame):
    """Mean and deviation of every bin after the clip loop."""
    P, C, _, _ = _matrix(_key(c))
    v = _values(c, frame)[P]
    w = C
    if c["norm"]:
        w = C * _planes(*(c[k] for k in DET_KEYS))[3].double()[P]
    w = w.float().double() if (c["norm"] or c["split"] == 0) else w

    def moments(use):
        ww = w * use
        w2 = ww * ww
        om, oo = ww.sum(1), w2.sum(1)
        mu = torch.where(om > 0, (ww * v).sum(1) / om, 0.0)
        sd = torch.where(oo > 0, (w2 * (v - mu[:, None]) ** 2).sum(1) / oo, 0.0).sqrt()
        poisson = torch.where(oo > 0, (w2 * v).sum(1) / oo + DARK_VAR, 0.0).clamp(min=0).sqrt()
        return use.sum(1), mu, sd, poisson

    use = w > 0
    n, mu, sd, poisson = moments(use)
    going = torch.ones_like(n, dtype=torch.bool)
    for _ in range(N_ITER):
        k = torch.full_like(mu, K_CLIP)
        if c["chauvenet"]:
            going = going & (n > 2)
            k = (2 * torch.log(n.clamp(min=3).double() / math.sqrt(2 * math.pi))).sqrt()
        s = poisson if c["model"] == "poisson" else sd
        use2 = use & ((v - mu[:, None]).abs() <= (k * s)[:, None])
        going = going & (use2.sum(1) < n)
        if not bool(going.any()):
            break
        use = torch.where(going[:, None], use2, use)
        n, mu, sd, poisson = moments(use)
    return mu, sd if c["model"] == "azimuthal" else torch.where(n > 0, poisson, 0.0)


def _background(c, levels):
    """A profile at every pixel (NaN where there is none): its bin's level, or between the bin centres."""
    _, _, lo, hi = _matrix(_key(c))
    B = c["nbins"]
    valid = torch.from_numpy(_planes(*(c[k] for k in DET_KEYS))[0] == 0).to(DEV)
    u = (_radial(c, 0.5, 0.5) - lo) / (hi - lo) * B
    if c["smooth"]:
        u = (u - 0.5).clamp(0, B - 1)
        a = u.floor().long()
        t = u - a
        x = (1 - t) * levels[a] + t * levels[(a + 1).clamp(max=B - 1)]
    else:
        x = levels[u.floor().long().clamp(0, B - 1)]
    return torch.where(valid, x, math.nan)


def exact(case, seed):
    c = dict(case)
    kind = c["kind"]
    if kind == "grad":
        s = prepare(c, seed)
        p = torch.from_numpy(_weights(seed)).bfloat16().double().to(DEV).requires_grad_()
        W1, b1, W2, b2, W3, b3 = torch.split(p, [1280, 64, 4096, 64, 128, 2])
        gelu = torch.nn.functional.gelu
        h = gelu(gelu(s["x"].double() @ W1.view(64, 20).T + b1) @ W2.view(64, 64).T + b2)
        loss = ((h @ W3.view(2, 64).T + b3 - s["t"].double()) ** 2).sum(1).mean()
        return {"loss": loss.detach().reshape(1), "grad": torch.autograd.grad(loss, p)[0]}
    if kind == "mixed":
        mean, sigma = [], []
        for d, m in enumerate(_mixed_counts(c["frames"])):
            det = _detector("mixed", MIXED[d])
            for frame in _frames(det, seed, m):
                mu, sd = _clip(det, frame)
                mean.append(mu)
                sigma.append(sd)
        return {"mean": torch.cat(mean), "sigma": torch.cat(sigma)}   # counts and lists: whole numbers
    if kind in ("path", "host", "clip"):
        frames = _frames(c, seed, c["frames"])
        mean, sigma = (torch.stack(x) for x in zip(*[_clip(c, f) for f in frames]))
        return {"mean": mean, "sigma": sigma}   # counts and lists: whole numbers
    if kind == "correct":
        valid = torch.from_numpy(_planes(*(c[k] for k in DET_KEYS))[0] == 0).to(DEV)
        return {"frames": torch.stack([torch.where(valid, _values(c, f), math.nan) for f in _frames(c, seed, c["frames"])])}
    s = prepare(c, seed)
    out = []
    for f in range(c["frames"]):
        x = _background(c, s["mean"][f].double())
        if kind == "compress":
            v = _values(c, s["frames"][f])
            at = _background(dict(c, smooth=c["smooth"]), s["mean"][f].double() + K_PICK * s["sigma"][f].double())
            x = torch.where(v > at, v, x)
        else:
            if c["noise"]:
                x = x + _background(c, s["sigma"][f].double()) * s["noise"][f].double()
            k = int(s["n_kept"][f])
            x[s["idx"][f, :k].long()] = s["val"][f, :k].double()
        out.append(x)
    return {"n_kept": None, "dense": torch.stack(out)} if kind == "compress" else {"dense": torch.stack(out)}
