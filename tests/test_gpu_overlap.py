"""Outputs that lie over the frames they are computed from: the frames are read
whole before the first output byte is written, so the results are those of a
call with buffers of its own, bit for bit."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09515_gb300 import SEP_DTYPE_F32, SEP_DTYPE_U16_JF, Separator, _binding as B  # noqa: E402


def _detector(rows, cols):
    return synth.Detector("o", rows, cols, dist_m=0.05, center_px=(0.4 * cols, 0.6 * rows), nbins=40, split=2)


def _separator(det, raw, with_norm):
    rng = np.random.default_rng(det.npix)
    mask = (rng.random(det.npix) < 0.05).astype(np.uint8)
    norm = rng.uniform(0.5, 2.0, det.npix).astype(np.float32) if with_norm else None
    cal = synth.jf_calib(det.npix, seed=2) if raw else None
    return Separator.from_detector(det, mask=mask, calib=cal, norm=norm, patch=3, min_count=1), mask, norm, cal


@pytest.mark.parametrize("with_norm", [False, True])
@pytest.mark.parametrize("raw,shift", [(True, 0), (True, 4), (True, -1), (False, 0), (False, 3), (False, -5)])
@pytest.mark.parametrize("rows,cols,F", [(64, 64, 3), (61, 67, 17), (256, 256, 80)])
def test_correct(rows, cols, F, raw, shift, with_norm):
    """Frames that start at, `shift` words into, or (-1) in the last words of the output buffer."""
    det = _detector(rows, cols)
    n = det.npix
    sep, mask, norm, cal = _separator(det, raw, with_norm)
    rng = np.random.default_rng(F)
    if raw:
        words = rng.integers(0, 1 << 16, (F, n), dtype=np.uint16)
        want = np.stack([oracle.jf_photons(w, cal[0], cal[1]) for w in words])
    else:
        words = rng.normal(10, 3, (F, n)).astype(np.float32)
        want = words.copy()
    if with_norm:
        want = (want / norm).astype(np.float32)
    want[:, mask != 0] = np.nan
    size = 2 if raw else 4
    buf = torch.zeros(F * n * 4 + 128, dtype=torch.uint8, device="cuda")
    out = buf[64:64 + F * n * 4].view(torch.float32).view(F, n)
    at = 64 + shift * size if not raw or shift >= 0 else 64 + F * n * (4 - size)
    t = torch.from_numpy(words.view(np.int16) if raw else words)
    frames = buf[at:at + F * n * size].view(t.dtype).view(F, n)
    assert at + F * n * size <= buf.numel() and at >= 0
    frames.copy_(t)
    B.sep_correct(sep.ctx, sep.csr, sep.calib, frames, SEP_DTYPE_U16_JF if raw else SEP_DTYPE_F32, F, out)
    torch.cuda.synchronize()
    got = out.cpu().numpy()
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan].view(np.uint32), want[~nan].view(np.uint32))
    sep.close()


KEYS = ("mean", "sigma", "count", "idx", "val", "n_kept", "peaks", "n_peaks")


def _equal(got, want):
    for k in KEYS:
        assert np.array_equal(got[k].view(np.uint32), want[k].view(np.uint32)), k


def _zero_tails(o):
    o = {k: v.cpu().numpy().copy() for k, v in o.items() if k in KEYS}
    for f, (k, p) in enumerate(zip(o["n_kept"], o["n_peaks"])):
        o["idx"][f, k:], o["val"][f, k:], o["peaks"][f, p:] = 0, 0, 0
    return o


@pytest.mark.parametrize("smooth", [0, 1])
@pytest.mark.parametrize("raw,with_norm", [(False, False), (False, True), (True, False)])
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("over", ["mean", "sigma", "val", "idx", "peaks"])
def test_batch(over, mixed, graph, raw, with_norm, smooth):
    """One output of the whole path in the frames' own memory (in place: the frames' results over the frames)."""
    F, det = 9, _detector(131, 126)
    n, kcap, pcap = det.npix, 3000, 600
    sep, _, norm, cal = _separator(det, raw, with_norm)
    sep.set_params(interpolate=smooth, k_pick=2.0)
    rng = np.random.default_rng(5)
    if raw:
        words = (cal[0][0] + cal[1][0] * rng.poisson(6, (F, n))).clip(0, 16383).astype(np.uint16).view(np.int16)
    else:
        words = (rng.poisson(6, (F, n)) * (norm if with_norm else 1)).astype(np.float32)
    t = torch.from_numpy(words).cuda()
    dtype = SEP_DTYPE_U16_JF if raw else SEP_DTYPE_F32
    stream = torch.cuda.Stream() if graph else None

    def call(frames, o):
        if mixed:
            B.sep_process_mixed(sep.ctx, [sep.csr], [sep.calib], [(0, dtype, frames[f]) for f in range(F)], sep.params,
                                o["mean"], o["sigma"], o["count"], o["idx"], o["val"], kcap, o["n_kept"], o["peaks"],
                                pcap, o["n_peaks"], int(graph), stream)
        else:
            B.sep_process_batch(sep.ctx, sep.csr, sep.calib, frames, dtype, F, sep.params, o["mean"], o["sigma"],
                                o["count"], o["idx"], o["val"], kcap, o["n_kept"], o["peaks"], pcap, o["n_peaks"],
                                int(graph), stream)
        torch.cuda.synchronize()
        assert sep.device_status() == 0
        return _zero_tails(o)

    want = call(t, sep.alloc_outputs(F, kcap, pcap))
    assert want["n_kept"].min() > 0 and want["n_peaks"].min() > 0
    for _ in range(2):   # (the second call replays the graph)
        frames = t.clone()
        o = sep.alloc_outputs(F, kcap, pcap)
        size = o[over].numel() * 4
        assert size <= frames.numel() * frames.element_size()
        o[over] = frames.view(-1).view(torch.uint8)[:size].view(o[over].dtype).view(o[over].shape)
        torch.cuda.synchronize()
        _equal(call(frames, o), want)
    sep.close()


@pytest.mark.parametrize("F", [16, 64])
@pytest.mark.parametrize("over", ["idx", "val", "peaks"])
def test_host_batch(over, F):
    """Results of a batch of one chunk over its own host frames."""
    det = _detector(800, 811)   # (2.6 MB a frame: default chunks of less than 16 frames)
    n, kcap, pcap = det.npix, 40000, 4000
    sep, _, _, _ = _separator(det, False, False)
    words = torch.from_numpy(np.random.default_rng(6).poisson(6, (F, n)).astype(np.float32)).pin_memory()
    ref = sep.process_host(words, sep.alloc_host_outputs(F, kcap, pcap), kcap, pcap)
    torch.cuda.synchronize()
    want = _zero_tails(ref)
    frames = words.clone().pin_memory()
    o = sep.alloc_host_outputs(F, kcap, pcap)
    flat = frames.view(-1).view(torch.uint8)
    size = o[over].numel() * 4
    # the last words: the frames that are copied in last
    o[over] = flat[flat.numel() - size:].view(o[over].dtype).view(o[over].shape)
    sep.process_host(frames, o, kcap, pcap)
    torch.cuda.synchronize()
    _equal(_zero_tails(o), want)
    sep.close()
