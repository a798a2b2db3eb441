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
