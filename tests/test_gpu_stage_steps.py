"""The staging kernel over several steps a group of frames (ring slots that are
refilled, both tile buffers, a last step of one to three frames), for every way
a thread's words reach it, gain level and calibration: each frame's staged
values in image order (a corrected batch whose output lies over its frames is
written from the staged copy) and the kept values of a frame list, bit for bit."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09515_gb300 import (SEP_DTYPE_F32, SEP_DTYPE_U16_JF, Context, Separator,  # noqa: E402
                                    _binding as B, process_mixed)


def _calib(n, mask, rng):
    """Masked pixels without a usable calibration (gain 0, NaN), and a few used ones outside the usual range."""
    ped, gain = synth.jf_calib(n, seed=3)
    off = np.flatnonzero(mask)
    ped[:, off[::2]], gain[:, off[::2]] = 0, 0
    gain[0, off[1::4]], ped[1, off[1::4]] = np.nan, np.nan
    used = np.flatnonzero(mask == 0)
    at = rng.permutation(used)
    gain[0, at[:n // 50]] = np.float32(2.0 ** -41)
    ped[0, at[n // 50:n // 25]] = 1e-30
    return ped, gain


def _words(F, n, mask, rng):
    """Frames with a few, some, and only words of other gain levels; level 3 under the mask."""
    share = np.array([0.0, 0.001, 0.05, 0.5, 1.0])[np.arange(F) % 5]
    level = np.where(rng.random((F, n)) < share[:, None], rng.integers(1, 4, (F, n)), 0)
    w = (rng.integers(1000, 1 << 14, (F, n)) | level << 14).astype(np.uint16)
    w[:, mask != 0] |= 3 << 14
    return w


# (81 tiles x 67 frames: eight frames a group and a remainder of three; 9 x 1102: sixteen and fourteen; up to eight
# frames: pairs of them a CTA; 169 tiles x 11: one group)
@pytest.mark.parametrize("with_norm", [False, True])
@pytest.mark.parametrize("raw", [False, True])
@pytest.mark.parametrize("rows,cols,F", [(520, 520, 67), (520, 518, 67), (521, 519, 66), (130, 131, 1102), (129, 132, 1),
                                         (129, 131, 2), (65, 126, 3), (521, 516, 65), (521, 518, 8), (520, 519, 5),
                                         (129, 130, 9), (830, 831, 11)])
def test_staged_values_over_steps(rows, cols, F, raw, with_norm):
    rng = np.random.default_rng(rows + cols + F)
    det = synth.Detector("s", rows, cols, dist_m=0.05, center_px=(0.4 * cols, 0.6 * rows), nbins=60, split=2)
    n = det.npix
    mask = (rng.random(n) < 0.05).astype(np.uint8)
    mask.reshape(rows, cols)[:, 60:70] = 1   # (a module gap)
    cal = _calib(n, mask, rng) if raw else None
    norm = rng.uniform(0.5, 2.0, n).astype(np.float32) if with_norm else None
    ctx = Context(0)
    sep = Separator.from_detector(det, mask=mask, calib=cal, norm=norm, k_pick=0.0, context=ctx)
    if raw:
        words = _words(F, n, mask, rng)
        with np.errstate(all="ignore"):
            v = np.stack([oracle.jf_photons(w, cal[0], cal[1]) for w in words])
    else:
        words = rng.normal(10, 3, (F, n)).astype(np.float32)
        v = words
    with np.errstate(all="ignore"):
        v = v if norm is None else (v / norm).astype(np.float32)
    used = mask == 0
    want = v[:, used].view(np.uint32)
    t = torch.from_numpy(words.view(np.int16) if raw else words)
    size, dtype = (2, SEP_DTYPE_U16_JF) if raw else (4, SEP_DTYPE_F32)
    for shift in (0, 1, 2):   # words past an aligned address
        buf = torch.zeros(F * n * 4 + 64, dtype=torch.uint8, device="cuda")
        frames = buf[shift * size:shift * size + F * n * size].view(t.dtype).view(F, n)
        frames.copy_(t)
        out = buf[:F * n * 4].view(torch.float32).view(F, n)
        B.sep_correct(sep.ctx, sep.csr, sep.calib, frames, dtype, F, out)
        got = out.cpu().numpy()
        assert np.array_equal(got[:, used].view(np.uint32), want)
        assert np.isnan(got[:, ~used]).all()
    # a list of frames, aligned or every other one at an odd address
    m = min(F, 70)
    for odd in (False, True):
        lst = [t[f].cuda() for f in range(m)]
        for f in range(0, m, 2) if odd else ():
            x = torch.empty(n + 1, dtype=t.dtype, device="cuda")
            x[1:] = lst[f]
            lst[f] = x[1:]
        q = process_mixed([sep], [(0, x) for x in lst], n, 64)
        torch.cuda.synchronize()
        nk = q["n_kept"].cpu().numpy()
        for f in range(m):
            i = q["idx"][f, :nk[f]].cpu().numpy()
            assert nk[f] > 0 and np.array_equal(q["val"][f, :nk[f]].cpu().numpy().view(np.uint32), v[f, i].view(np.uint32))
    sep.close()
    ctx.close()
