"""Calls that must not fall far behind their ordinary form: each times a call on
inputs that once sent it to a slow path against the same call on usual inputs,
in one process on one GPU (best of several, so that other work on the host does
not count). The limits lie between the ratio with the slow path and without."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09515_gb300 import Separator  # noqa: E402


def _best(*calls, rounds=12, repeat=10):
    """Shortest time of `repeat` runs of each call, the calls taken in turn."""
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    best = [np.inf] * len(calls)
    for r in range(rounds):
        for k, call in enumerate(calls):
            a.record()
            for _ in range(repeat):
                call()
            b.record()
            torch.cuda.synchronize()
            if r > 1:
                best[k] = min(best[k], a.elapsed_time(b))
    return best


def _detector(rows, cols, nbins=500):
    return synth.Detector("t", rows, cols, dist_m=0.1, center_px=(0.45 * cols, 0.55 * rows), nbins=nbins, split=1)


@pytest.mark.parametrize("what,limit", [("gain levels", 1.25), ("mask", 1.15)])
def test_staging(what, limit):
    """A pixel in a thousand at another gain level; gain 0 under a mask of two pixels in a hundred."""
    det, F = _detector(1500, 1500), 64
    n = det.npix
    rng = np.random.default_rng(1)
    mask = (rng.random(n) < 0.02).astype(np.uint8)
    ped, gain = synth.jf_calib(n, seed=1)
    bad_ped, bad_gain = ped.copy(), gain.copy()
    bad_ped[:, mask != 0], bad_gain[:, mask != 0] = 0, 0
    g = torch.Generator(device="cuda")
    g.manual_seed(2)
    word = torch.from_numpy(ped[0]).cuda() + torch.from_numpy(gain[0]).cuda() * torch.poisson(
        torch.full((F, n), 2.0, device="cuda"), generator=g)
    word = word.clamp(0, 16383).to(torch.int16)
    other = word.clone()
    other[torch.rand((F, n), generator=g, device="cuda") < 1e-3] |= 1 << 14
    kw = {"mask": mask, "n_iter": 0}
    usual = Separator.from_detector(det, calib=(ped, gain), **kw)
    odd = Separator.from_detector(det, calib=(bad_ped, bad_gain), **kw)
    if what == "mask":
        t, t0 = _best(lambda: odd.integrate_clip(word), lambda: usual.integrate_clip(word))
    else:
        t, t0 = _best(lambda: usual.integrate_clip(other), lambda: usual.integrate_clip(word))
    assert t < limit * t0, t / t0
    usual.close()
    odd.close()


def test_peaks_of_many_candidates():
    """Five by five patches around one pixel in six, against three by three."""
    det, F = _detector(1500, 1500), 16
    sep = Separator.from_detector(det, k_pick=1.0)
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    frames = torch.randn((F, det.npix), generator=g, device="cuda")
    m = torch.zeros((F, sep.nbins), dtype=torch.float32, device="cuda")
    s = torch.ones_like(m)
    k = sep.sparsify(frames, m, s, det.npix // 4)

    def peaks(patch):
        sep.set_params(patch=patch, min_count=3)
        sep.peakfind(frames, m, s, k["idx"], k["n_kept"], det.npix // 16)

    t, t0 = _best(lambda: peaks(5), lambda: peaks(3), rounds=8, repeat=4)
    assert t < 2.8 * t0, t / t0
    sep.close()


def test_compaction_of_a_full_small_frame():
    """Every pixel of a few small frames kept, against one in a hundred."""
    det, F = _detector(300, 301, 60), 7
    sep = Separator.from_detector(det, k_pick=1.0)
    full = torch.full((F, det.npix), 2.0, device="cuda")
    few = full * (torch.arange(det.npix, device="cuda") % 100 == 0)
    m = torch.zeros((F, sep.nbins), dtype=torch.float32, device="cuda")
    s = torch.ones_like(m)
    t, t0 = _best(lambda: sep.sparsify(full, m, s, det.npix), lambda: sep.sparsify(few, m, s, det.npix), repeat=30)
    assert t < 3 * t0, t / t0
    sep.close()


def test_one_smooth_dense_frame():
    """A frame of a 16M detector from its smooth profile, against its profile by bin."""
    det = _detector(4362, 4148, 2000)
    sep = Separator.from_detector(det)
    m = torch.rand((1, sep.nbins), device="cuda") + 1
    out = torch.empty((1, det.npix), dtype=torch.float32, device="cuda")

    def dense(smooth):
        sep.densify(m, m, None, None, None, out=out, interpolate=smooth)

    t, t0 = _best(lambda: dense(True), lambda: dense(False), repeat=20)
    assert t < 1.8 * t0, t / t0
    sep.close()
