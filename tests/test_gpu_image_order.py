"""The image-order kernels (kept-pixel marks, corrected and dense frames) against NumPy at the sizes where
they can go wrong: fewer pixels than a warp's 128, one more, bitmap words that
end inside a warp, frame counts that leave a remainder behind a thread's group
of frames, frames at addresses aligned to one word only, and values on,
directly above and directly below their thresholds."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09515_gb300 import Separator, _binding as B  # noqa: E402

# rows, columns, frames (the last: several frames a thread, and a remainder)
SIZES = [(5, 7, 3), (16, 8, 2), (3, 43, 2), (31, 33, 5), (61, 67, 17), (256, 256, 403)]


def _det(rows, cols, nbins):
    return synth.Detector("i", rows, cols, dist_m=0.05, center_px=(0.4 * cols + 0.3, 0.6 * rows + 0.2), nbins=nbins,
                          split=1, unit=synth.UNIT_R_MM)


def _values(words, cal, norm):
    v = words if cal is None else np.stack([oracle.jf_photons(w, cal[0], cal[1]) for w in words])
    return v.astype(np.float32) if norm is None else (v.astype(np.float32) / norm).astype(np.float32)


def _calib(n, rng):
    """A Jungfrau calibration with pixels outside the usual range: gains near powers of two and near all-ones
    significands, zero, tiny and huge pedestals and gains (the division-free path's limits and beyond them)."""
    ped, gain = synth.jf_calib(n, seed=4)
    at = rng.permutation(n)
    for k, g in enumerate([1.0, np.nextafter(np.float32(2), np.float32(0)), 3.0, 2.0 ** -40, 2.0 ** 40, 2.0 ** -41,
                           2.0 ** 41, 1e-38, 1e38, -7.0]):
        gain[0, at[k::31]] = g
    for k, p in enumerate([0.0, 2.0 ** -60, 2.0 ** 60, 1e-30, 1e30, 16383.0, 0.5]):
        ped[0, at[k + 11::37]] = p
    return ped, gain


def _unaligned(a):
    """The array on the GPU one element past an aligned address."""
    t = torch.from_numpy(a.view(np.int16) if a.dtype == np.uint16 else a)
    buf = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")
    buf[1:] = t.reshape(-1).cuda()
    return buf[1:].view(t.shape)


def _threshold(sep, mean, sigma, k, smooth, bop):
    """Per pixel, binary64 (the library compares with this sum exactly)."""
    if not smooth:
        b = np.maximum(bop, 0)
        return mean[:, b].astype(np.float64) + np.float64(np.float32(k)) * sigma[:, b].astype(np.float64)
    a, t = B.sep_csr_interp(sep.csr)
    up = np.minimum(a + 1, mean.shape[1] - 1)

    def at(p):
        hi = np.where(a + 1 < p.shape[1], p[:, up], np.float32(0))
        return ((np.float32(1) - t) * p[:, a]).astype(np.float32) + (t * hi).astype(np.float32)

    return at(mean).astype(np.float64) + np.float64(np.float32(k)) * at(sigma).astype(np.float64)


@pytest.mark.parametrize("smooth", [0, 1])
@pytest.mark.parametrize("raw,with_norm", [(False, False), (False, True), (True, False), (True, True)])
@pytest.mark.parametrize("rows,cols,F", SIZES)
def test_sparsify_marks(rows, cols, F, raw, with_norm, smooth):
    rng = np.random.default_rng(rows * cols + F + 2 * raw + with_norm)
    det = _det(rows, cols, nbins=min(40, max(2, rows * cols // 20)))
    n = det.npix
    norm = rng.uniform(0.5, 2.0, n).astype(np.float32) if with_norm else None
    cal = _calib(n, rng) if raw else None
    mask = (rng.random(n) < 0.1).astype(np.uint8)
    sep = Separator.from_detector(det, mask=mask, norm=norm, calib=cal)
    sep.set_params(interpolate=smooth, k_pick=2.7)
    bop = B.sep_csr_export(sep.csr)["bin_of_pixel"]
    mean = rng.uniform(0.2, 30, (F, det.nbins)).astype(np.float32)
    sigma = rng.uniform(0.1, 3, (F, det.nbins)).astype(np.float32)
    thr = _threshold(sep, mean, sigma, 2.7, smooth, bop)
    if raw:
        words = rng.integers(0, 1 << 16, (F, n), dtype=np.uint16)   # all three gain levels
    else:
        # around the threshold: on its binary32 neighbours, and further off
        near = thr.astype(np.float32)
        step = rng.integers(-2, 3, (F, n))
        words = near.copy()
        for d in (-2, -1, 1, 2):
            x = near
            for _ in range(abs(d)):
                x = np.nextafter(x, np.float32(np.sign(d) * np.inf))
            words = np.where(step == d, x, words)
        far = rng.random((F, n)) < 0.5
        words = np.where(far, rng.uniform(0, 40, (F, n)), words).astype(np.float32)
        words[:, ::17] = np.nan
        words[:, 5::29] = np.inf
        if with_norm:
            words = (words * norm).astype(np.float32)
    v = _values(words, cal, norm)
    frames = _unaligned(words)
    cap = n
    m, s = torch.from_numpy(mean).cuda(), torch.from_numpy(sigma).cuda()
    o = sep.sparsify(frames, m, s, cap)
    torch.cuda.synchronize()
    keep = (bop >= 0) & (v.astype(np.float64) > thr)
    n_kept, idx, val = (o[k].cpu().numpy() for k in ("n_kept", "idx", "val"))
    assert np.array_equal(n_kept, keep.sum(1))
    for f in range(F):
        want = np.flatnonzero(keep[f])
        assert np.array_equal(idx[f, :want.size], want), f
        assert np.array_equal(val[f, :want.size].view(np.uint32), v[f, want].view(np.uint32)), f
    assert sep.device_status() == 0
    sep.close()


@pytest.mark.parametrize("raw,with_norm", [(False, False), (False, True), (True, False), (True, True)])
@pytest.mark.parametrize("rows,cols,F", SIZES)
def test_corrected_frames(rows, cols, F, raw, with_norm):
    rng = np.random.default_rng(7 * rows * cols + F)
    det = _det(rows, cols, nbins=min(40, max(2, rows * cols // 20)))
    n = det.npix
    norm = rng.uniform(0.5, 2.0, n).astype(np.float32) if with_norm else None
    cal = _calib(n, rng) if raw else None
    mask = (rng.random(n) < 0.1).astype(np.uint8)
    sep = Separator.from_detector(det, mask=mask, norm=norm, calib=cal)
    if raw:
        words = rng.integers(0, 1 << 16, (F, n), dtype=np.uint16)
    else:
        words = rng.normal(3, 10, (F, n)).astype(np.float32)
        words[:, ::17], words[:, 5::29] = np.nan, np.inf
    with np.errstate(over="ignore", under="ignore"):
        v = _values(words, cal, norm)
    used = mask == 0
    aligned = torch.from_numpy(words.view(np.int16) if raw else words).cuda()   # (vector accesses where they fit)
    for frames in (_unaligned(words), aligned):
        got = sep.correct(frames).cpu().numpy()
        assert np.isnan(got[:, ~used]).all()
        a, b = got[:, used], v[:, used]
        assert np.array_equal(np.isnan(a), np.isnan(b))
        assert np.array_equal(a[~np.isnan(a)].view(np.uint32), b[~np.isnan(b)].view(np.uint32))
    sep.close()


@pytest.mark.parametrize("smooth", [False, True])
@pytest.mark.parametrize("noisy", [False, True])
@pytest.mark.parametrize("rows,cols,F", SIZES)
def test_dense_background(rows, cols, F, noisy, smooth):
    rng = np.random.default_rng(3 * rows * cols + F)
    det = _det(rows, cols, nbins=min(40, max(2, rows * cols // 20)))
    n = det.npix
    mask = (rng.random(n) < 0.1).astype(np.uint8)
    sep = Separator.from_detector(det, mask=mask)
    bop = B.sep_csr_export(sep.csr)["bin_of_pixel"]
    mean = rng.uniform(0.2, 30, (F, det.nbins)).astype(np.float32)
    sigma = rng.uniform(0.1, 3, (F, det.nbins)).astype(np.float32)
    z = rng.standard_normal((F, n)).astype(np.float32) if noisy else None

    def at(p):
        if not smooth:
            return p[:, np.maximum(bop, 0)]
        a, t = B.sep_csr_interp(sep.csr)
        hi = np.where(a + 1 < p.shape[1], p[:, np.minimum(a + 1, p.shape[1] - 1)], np.float32(0))
        return ((np.float32(1) - t) * p[:, a]).astype(np.float32) + (t * hi).astype(np.float32)

    want = at(mean)
    if noisy:
        want = (want + (at(sigma) * z).astype(np.float32)).astype(np.float32)
    want = np.where(bop >= 0, want, np.float32(-2.5)).astype(np.float32)
    got = sep.densify(torch.from_numpy(mean).cuda(), torch.from_numpy(sigma).cuda(), None, None, None,
                      noise=None if z is None else _unaligned(z), fill=-2.5, interpolate=smooth)
    torch.cuda.synchronize()
    assert np.array_equal(got.cpu().numpy().view(np.uint32), want.view(np.uint32))
    sep.close()
