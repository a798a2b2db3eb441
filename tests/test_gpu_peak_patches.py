"""Peak tests and records against the oracle over the patch sizes the library
takes: 1 to 15 pixels a side (several candidates of a warp side by side, one at
a time, one a lane), few and many kept pixels, borders, ties and masked
neighbours; records over the lists and slices they are written through; a
capacity that ends inside one; and a caller's list that names masked pixels."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09515_gb300 import Separator, peaks_to_numpy  # noqa: E402

# Records: binary32 sums of at most 225 positive terms (values above a zero
# mean), each sum within 225 2^-24 of itself, a quotient of two of them within
# twice that and one rounding.
RTOL = 2 * 225 * 2.0 ** -24 + 2.0 ** -23


def _detector(rows, cols, nbins=12):
    return synth.Detector("p", rows, cols, dist_m=0.05, center_px=(0.4 * cols, 0.6 * rows), nbins=nbins, split=1)


def _flat(sep, F):
    """Profiles of mean 0 and deviation 1: kept pixels are those above k_pick."""
    return (torch.zeros((F, sep.nbins), dtype=torch.float32, device="cuda"),
            torch.ones((F, sep.nbins), dtype=torch.float32, device="cuda"))


@pytest.mark.parametrize("patch,min_count", [(1, 1), (3, 1), (3, 3), (5, 2), (7, 3), (9, 4), (11, 1), (15, 1), (15, 30)])
@pytest.mark.parametrize("share", [0.02, 0.3, 1.0])
@pytest.mark.parametrize("rows,cols,F", [(9, 7, 2), (37, 61, 3), (128, 130, 2)])
def test_peaks_match_oracle(rows, cols, F, share, patch, min_count):
    det = _detector(rows, cols)
    rng = np.random.default_rng(rows + patch + int(10 * share))
    mask = (rng.random(det.npix) < 0.03).astype(np.uint8)
    sep = Separator.from_detector(det, mask=mask, k_pick=4.0, patch=patch, min_count=min_count)
    # whole numbers: many ties; some frames' pixels above the threshold in clumps
    fr = rng.integers(0, 4, (F, det.npix)).astype(np.float32)
    for f in range(F):
        up = rng.random((rows, cols)) < share
        if share < 0.1:
            up |= np.roll(up, 1, 0) | np.roll(up, 1, 1) | np.roll(up, (1, 1), (0, 1))
        fr[f] += np.where(up.reshape(-1), rng.integers(5, 30, det.npix), 0)
    frames = torch.from_numpy(fr).cuda()
    m, s = _flat(sep, F)
    k = sep.sparsify(frames, m, s, det.npix)
    o = sep.peakfind(frames, m, s, k["idx"], k["n_kept"], det.npix)
    torch.cuda.synchronize()
    W = oracle.weights(det, mask)
    for f in range(F):
        want = oracle.peaks(det, W, fr[f], np.zeros(det.nbins), np.ones(det.nbins), k_pick=4.0, patch=patch,
                            min_count=min_count)
        got = peaks_to_numpy(o["peaks"][f], o["n_peaks"][f])
        assert np.array_equal(got["idx"], want["idx"])
        assert np.array_equal(got["npix"], want["npix"])
        for q in ("I", "y", "x", "sigma"):
            assert np.allclose(got[q], want[q], rtol=RTOL, atol=0), q
    assert sep.device_status() == 0
    sep.close()


@pytest.mark.parametrize("raw", [False, True])
@pytest.mark.parametrize("patch,min_count", [(1, 1), (3, 3), (5, 1), (9, 6), (15, 2)])
def test_batch_gives_the_standalone_peaks(patch, min_count, raw):
    """Staged values and the clip kernel's marks in the place of frames and a list."""
    det = _detector(140, 133)
    rng = np.random.default_rng(patch)
    cal = synth.jf_calib(det.npix, seed=3) if raw else None
    sep = Separator.from_detector(det, calib=cal, k_pick=1.0, patch=patch, min_count=min_count)
    q = rng.poisson(7, (4, det.npix))
    fr = (cal[0][0] + cal[1][0] * q).clip(0, 16383).astype(np.uint16).view(np.int16) if raw else q.astype(np.float32)
    frames = torch.from_numpy(fr).cuda()
    o = sep.process_batch(frames, det.npix, det.npix)
    p = sep.peakfind(frames, o["mean"], o["sigma"], o["idx"], o["n_kept"], det.npix)
    torch.cuda.synchronize()
    for f in range(4):
        n = int(o["n_peaks"][f])
        assert n == int(p["n_peaks"][f]) and n > 0
        assert torch.equal(o["peaks"][f, :n], p["peaks"][f, :n])
    sep.close()


@pytest.mark.parametrize("rows,cols,F", [(600, 600, 64), (300, 331, 3), (41, 37, 400)])
def test_every_kept_pixel_a_peak(rows, cols, F):
    """Slices of more chunks than a pass and more peaks than a list hold, and capacities that end inside them."""
    det = _detector(rows, cols)
    sep = Separator.from_detector(det, k_pick=0.5, patch=1, min_count=1)
    g = torch.Generator(device="cuda")
    g.manual_seed(rows)
    frames = 1.0 + torch.randint(0, 9, (F, det.npix), generator=g, device="cuda").float()
    frames[0, ::3] = 0
    m, s = _flat(sep, F)
    k = sep.sparsify(frames, m, s, det.npix)
    n_kept = k["n_kept"].cpu().numpy()
    for pcap in (1, 255, 2049, int(n_kept[-1]) - 1, det.npix):
        if pcap > det.npix:
            continue
        o = sep.peakfind(frames, m, s, k["idx"], k["n_kept"], pcap)
        assert np.array_equal(o["n_peaks"].cpu().numpy(), n_kept)
        for f in {0, 1, F - 1}:
            n = min(pcap, int(n_kept[f]))
            i = k["idx"][f, :n].long()
            rec = o["peaks"][f, :n]
            v = rec.view(torch.float32)
            assert torch.equal(rec[:, 0].long(), i) and bool((rec[:, 5] == 1).all())
            # one pixel: I is its value, the centroid its centre (a product and a quotient: two roundings)
            assert torch.equal(v[:, 3], frames[f, i])
            assert torch.allclose(v[:, 1].double(), (i // cols).double() + 0.5, rtol=2.0 ** -22, atol=0)
            assert torch.allclose(v[:, 2].double(), (i % cols).double() + 0.5, rtol=2.0 ** -22, atol=0)
        assert (sep.device_status() != 0) == (n_kept.max() > pcap)
    sep.close()


@pytest.mark.parametrize("patch", [3, 7])
def test_a_list_that_names_masked_pixels(patch):
    """They count as listed neighbours, but are no peaks and give nothing to a record."""
    det = _detector(40, 45)
    rng = np.random.default_rng(patch)
    mask = (rng.random(det.npix) < 0.2).astype(np.uint8)
    sep = Separator.from_detector(det, mask=mask, patch=patch, min_count=4)
    fr = rng.permutation(det.npix).astype(np.float32)[None] + 1
    lst = np.flatnonzero(rng.random(det.npix) < 0.4).astype(np.int32)
    assert mask[lst].any()
    m, s = _flat(sep, 1)
    o = sep.peakfind(torch.from_numpy(fr).cuda(), m, s, torch.from_numpy(lst[None]).cuda(),
                     torch.tensor([lst.size], dtype=torch.int32, device="cuda"), det.npix)
    torch.cuda.synchronize()
    got = peaks_to_numpy(o["peaks"][0], o["n_peaks"][0])
    v, used = fr[0].reshape(det.rows, det.cols), (mask == 0).reshape(det.rows, det.cols)
    on = np.zeros(det.npix, bool)
    on[lst] = True
    on = on.reshape(det.rows, det.cols)
    h, want = patch // 2, []
    for i in lst:
        r, c = divmod(int(i), det.cols)
        w = np.s_[max(r - h, 0):r + h + 1, max(c - h, 0):c + h + 1]
        if used[r, c] and on[w].sum() >= 4 and v[r, c] == v[w][used[w]].max():
            both = on[w] & used[w]
            want.append((i, both.sum(), v[w][both].astype(np.float64).sum()))
    assert len(want) > 5
    assert np.array_equal(got["idx"], [x[0] for x in want])
    assert np.array_equal(got["npix"], [x[1] for x in want])
    assert np.allclose(got["I"], [x[2] for x in want], rtol=RTOL, atol=0)
    sep.close()
