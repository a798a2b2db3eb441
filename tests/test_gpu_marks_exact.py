"""Kept-pixel marks of the clip kernel, pixel by pixel: a batch keeps exactly the
pixels above its thresholds, where the row is scanned, where the tail alone is,
and where a warp's list fills several times; the counters show that a case
took the path it names."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09515_gb300 import SEP_PREC_KAHAN, Separator, _binding as B  # noqa: E402


@pytest.mark.parametrize("precision", [None, SEP_PREC_KAHAN])
@pytest.mark.parametrize("split,with_norm", [(1, False), (2, False), (2, True)])
@pytest.mark.parametrize("rows,cols,nbins,k_pick", [(256, 256, 64, 0.0), (300, 331, 9, 0.0), (300, 331, 9, 3.5),
                                                    (256, 256, 64, 3.5), (41, 37, 30, 1.0)])
def test_marks(rows, cols, nbins, k_pick, split, with_norm, precision):
    rng = np.random.default_rng(rows + nbins)
    det = synth.Detector("m", rows, cols, dist_m=0.1, center_px=(0.45 * cols, 0.55 * rows), nbins=nbins, split=split)
    norm = rng.uniform(0.5, 2.0, det.npix).astype(np.float32) if with_norm else None
    kw = {} if precision is None else {"precision": precision}
    sep = Separator.from_detector(det, norm=norm, k_pick=k_pick, **kw)
    bop = B.sep_csr_export(sep.csr)["bin_of_pixel"]
    v = rng.poisson(20, (2, det.npix)).astype(np.float32)
    v[1] += np.where(rng.random(det.npix) < 0.3, rng.exponential(60, det.npix), 0).astype(np.float32)
    fr = (v * norm).astype(np.float32) if with_norm else v
    if with_norm:
        v = (fr / norm).astype(np.float32)
    sep.clip_stats(1, read=False, reset=True)
    o = sep.process_batch(torch.from_numpy(fr).cuda(), det.npix, 4096)
    torch.cuda.synchronize()
    stats = sep.clip_stats(0)
    assert stats["items"] == 2 * nbins
    if rows == 300:
        assert stats["overflows"] > 0   # (a heavy upper side on long rows)
        assert np.bincount(bop, minlength=nbins).max() > 4096   # (at k_pick 0 more than a list's 1024 are kept)
    if k_pick > 3 and not with_norm:
        assert stats["tail_marked"] > 0
    mean, sigma = (o[q].cpu().numpy().astype(np.float64) for q in ("mean", "sigma"))
    for f in range(2):
        thr = (mean[f] + np.float64(np.float32(k_pick)) * sigma[f])[bop]
        # the batch's threshold is the unrounded mean's: within a unit in the last place of the
        # reported mean, k of the deviation's, and its own rounding
        slack = 2.0 ** -23 * (np.abs(mean[f]) + k_pick * sigma[f])[bop] + np.spacing(np.abs(thr).astype(np.float32))
        kept = np.zeros(det.npix, bool)
        n = int(o["n_kept"][f])
        idx = o["idx"][f, :n].cpu().numpy()
        assert np.all(np.diff(idx) > 0) and n > 0
        kept[idx] = True
        differ = kept != (v[f].astype(np.float64) > thr)
        assert np.all(np.abs(v[f][differ] - thr[differ]) <= slack[differ])
        assert np.array_equal(o["val"][f, :n].cpu().numpy().view(np.uint32), v[f, idx].view(np.uint32))
    assert sep.device_status() & 2 == 0
    sep.close()
