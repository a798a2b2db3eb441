"""The clip kernel's kept-pixel marks where a bin keeps many pixels: thresholds
at and below the core (the whole row is scanned), bins with more kept entries
than a warp lists at once, and tails that overflow. The batch's lists equal
those of the standalone call on the same profiles, bit for bit."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09515_gb300 import SEP_PREC_KAHAN, Separator  # noqa: E402


@pytest.mark.parametrize("precision", [None, SEP_PREC_KAHAN])
@pytest.mark.parametrize("split,with_norm", [(1, False), (2, False), (2, True)])
@pytest.mark.parametrize("rows,cols,nbins,k_pick", [(256, 256, 64, 0.0), (256, 256, 64, 1.0), (300, 331, 9, 0.0),
                                                    (300, 331, 9, 2.5), (41, 37, 30, 0.0)])
def test_marks_equal_sparsify(rows, cols, nbins, k_pick, split, with_norm, precision):
    rng = np.random.default_rng(rows + nbins)
    det = synth.Detector("m", rows, cols, dist_m=0.1, center_px=(0.45 * cols, 0.55 * rows), nbins=nbins, split=split)
    norm = rng.uniform(0.5, 2.0, det.npix).astype(np.float32) if with_norm else None
    kw = {} if precision is None else {"precision": precision}
    sep = Separator.from_detector(det, norm=norm, k_pick=k_pick, **kw)
    # a background with a heavy upper side in the second frame: its tails overflow
    fr = rng.poisson(20, (2, det.npix)).astype(np.float32)
    fr[1] += np.where(rng.random(det.npix) < 0.3, rng.exponential(60, det.npix), 0).astype(np.float32)
    if with_norm:
        fr *= norm
    frames = torch.from_numpy(fr).cuda()
    o = sep.process_batch(frames, det.npix, 4096)
    s = sep.sparsify(frames, o["mean"], o["sigma"], det.npix)
    torch.cuda.synchronize()
    n_batch, n_alone = o["n_kept"].cpu().numpy(), s["n_kept"].cpu().numpy()
    for f in range(2):
        a = o["idx"][f, :n_batch[f]].cpu().numpy()
        b = s["idx"][f, :n_alone[f]].cpu().numpy()
        # the batch decides with the unrounded mean: a value on its threshold's
        # last place may go either way
        odd = np.setxor1d(a, b)
        assert odd.size <= max(2, det.npix // 20000), (f, odd.size)
        both = np.intersect1d(a, b)
        va = o["val"][f, :n_batch[f]].cpu().numpy()[np.isin(a, both)]
        vb = s["val"][f, :n_alone[f]].cpu().numpy()[np.isin(b, both)]
        assert np.array_equal(va.view(np.uint32), vb.view(np.uint32))
        assert np.all(np.diff(a) > 0) and a.size > 0
    assert sep.device_status() & 2 == 0
    sep.close()
