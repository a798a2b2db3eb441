"""Entry weights (a norm, area fractions) over the range of row lengths the clip
kernel takes: rows shorter than a warp's first loads, ordinary rows, and rows
so long that their tails hold few slots or none (every step a full pass)."""
import numpy as np
import pytest

import oracle
import synth
from parity import check_frame

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09515_gb300 import SepError, Separator  # noqa: E402


def detector(rows, cols, nbins):
    return synth.Detector("w", rows, cols, dist_m=0.1, center_px=(0.5 * cols, 0.5 * rows), nbins=nbins, split=1)


@pytest.mark.parametrize("rows,cols,nbins", [(9, 11, 40), (41, 37, 30), (256, 256, 2), (235, 234, 1)])
def test_rows_of_entry_weights(rows, cols, nbins):
    det = detector(rows, cols, nbins)
    rng = np.random.default_rng(rows)
    norm = rng.uniform(0.5, 2.0, det.npix).astype(np.float32)
    fr = (rng.normal(50, 7, (3, det.npix)) * norm).astype(np.float32)
    # a third frame with a heavy upper side: its tails run out of slots
    fr[2] += np.where(rng.random(det.npix) < 0.2, rng.exponential(90, det.npix), 0).astype(np.float32) * norm
    sep = Separator.from_detector(det, norm=norm)
    d = torch.from_numpy(fr).cuda()
    o = sep.process_batch(d, det.npix, 8192)
    bnd = sep.integrate_clip(d, bounds=True)["bounds"].cpu().numpy()
    o = {k: v.cpu().numpy() for k, v in o.items()}
    W = oracle.weights(det)
    for f in range(3):
        check_frame(det, W, fr[f], o, f, kcap=det.npix, bounds=bnd[f], norm=norm)
    sep.close()


def test_a_row_beyond_the_limit_is_refused():
    det = detector(250, 250, 1)
    sep = Separator.from_detector(det, norm=np.ones(det.npix, np.float32))
    with pytest.raises(SepError, match="shared memory"):
        sep.process_batch(torch.zeros((1, det.npix), dtype=torch.float32, device="cuda"), 16, 16)
    sep.close()
