"""The dense background of few frames (four consecutive pixels a thread, vector
accesses) against NumPy, by bin and interpolated, with and without deviates, bit
for bit; an output or deviates off a 16-byte boundary take the other kernel."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09515_gb300 import Separator, _binding as B  # noqa: E402


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("smooth", [False, True])
@pytest.mark.parametrize("noisy", [False, True])
@pytest.mark.parametrize("rows,cols,F", [(2, 2, 1), (16, 8, 2), (33, 36, 1), (256, 256, 3), (1030, 1064, 1)])
def test_few_dense_frames(rows, cols, F, noisy, smooth, shift):
    rng = np.random.default_rng(rows + F)
    det = synth.Detector("d", rows, cols, dist_m=0.05, center_px=(0.4 * cols + 0.3, 0.6 * rows + 0.2),
                         nbins=min(40, max(2, rows * cols // 20)), split=1, unit=synth.UNIT_R_MM)
    n = det.npix
    mask = (rng.random(n) < 0.1).astype(np.uint8) if n > 4 else None
    sep = Separator.from_detector(det, mask=mask)
    bop = B.sep_csr_export(sep.csr)["bin_of_pixel"]
    mean = rng.uniform(0.2, 30, (F, det.nbins)).astype(np.float32)
    sigma = rng.uniform(0.1, 3, (F, det.nbins)).astype(np.float32)
    z = rng.standard_normal((F, n)).astype(np.float32)

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
    buf = torch.full((F * n + 1,), 7.0, device="cuda")
    out = buf[shift:shift + F * n].view(F, n)
    sep.densify(torch.from_numpy(mean).cuda(), torch.from_numpy(sigma).cuda(), None, None, None,
                noise=torch.from_numpy(z).cuda() if noisy else None, fill=-2.5, interpolate=smooth, out=out)
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().view(np.uint32), want.view(np.uint32))
    assert float(buf[0 if shift else -1]) == 7.0
    sep.close()
