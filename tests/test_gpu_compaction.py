"""The ordered compaction with every pixel kept, at sizes around a tile of the
bitmap (2048 words), for grids on both sides of the rule on threads a tile, and
with capacities that end inside a tile and inside a list."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09515_gb300 import Separator  # noqa: E402


@pytest.mark.parametrize("share", [1.0, 0.5, 0.01])
@pytest.mark.parametrize("rows,cols,F", [(8, 4, 1), (256, 256, 1), (257, 256, 2), (300, 301, 40), (512, 521, 3),
                                         (60, 61, 303), (60, 61, 305), (300, 301, 160)])
def test_kept_lists(rows, cols, F, share):
    n = rows * cols
    det = synth.Detector("c", rows, cols, dist_m=0.05, center_px=(0.4 * cols, 0.6 * rows), nbins=8, split=1)
    sep = Separator.from_detector(det, k_pick=1.0)
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    frames = 2 + torch.rand((F, n), generator=g, device="cuda")
    if share < 1:
        frames[torch.rand((F, n), generator=g, device="cuda") >= share] = 0
    m = torch.zeros((F, sep.nbins), dtype=torch.float32, device="cuda")
    s = torch.ones_like(m)
    n_kept = (frames > 1).sum(1)
    for cap in {n, max(1, n // 2 - 1), 2049, 5}:
        o = sep.sparsify(frames, m, s, cap)
        assert torch.equal(o["n_kept"].long(), n_kept)
        for f in range(0, F, max(1, F // 5)):
            want = (frames[f] > 1).nonzero()[:cap, 0]
            assert torch.equal(o["idx"][f, :want.numel()].long(), want)
            assert torch.equal(o["val"][f, :want.numel()], frames[f, want])
        assert (sep.device_status() != 0) == (int(n_kept.max()) > cap)
    sep.close()
