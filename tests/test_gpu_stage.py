"""The staging kernel's load paths (vector, word and plain loads) and its
groups of frames: the values of kept pixels and the profiles of a batch are
the same for aligned and unaligned frames, for every width modulo 4, and for
frame counts that leave a remainder behind a step, bit for bit."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09515_gb300 import Context, Separator, process_mixed  # noqa: E402


@pytest.mark.parametrize("with_norm", [False, True])
@pytest.mark.parametrize("raw", [False, True])
@pytest.mark.parametrize("rows,cols,F", [(64, 64, 4), (65, 66, 5), (70, 131, 3), (127, 129, 9), (130, 200, 1),
                                         (40, 61, 700)])
def test_staged_values(rows, cols, F, raw, with_norm):
    rng = np.random.default_rng(rows * cols + F)
    det = synth.Detector("s", rows, cols, dist_m=0.05, center_px=(0.4 * cols, 0.6 * rows), nbins=20, split=2)
    n = det.npix
    mask = (rng.random(n) < 0.05).astype(np.uint8)
    cal = synth.jf_calib(n, seed=2) if raw else None
    norm = rng.uniform(0.5, 2.0, n).astype(np.float32) if with_norm else None
    ctx = Context(0)
    sep = Separator.from_detector(det, mask=mask, calib=cal, norm=norm, k_pick=0.0, context=ctx)
    if raw:
        words = rng.integers(0, 1 << 16, (F, n), dtype=np.uint16)
        v = np.stack([oracle.jf_photons(w, cal[0], cal[1]) for w in words])
    else:
        words = rng.normal(10, 3, (F, n)).astype(np.float32)
        v = words
    v = v if norm is None else (v / norm).astype(np.float32)
    t = torch.from_numpy(words.view(np.int16) if raw else words)
    aligned = t.cuda()
    outs = []
    for shift in (0, 1, 2):   # elements past an aligned address
        buf = torch.zeros(t.numel() + shift, dtype=t.dtype, device="cuda")
        frames = buf[shift:].view(t.shape)
        frames.copy_(aligned)
        o = sep.process_batch(frames, n, 64)
        torch.cuda.synchronize()
        outs.append({k: x.cpu().numpy() for k, x in o.items()})
    for o in outs:
        assert np.array_equal(o["mean"].view(np.uint32), outs[0]["mean"].view(np.uint32))
        assert np.array_equal(o["sigma"].view(np.uint32), outs[0]["sigma"].view(np.uint32))
        assert np.array_equal(o["n_kept"], outs[0]["n_kept"])
        for f in range(0, F, max(1, F // 7)):
            k = o["n_kept"][f]
            i = o["idx"][f, :k]
            assert k > 0 and np.array_equal(o["val"][f, :k].view(np.uint32), v[f, i].view(np.uint32))
    # a list of frames at mixed addresses
    m = min(F, 6)
    lst = [(0, aligned[f].clone() if f % 2 else buf[2:].view(t.shape)[f]) for f in range(m)]
    q = process_mixed([sep], lst, n, 64)
    torch.cuda.synchronize()
    assert np.array_equal(q["mean"].cpu().numpy().reshape(m, -1).view(np.uint32), outs[0]["mean"][:m].view(np.uint32))
    assert np.array_equal(q["n_kept"].cpu().numpy(), outs[0]["n_kept"][:m])
    sep.close()
    ctx.close()
