"""Loss and gradient of the surrogate network where a CTA walks several tiles of
rows (304 CTAs of 64 rows at once), with a ragged last one, and with a gradient
output that is not aligned for vector atomics."""
import numpy as np
import pytest

from oracle import mlp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2411_09515_gb300 import Context, Surrogate, _binding as B  # noqa: E402


@pytest.mark.parametrize("n,shift", [(64, 1), (777, 1), (19457, 0), (60001, 0), (60001, 3)])
def test_gradient_over_tiles(n, shift):
    ctx = Context(0)
    s = Surrogate(ctx, seed=3)
    theta = (mlp.init(9) * 0.9).astype(np.float32)
    s.params(theta)
    rng = np.random.default_rng(n)
    x = rng.normal(0, 1, (n, mlp.N_IN)).astype(np.float32)
    t = rng.normal(0, 1, (n, mlp.N_OUT)).astype(np.float32)
    buf = torch.full((B.SEP_MLP_PARAMS + 8,), 7.0, dtype=torch.float32, device="cuda")
    g = buf[shift:shift + B.SEP_MLP_PARAMS]
    loss = torch.full((1,), 7.0, dtype=torch.float32, device="cuda")
    B.sep_mlp_loss_grad(s.ctx, s.model, torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), n, g, loss)
    torch.cuda.synchronize()
    th = torch.from_numpy(theta).to(torch.bfloat16).double().numpy()
    want = mlp.grad(th, x.astype(np.float64), t.astype(np.float64))
    got = g.cpu().numpy().astype(np.float64)
    assert float(loss) == pytest.approx(mlp.loss(th, x.astype(np.float64), t.astype(np.float64)), rel=1e-4)
    assert np.linalg.norm(got - want) < 1e-4 * np.linalg.norm(want)
    assert np.allclose(got, want, rtol=1e-3, atol=1e-4 * np.abs(want).max())
    rest = buf.cpu().numpy()
    assert (rest[:shift] == 7).all() and (rest[shift + B.SEP_MLP_PARAMS:] == 7).all()
    s.close()
    ctx.close()
