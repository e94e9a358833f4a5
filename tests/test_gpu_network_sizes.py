"""The band network's kernels at the edges of their 64-sample chunks and past
the blocks that run at once, against the float64 network."""
import numpy as np
import pytest

from oracle import mlp

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau", [0.0, 0.9])
@pytest.mark.parametrize("m", [1, 63, 64, 65, 1024, 19_520, 20_001])
def test_forward_and_gradient_at_chunk_edges(m, tau):
    import torch
    import paper_1810_08833_gb300 as mj
    rng = np.random.Generator(np.random.PCG64(m))
    x = rng.random((m, mj.BAND_FEATURES)).astype(np.float32)
    y = rng.random(m).astype(np.float32)
    w = rng.normal(0, 0.3, mj.BAND_PARAMS).astype(np.float32)
    with mj.Context(0) as ctx:
        ctx.band_init(seed=1)
        ctx.band_set_weights(w)
        xd, yd = torch.from_numpy(x).cuda(), torch.from_numpy(y).cuda()
        got = ctx.band_forward(xd).cpu().numpy()
        g, loss = ctx.band_grad(xd, yd, tau=tau)
        again, loss2 = ctx.band_grad(xd, yd, tau=tau)
    want = mlp.forward(w.astype(np.float64), x.astype(np.float64))
    # FP32 sums of 64 products over three layers: a few hundred roundings of 6e-8
    assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
    args = (w.astype(np.float64), x.astype(np.float64), y.astype(np.float64), tau)
    wl, wg = mlp.grad(*args)
    assert abs(loss - wl) <= 1e-5 * abs(wl)
    assert np.linalg.norm(g.cpu().numpy() - wg) <= 1e-4 * np.linalg.norm(wg)
    assert loss == loss2 and torch.equal(g, again)   # summed in a fixed order
