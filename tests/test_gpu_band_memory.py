"""Device memory of the band network: a context that is given weights makes room
for gradients only when it takes one, and an allocation that fails then leaves it
usable."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_partial_sums_wait_for_a_gradient():
    import paper_1810_08833_gb300 as mj
    import torch
    lib = mj.library()
    rng = np.random.Generator(np.random.PCG64(3))
    x = torch.from_numpy(rng.random((300, mj.BAND_FEATURES), dtype=np.float32)).cuda()
    y = torch.from_numpy(rng.random(300, dtype=np.float32)).cuda()
    with mj.Context(0) as a:
        a.band_init(seed=3)
        w = a.band_weights()
        want, loss = a.band_grad(x, y, tau=0.9)
        with mj.Context(0) as b:
            b.band_set_weights(w)
            try:
                lib.mj_inject_alloc_failure(1)   # no allocation: the injection stays armed
                assert torch.equal(b.band_forward(x), a.band_forward(x))
                with pytest.raises(mj.MinJoinError) as e:
                    b.band_grad(x, y, tau=0.9)
                assert e.value.status == -3
            finally:
                lib.mj_inject_alloc_failure(0)
            got, other = b.band_grad(x, y, tau=0.9)
            assert torch.equal(got, want) and other == loss
