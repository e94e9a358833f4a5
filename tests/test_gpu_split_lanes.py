"""Short verification lists take from 2 to 32 lanes of each warp, by the number
of pairs: every count on both sides of a change gives the oracle's distances."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_1810_08833_gb300 as mj
    from paper_1810_08833_gb300 import build
    build.build()
    c = mj.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("symbols,K", [(4, 20), (20, 70), (100, 130), (250, 40)])
def test_every_number_of_lanes(ctx, symbols, K):
    import torch
    rng = np.random.Generator(np.random.PCG64(77 + K))
    abc = rng.permutation(np.arange(1, 256, dtype=np.uint8))[:symbols]
    strs = []
    for t in range(40):
        a = abc[rng.integers(0, symbols, size=int(rng.integers(1, 6 * K)))]
        b = synth.mutate(rng, a, float(rng.choice([0.02, 0.1, 0.5])), abc)
        strs += [a.tobytes(), b.tobytes()]
    strs += [b"", strs[0]]
    s = synth.from_strings(strs, K=K, T=max(2, K // 2))
    pairs = np.arange(len(strs), dtype=np.int64).reshape(-1, 2)
    want = oracle.ed_band_pairs(s.bytes, s.offsets, pairs, K, cutoff=True)
    data, off = to_device(s)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for lanes in (2, 4, 8, 16):
        for m in (2 * sms * lanes, 2 * sms * lanes + 1):   # a warp per scheduler, and one pair more
            take = np.arange(m) % len(pairs)
            i = torch.from_numpy(pairs[take, 0].astype(np.int32)).cuda()
            j = torch.from_numpy(pairs[take, 1].astype(np.int32)).cuda()
            got = ctx.verify(data, off, i, j, K).cpu().numpy().astype(np.int64)
            assert np.array_equal(got, want[take]), (lanes, m, np.nonzero(got != want[take])[0][:10])
    one = ctx.verify(data, off, i[:1].contiguous(), j[:1].contiguous(), K).cpu().numpy()
    assert one[0] == want[0]
