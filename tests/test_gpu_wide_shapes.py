"""Wide-band verification with several 32-row words per lane: bands at the
widest that each shape holds and one row more, over alphabets of two, five and
eight bit-planes, with pair lists long enough for the shapes that share a warp
and short ones.  Equal to the oracle's banded DP."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import to_device

pytestmark = pytest.mark.gpu

WAVEFRONT = 2

# G lanes of V words hold bands of G (32 V + 1) - 32 V rows + 1
WIDEST = [G * (32 * V + 1) - 32 * V
          for G, V in [(4, 4), (8, 2), (4, 6), (8, 3), (8, 4), (16, 2), (8, 5), (16, 3), (32, 2), (16, 5), (32, 3), (32, 4), (32, 6),
                       (32, 8)]]


@pytest.fixture(scope="module")
def ctx():
    import paper_1810_08833_gb300 as mj
    from paper_1810_08833_gb300 import build
    build.build()
    c = mj.Context(0)
    yield c
    c.close()


def _pairs(seed, K, symbols):
    """Pairs on both sides of K: planted edits near K and below it, length
    differences of K and K + 1, unrelated strings, short and empty ones."""
    rng = np.random.Generator(np.random.PCG64(seed))
    abc = rng.permutation(np.arange(1, 256, dtype=np.uint8))[:symbols]
    strs = []
    for t in range(12):
        L = int(rng.integers(K + 2, 3 * K + 200))
        a = abc[rng.integers(0, symbols, size=L)]
        if t % 6 == 0:
            b = synth.mutate(rng, a, min(0.9, 1.2 * K / L), abc)
        elif t % 6 == 1:
            b = a[:L - K]
        elif t % 6 == 2:
            b = a[:L - K - 1]
        elif t % 6 == 3:
            b = synth.mutate(rng, a, 0.4 * K / L, abc)
        elif t % 6 == 4:
            b = abc[rng.integers(0, symbols, size=max(1, L - int(rng.integers(0, K))))]
        else:
            a = a[:int(rng.integers(1, 300))]
            b = synth.mutate(rng, a, 0.3, abc)
        strs += [a.tobytes(), b.tobytes()]
    strs += [b"", strs[0]]
    n = len(strs)
    pairs = np.arange(n, dtype=np.int64).reshape(-1, 2)
    return synth.from_strings(strs, K=K, T=max(2, K // 5)), pairs


@pytest.mark.parametrize("symbols", [4, 20, 200])
@pytest.mark.parametrize("K", sorted({k + d for k in WIDEST for d in (0, 1)}))
def test_widest_band_of_each_shape(ctx, K, symbols):
    import torch
    s, pairs = _pairs(9000 + K + symbols, K, symbols)
    want = oracle.ed_band_pairs(s.bytes, s.offsets, pairs, K, cutoff=True)
    data, off = to_device(s)
    ctx.set_verify_config(WAVEFRONT, 0)
    try:
        for copies in ((1, 300, 3000) if K < 1000 else (1, 200)):
            i = torch.from_numpy(np.tile(pairs[:, 0], copies).astype(np.int32)).cuda()
            j = torch.from_numpy(np.tile(pairs[:, 1], copies).astype(np.int32)).cuda()
            got = ctx.verify(data, off, i, j, K).cpu().numpy().astype(np.int64)
            assert np.array_equal(got, np.tile(want, copies)), np.nonzero(got != np.tile(want, copies))[0][:10]
            swapped = ctx.verify(data, off, j, i, K).cpu().numpy().astype(np.int64)
            assert np.array_equal(swapped, got)
    finally:
        ctx.set_verify_config(0, 0)


@pytest.mark.parametrize("symbols", [4, 200])
@pytest.mark.parametrize("K", [3, 63, 64, 200, 256, 300])
def test_narrow_bands_in_wide_shapes(ctx, K, symbols):
    """Bands that the narrowest shape holds with room to spare."""
    import torch
    s, pairs = _pairs(700 + K + symbols, K, symbols)
    want = oracle.ed_band_pairs(s.bytes, s.offsets, pairs, K, cutoff=True)
    data, off = to_device(s)
    i = torch.from_numpy(np.tile(pairs[:, 0], 1600).astype(np.int32)).cuda()
    j = torch.from_numpy(np.tile(pairs[:, 1], 1600).astype(np.int32)).cuda()
    ctx.set_verify_config(WAVEFRONT, 0)
    try:
        got = ctx.verify(data, off, i, j, K).cpu().numpy().astype(np.int64)
    finally:
        ctx.set_verify_config(0, 0)
    assert np.array_equal(got, np.tile(want, 1600)), np.nonzero(got != np.tile(want, 1600))[0][:10]
