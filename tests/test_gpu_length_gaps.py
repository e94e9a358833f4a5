"""Plain joins of strings whose lengths leave gaps: the table of the first rank of
every length, against the general path, forced by a dedup flag."""
import numpy as np
import pytest

import synth
from gpu_util import to_device

pytestmark = pytest.mark.gpu


# the longest string, its T; 2^22 is the longest for which the table is made
@pytest.mark.parametrize("longest,T", [(200, 9), (5_000, 9), (70_000, 70), (1 << 20, 1000), (1 << 22, 4000),
                                       ((1 << 22) + 1, 4000)])
def test_one_long_string_among_short_ones(longest, T):
    import paper_1810_08833_gb300 as mj
    rng = np.random.Generator(np.random.PCG64(longest))
    strs = [b"", b"A", b"AC"]
    for _ in range(150):
        a = synth.DNA[rng.integers(0, 4, size=int(rng.choice([30, 31, 60, 64, 150])))]
        strs += [a.tobytes()] + [synth.mutate(rng, a, 0.03, synth.DNA).tobytes() for _ in range(3)]
    a = synth.DNA[rng.integers(0, 4, size=longest)]
    strs += [a.tobytes(), a[:-3].tobytes()]
    s = synth.from_strings(strs, K=9, T=T)
    data, off = to_device(s)
    with mj.Context(0) as ctx:
        ref = ctx.join(data, off, mj.params(s.K, T=s.T, flags=mj.MJ_FLAG_DEDUP_SORT))
        want = ctx.stats()
        got = ctx.join(data, off, mj.params(s.K, T=s.T))
        have = ctx.stats()
    assert want["n_output"] > 0
    for x, y in zip(ref, got):
        assert np.array_equal(x.cpu().numpy(), y.cpu().numpy())
    for key in ("n_partitions", "n_raw_pairs", "n_candidates", "n_output", "band_cells"):
        assert want[key] == have[key], key
