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
@pytest.mark.parametrize("alone", [False, True])
def test_a_long_string_among_short_ones(longest, T, alone):
    """alone: no other string is within K of its length (its records are in no
    window, so they do not decide the form of the visit words)."""
    import paper_1810_08833_gb300 as mj
    rng = np.random.Generator(np.random.PCG64(longest))
    strs = [b"", b"A", b"AC"]
    for _ in range(150):
        a = synth.DNA[rng.integers(0, 4, size=int(rng.choice([30, 31, 60, 64, 150])))]
        strs += [a.tobytes()] + [synth.mutate(rng, a, 0.03, synth.DNA).tobytes() for _ in range(3)]
    a = synth.DNA[rng.integers(0, 4, size=longest)]
    strs += [a.tobytes()] if alone else [a.tobytes(), a[:-3].tobytes()]
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


def test_bounds_leave_long_strings_to_the_verifier():
    """A list long enough for the lower bounds, with strings just below, at and
    above 2^15 symbols, from where a string has no signature."""
    import oracle
    import paper_1810_08833_gb300 as mj
    import torch
    rng = np.random.Generator(np.random.PCG64(9))
    K, strs = 9, []
    for L in (100, 2_000, (1 << 15) - 1, 1 << 15, 40_000):
        a = synth.PROTEIN[rng.integers(0, 20, size=L)]
        b = a.copy()
        b[[L // 3, L // 2]] = synth.PROTEIN[:2]
        strs += [a.tobytes(), b.tobytes(), synth.PROTEIN[rng.integers(0, 20, size=L - 2)].tobytes()]
    s = synth.from_strings(strs, K=K, T=K)
    n, m = len(strs), (1 << 20) + 5
    every = np.stack(np.meshgrid(np.arange(n), np.arange(n), indexing="ij"), axis=-1).reshape(-1, 2).astype(np.int64)
    want = oracle.ed_band_pairs(s.bytes, s.offsets, every, K, cutoff=True).reshape(n, n)
    pairs = rng.integers(0, n, size=(m, 2))
    data, off = to_device(s)
    with mj.Context(0) as ctx:
        i, j = (torch.from_numpy(pairs[:, c].astype(np.int32)).cuda() for c in (0, 1))
        got = ctx.verify(data, off, i, j, K).cpu().numpy().astype(np.int64)
    assert np.array_equal(got, want[pairs[:, 0], pairs[:, 1]])
