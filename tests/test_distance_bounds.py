"""The lower bound behind the candidates' signatures (CPU): for strings a and b
with counts of their q-grams, in any buckets and cut off at any count, the sum
of the counts' differences plus the length difference is at most 2 q ED."""
import numpy as np
import pytest

import oracle
import synth


def _counts(codes, q, buckets, cap, table):
    c = np.zeros(buckets, np.int64)
    for i in range(len(codes) - q + 1):
        c[table[int(sum(int(x) * 257 ** k for k, x in enumerate(codes[i:i + q])) % len(table))]] += 1
    return np.minimum(c, cap)


@pytest.mark.parametrize("symbols,q", [(synth.DNA, 1), (synth.DNA, 4), (synth.PROTEIN, 2), (synth.PRINTABLE, 1),
                                       (synth.PRINTABLE, 3)], ids=["dna1", "dna4", "protein2", "text1", "text3"])
@pytest.mark.parametrize("buckets,cap", [(28, 255), (256, 15), (8, 3)])
def test_gram_counts_bound_the_distance(symbols, q, buckets, cap):
    rng = np.random.Generator(np.random.PCG64(1000 * q + buckets + len(symbols)))
    table = rng.integers(0, buckets, size=4099)
    strs = []
    for _ in range(12):
        root = symbols[rng.integers(0, len(symbols), size=int(rng.integers(0, 60)))]
        strs += [root] + [synth.mutate(rng, root, r, symbols) for r in (0.05, 0.3, 0.9)]
    s = synth.from_strings([x.tobytes() for x in strs], K=4, T=4)
    pairs = np.array([(i, j) for i in range(s.n) for j in range(i + 1, s.n)], np.int64)
    ed = oracle.ed_band_pairs(s.bytes, s.offsets, pairs, 200)   # 200 exceeds every length: the full distance
    cnt = [_counts(x, q, buckets, cap, table) for x in strs]
    for (i, j), d in zip(pairs.tolist(), ed.tolist()):
        total = int(np.abs(cnt[i] - cnt[j]).sum()) + abs(len(strs[i]) - len(strs[j]))
        assert total <= 2 * q * d, (i, j, total, d)
