"""Plain joins whose windows hold 2^16 ranks and more: with few candidates they
take the general path, with many they go string by string, and both equal the
general path forced by a dedup flag."""
import numpy as np
import pytest

import synth
from gpu_util import to_device

pytestmark = pytest.mark.gpu

N, L, K = 72_000, 30, 4


def _set(copies, pair_of_long):
    """N strings of one length, in families of `copies` with a substitution each."""
    rng = np.random.Generator(np.random.PCG64(copies))
    x = synth.PROTEIN[rng.integers(0, 20, size=(N // copies, L))].repeat(copies, axis=0)
    x[np.arange(N), rng.integers(0, L, size=N)] = synth.PROTEIN[rng.integers(0, 20, size=N)]
    x = x[rng.permutation(N)]
    strs = [r.tobytes() for r in x]
    if pair_of_long:   # visit words of 24 bytes
        a = synth.PROTEIN[rng.integers(0, 20, size=70_000)]
        b = a.copy()
        b[[5, 69_000]] = synth.PROTEIN[:2]
        strs += [a.tobytes(), b.tobytes()]
    return synth.from_strings(strs, K=K, T=16 if pair_of_long else K)   # the radius of 70,000 symbols fits


@pytest.mark.parametrize("copies,many", [(2, False), (40, True)])
@pytest.mark.parametrize("pair_of_long", [False, True])
@pytest.mark.parametrize("repeats", [1, 2])
def test_wide_windows(copies, many, pair_of_long, repeats):
    import paper_1810_08833_gb300 as mj
    s = _set(copies, pair_of_long)
    data, off = to_device(s)
    with mj.Context(0) as ctx:
        ref = ctx.join(data, off, mj.params(K, T=s.T, repeats=repeats, flags=mj.MJ_FLAG_DEDUP_SORT))
        want = ctx.stats()
        for _ in range(2):
            got = ctx.join(data, off, mj.params(K, T=s.T, repeats=repeats))
            have = ctx.stats()
            if repeats == 1 and not pair_of_long:   # the general path counts its pairs first
                assert (have["ms_section"]["pair_emission"] == 0) == many
            for x, y in zip(ref, got):
                assert np.array_equal(x.cpu().numpy(), y.cpu().numpy())
            for key in ("n_partitions", "n_raw_pairs", "n_candidates", "n_output", "band_cells"):
                assert want[key] == have[key], key
