"""Room for the pairs of a plain join by strings: lists sized by a sample that
misses most candidates are made again, and the output and the counters are those
of the general path."""
import numpy as np
import pytest

import synth
from gpu_util import to_device

pytestmark = pytest.mark.gpu

N, L, K = 2_100, 40, 3   # two strings in a stride of the sample


def _set(seen):
    """Half of the strings are copies of one, at the ranks that the sample visits
    or (strings of one length have ranks in order of their ids) at the others."""
    rng = np.random.Generator(np.random.PCG64(7))
    root = synth.DNA[rng.integers(0, 4, size=L)].tobytes()
    strs = [root if (t & 1) == (0 if seen else 1) else synth.DNA[rng.integers(0, 4, size=L)].tobytes()
            for t in range(N)]
    return synth.from_strings(strs, K=K, T=K)


def test_lists_that_the_sample_makes_too_short():
    import paper_1810_08833_gb300 as mj
    launches = {}
    for seen in (True, False):
        s = _set(seen)
        data, off = to_device(s)
        with mj.Context(0) as ctx:
            ref = ctx.join(data, off, mj.params(K, T=K, flags=mj.MJ_FLAG_DEDUP_SORT))
            want = ctx.stats()
        assert want["n_candidates"] >= (N // 2) * (N // 2 - 1) // 2
        with mj.Context(0) as ctx:
            for again in (False, True):   # lists that have grown stay as long
                got = ctx.join(data, off, mj.params(K, T=K))
                have = ctx.stats()
                for x, y in zip(ref, got):
                    assert np.array_equal(x.cpu().numpy(), y.cpu().numpy())
                for key in ("n_raw_pairs", "n_candidates", "n_output", "band_cells"):
                    assert want[key] == have[key], key
                launches[seen, again] = have["n_launches"]
    assert launches[False, False] == launches[True, False] + 2   # the pair kernel and the list kernel once more
    assert launches[False, True] == launches[True, True] == launches[True, False]


def test_more_pairs_than_a_first_list_holds():
    """700 copies of one string: windows of few ranks, but more pairs than the lists
    of a context's first joins hold."""
    import paper_1810_08833_gb300 as mj
    rng = np.random.Generator(np.random.PCG64(6))
    root = synth.DNA[rng.integers(0, 4, size=L)].tobytes()
    s = synth.from_strings([root] * 700 + [root[:-1]] * 40, K=K, T=K)
    data, off = to_device(s)
    with mj.Context(0) as ctx:
        ref = ctx.join(data, off, mj.params(K, T=K, flags=mj.MJ_FLAG_DEDUP_SORT))
        assert ref[0].shape[0] == 740 * 739 // 2
    with mj.Context(0) as ctx:
        got = ctx.join(data, off, mj.params(K, T=K))
    for x, y in zip(ref, got):
        assert np.array_equal(x.cpu().numpy(), y.cpu().numpy())


def test_only_the_second_list_is_made_again():
    """More pairs pass the second bound than there is room for at first (2^24):
    6,200 copies of one string under the bounds, all pairs relatives."""
    import paper_1810_08833_gb300 as mj
    rng = np.random.Generator(np.random.PCG64(8))
    n = 6_200
    root = synth.PROTEIN[rng.integers(0, 20, size=60)]
    strs = []
    for _ in range(n):
        c = root.copy()
        c[rng.integers(0, 60)] = synth.PROTEIN[rng.integers(0, 20)]
        strs.append(c.tobytes())
    s = synth.from_strings(strs, K=4, T=4)
    data, off = to_device(s)
    with mj.Context(0) as ctx:
        ref = ctx.join(data, off, mj.params(4, T=4, flags=mj.MJ_FLAG_DEDUP_SORT))
        want = ctx.stats()
        assert want["n_output"] > 1 << 24
        got = ctx.join(data, off, mj.params(4, T=4))
        have = ctx.stats()
    for x, y in zip(ref, got):
        assert np.array_equal(x.cpu().numpy(), y.cpu().numpy())
    for key in ("n_raw_pairs", "n_candidates", "n_output", "band_cells"):
        assert want[key] == have[key], key
