"""Plain joins string by string (mj_pairs.cu) against the general path, forced
by a dedup flag: the same output and counters for every window kernel (16-bit
and wide windows, packed and unpacked visit words), alphabet, repetition count
and band, with and without the lower bounds on the distance."""
import numpy as np
import pytest

import synth
from tests.gpu_util import to_device

pytestmark = pytest.mark.gpu

N = 66_000   # more strings than a 16-bit window holds


def _set(seed, n, lo, hi, symbols, K, rate=0.05, extra=(), T=0):
    """n strings, half of them near copies in families of four."""
    rng = np.random.Generator(np.random.PCG64(seed))
    lens = rng.integers(lo, hi + 1, size=n // 4 + 1)
    parts = []
    for L in lens:
        root = symbols[rng.integers(0, len(symbols), size=int(L))]
        parts.append(root)
        parts.append(symbols[rng.integers(0, len(symbols), size=int(L))])
        parts += [synth.mutate(rng, root, rate, symbols) for _ in range(2)]
    strs = [p.tobytes() for p in parts[:n - len(extra)]] + list(extra)
    return synth.from_strings(strs, K=K, T=T or K)


CASES = [
    # name, set, repeats
    ("dna_few_candidates", lambda: _set(1, N, 60, 160, synth.DNA, K=6), 1),
    ("protein_bounds", lambda: _set(2, N, 40, 140, synth.PROTEIN, K=9), 1),
    ("two_letters_many_candidates", lambda: _set(3, N, 20, 40, synth.DNA[:2], K=3), 1),
    ("printable_two_repetitions", lambda: _set(4, N, 30, 90, synth.PRINTABLE, K=12), 2),
    ("one_length_wide_windows", lambda: _set(5, 72_000, 48, 48, synth.PROTEIN, K=5, rate=0.02), 1),
    ("odd_band_empty_strings", lambda: _set(6, N, 0, 50, synth.PROTEIN, K=7, extra=[b""] * 5), 1),
    ("a_string_over_2_16", lambda: _set(7, N, 30, 60, synth.PROTEIN, K=5, extra=[b"ACD" * 30_000], T=30), 1),
]


@pytest.mark.parametrize("name,factory,repeats", CASES, ids=[c[0] for c in CASES])
def test_join_by_strings_equals_general_path(name, factory, repeats):
    import paper_1810_08833_gb300 as mj
    s = factory()
    data, off = to_device(s)
    with mj.Context(0) as ctx:
        ref = ctx.join(data, off, mj.params(s.K, T=s.T, repeats=repeats, flags=mj.MJ_FLAG_DEDUP_SORT))
        want = ctx.stats()
        got = ctx.join(data, off, mj.params(s.K, T=s.T, repeats=repeats))
        have = ctx.stats()
        assert want["n_output"] > 0 and want["n_candidates"] > 0
        for a, b in zip(ref, got):
            assert np.array_equal(a.cpu().numpy(), b.cpu().numpy())
        for key in ("n_partitions", "n_raw_pairs", "n_candidates", "n_output", "band_cells"):
            assert want[key] == have[key], key


def test_candidates_after_a_join_by_strings():
    """mj_candidates_copy after a plain join still gives the join's candidates,
    also when partitions of another input were made in between."""
    import paper_1810_08833_gb300 as mj
    s = _set(11, N, 40, 120, synth.PROTEIN, K=8)
    other = _set(12, 500, 40, 120, synth.PROTEIN, K=8)
    data, off = to_device(s)
    d2, o2 = to_device(other)
    p = mj.params(s.K, T=s.T)
    with mj.Context(0) as ctx:
        want = [t.cpu().numpy() for t in ctx.candidates(data, off, p)]
        for between in (False, True):
            ctx.join(data, off, p)
            m = ctx.stats()["n_candidates"]
            assert m == want[0].shape[0]
            if between:
                ctx.partition(d2, o2, p)
            ci, cj = ctx._copy_candidates(m, data.device)
            assert np.array_equal(ci.cpu().numpy(), want[0]) and np.array_equal(cj.cpu().numpy(), want[1])


@pytest.mark.parametrize("bands", [False, True])
def test_long_list_under_the_bounds(bands):
    """Verification of a list long enough for the lower bounds, most of its
    pairs unrelated, equals the oracle."""
    import oracle
    import paper_1810_08833_gb300 as mj
    import torch
    s = _set(51, 160, 60, 110, synth.PROTEIN, K=9)
    m, K = (1 << 20) + 77, 9
    rng = np.random.Generator(np.random.PCG64(52))
    pairs = rng.integers(0, 160, size=(m, 2))
    k = rng.integers(2, K + 1, size=m) if bands else np.full(m, K)
    every = np.stack(np.meshgrid(np.arange(160), np.arange(160), indexing="ij"), axis=-1).reshape(-1, 2)
    full = oracle.ed_band_pairs(s.bytes, s.offsets, every.astype(np.int64), K, cutoff=True).reshape(160, 160)
    want = np.minimum(full[pairs[:, 0], pairs[:, 1]], k + 1)
    data, off = to_device(s)
    with mj.Context(0) as ctx:
        i, j = (torch.from_numpy(pairs[:, c].astype(np.int32)).cuda() for c in (0, 1))
        bd = torch.from_numpy(k.astype(np.int32)).cuda() if bands else None
        got = ctx.verify(data, off, i, j, K, k=bd).cpu().numpy().astype(np.int64)
    assert np.array_equal(got, want), np.nonzero(got != want)[0][:10]
