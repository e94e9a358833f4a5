"""What a replayed verification graph may not take from the call that captured
it: results and counters of calls that differ in something the captured
launches hold by value equal those of a context without graphs."""
import numpy as np
import pytest

import synth
from gpu_util import to_device

pytestmark = pytest.mark.gpu

COUNTERS = ("n_partitions", "n_raw_pairs", "n_candidates", "n_output", "band_cells", "verify_word_columns")


@pytest.mark.parametrize("flag", ["MJ_FLAG_DEDUP_SORT", "MJ_FLAG_DEDUP_BITMAP", "MJ_FLAG_KEY_CHECK"])
def test_joins_by_another_path_after_a_capture(flag):
    """A plain join's graph holds no ordering, and with it no sum of the
    K-band cells; the general path's joins of the same input read that sum."""
    import paper_1810_08833_gb300 as mj
    import torch
    s = synth.make_config(1, n_roots=20)
    data, off = to_device(s)
    plain, other = mj.params(s.K, T=s.T), mj.params(s.K, T=s.T, flags=getattr(mj, flag))
    with mj.Context(0) as ctx:
        ctx.join(data, off, other)
        want = ctx.stats()
    assert want["band_cells"] > 0
    stream = torch.cuda.Stream()
    with mj.Context(0) as ctx:
        ctx.set_verify_config(mj.MJ_VERIFY_KERNEL_AUTO, 0, 0, 1)
        for p in (plain, plain, plain, other, other, other, plain):   # uncaptured, captured, replayed
            ctx.join(data, off, p, stream=stream)
            have = ctx.stats()
            for key in COUNTERS:
                assert have[key] == want[key], (key, p.flags)


def test_another_alphabet_in_the_same_buffers():
    """Bytes refilled in place with another alphabet of as many bits: the
    replay reads the new rank codes (ACGT, then ACGN and CGNT: the order of the
    codes changes with the letters)."""
    import oracle
    import paper_1810_08833_gb300 as mj
    import torch
    rng = np.random.Generator(np.random.PCG64(91))
    K, strs, pairs = 20, [], []
    for t in range(200):
        a = synth.DNA[rng.integers(0, 4, size=int(rng.integers(40, 300)))]
        strs += [a.tobytes(), synth.mutate(rng, a, 0.04, synth.DNA).tobytes()]
        pairs.append((2 * t, 2 * t + 1))
    s = synth.from_strings(strs, K=K, T=K)
    pairs = np.asarray(pairs, dtype=np.int64)
    data, off = to_device(s)
    i, j = (torch.from_numpy(pairs[:, c].astype(np.int32)).cuda() for c in (0, 1))
    stream = torch.cuda.Stream()
    with mj.Context(0) as ctx:
        ctx.set_verify_config(mj.MJ_VERIFY_KERNEL_AUTO, 0, 0, 1)
        for letters in (b"ACGT", b"ACGN", b"CGNT"):
            table = np.zeros(256, dtype=np.uint8)
            for x, y in zip(b"ACGT", letters):
                table[x] = y
            new = table[s.bytes]
            want = oracle.ed_band_pairs(new, s.offsets, pairs, K)
            data.copy_(torch.from_numpy(new))
            torch.cuda.synchronize()
            for _ in range(3):
                got = None   # its memory again: the key holds the output's address
                with torch.cuda.stream(stream):
                    got = ctx.verify(data, off, i, j, K, stream=stream)
                stream.synchronize()
                assert np.array_equal(got.cpu().numpy().astype(np.int64), want), letters
