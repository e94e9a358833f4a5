"""Joins whose partition records fall on both sides of each size class of the
one-block sort: the records' keys (u32) and the general path's (u64) are
sorted by different classes, and both joins agree."""
import numpy as np
import pytest

import synth
from tests.gpu_util import to_device
from tests.test_gpu_string_joins import _set

pytestmark = pytest.mark.gpu


def test_records_of_every_size_class():
    import paper_1810_08833_gb300 as mj
    s = _set(41, 2600, 60, 140, synth.PROTEIN, K=9)
    seen = set()
    with mj.Context(0) as ctx:
        for n in range(60, 2600, 60):
            part = synth.from_strings([s.bytes[s.offsets[k]:s.offsets[k + 1]].tobytes() for k in range(n)], K=9, T=9)
            data, off = to_device(part)
            ref = ctx.join(data, off, mj.params(9, T=9, flags=mj.MJ_FLAG_DEDUP_SORT))
            want = ctx.stats()
            got = ctx.join(data, off, mj.params(9, T=9))
            have = ctx.stats()
            assert want["n_output"] > 0
            for a, b in zip(ref, got):
                assert np.array_equal(a.cpu().numpy(), b.cpu().numpy()), n
            for key in ("n_partitions", "n_raw_pairs", "n_candidates", "n_output"):
                assert want[key] == have[key], (n, key)
            seen.add(sum(want["n_partitions"] > e for e in (1024, 4096, 8192, 12288, 16384)))
    assert seen == {0, 1, 2, 3, 4, 5}, seen
