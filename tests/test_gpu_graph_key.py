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
