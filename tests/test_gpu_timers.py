"""The phase and section times of mj_join, when the call passes more points than
usual: many repetitions, or a verification launch per length bucket."""
import numpy as np
import pytest

import synth
from gpu_util import to_device

pytestmark = pytest.mark.gpu

PHASES = ("ms_derive", "ms_partition", "ms_join_filter", "ms_verify")


def _check(st, sections):
    for key in PHASES:
        assert st[key] > 0, (key, st)
    # the phases follow one another on one stream; each time is rounded to 0.5 us
    assert abs(sum(st[k] for k in PHASES) - st["ms_total"]) <= 0.02 + 1e-3 * st["ms_total"], st
    for key in sections:
        assert 0 < st["ms_section"][key] <= st["ms_total"], (key, st)
    assert st["ms_section"]["anchor_test"] <= st["ms_partition"] + 0.01
    assert st["ms_section"]["verify_kernel"] <= st["ms_verify"] + 0.01
    assert st["ms_section"]["pair_dedup"] <= st["ms_join_filter"] + 0.01


@pytest.mark.parametrize("repeats", [1, 16, 64])
@pytest.mark.parametrize("flag", [None, "MJ_FLAG_DEDUP_SORT"])
def test_times_of_many_repetitions(repeats, flag):
    import paper_1810_08833_gb300 as mj
    s = synth.make_config(1, n_roots=20)
    data, off = to_device(s)
    p = mj.params(s.K, T=s.T, repeats=repeats, flags=getattr(mj, flag) if flag else 0)
    with mj.Context(0) as ctx:
        for _ in range(2):
            ctx.join(data, off, p)
        _check(ctx.stats(), ("anchor_test", "partition_records", "record_sort", "pair_dedup", "verify_kernel",
                             "output_compaction"))


def test_times_of_a_launch_per_length_bucket():
    import paper_1810_08833_gb300 as mj
    rng = np.random.Generator(np.random.PCG64(5))
    strs = []
    for e in range(4, 14):   # lengths from 2^4 to 2^13
        for _ in range(6):
            a = synth.DNA[rng.integers(0, 4, size=int(rng.integers(2 ** e, 2 ** (e + 1))))]
            strs += [a.tobytes(), synth.mutate(rng, a, 4 / (2 ** e + 40), synth.DNA).tobytes()]
    s = synth.from_strings(strs, K=20, T=20)
    data, off = to_device(s)
    p = mj.params(s.K, T=s.T, repeats=8)
    with mj.Context(0) as ctx:
        ci, cj = ctx.candidates(data, off, p)
        ctx.autotune_verify(data, off, ci, cj, s.K, sample=32)
        ctx.set_verify_config(mj.MJ_VERIFY_KERNEL_TUNED, 0, 1, 0)
        for _ in range(2):
            ctx.join(data, off, p)
        _check(ctx.stats(), ("anchor_test", "verify_kernel", "output_compaction"))
