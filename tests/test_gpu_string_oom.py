"""Plain joins by strings where device memory runs out: an allocation that only
they make, made to fail on the host, sends the join to the general path, which
gives the same output; only the general path's own failures are MJ_ERR_OOM."""
import numpy as np
import pytest

import synth
from gpu_util import to_device

pytestmark = pytest.mark.gpu

KEYS = ("n_partitions", "n_raw_pairs", "n_candidates", "n_output", "band_cells")


def _wide():
    """Windows of 2^16 ranks with many pairs, which go by strings after the estimate."""
    rng = np.random.Generator(np.random.PCG64(5))
    x = synth.PROTEIN[rng.integers(0, 20, size=(1_800, 30))].repeat(40, axis=0)
    x[np.arange(72_000), rng.integers(0, 30, size=72_000)] = synth.PROTEIN[rng.integers(0, 20, size=72_000)]
    return synth.from_strings([r.tobytes() for r in x], K=4, T=4)


@pytest.mark.parametrize("name", ["reads", "protein", "wide"])
def test_every_allocation_of_a_join(name):
    import paper_1810_08833_gb300 as mj
    lib = mj.library()
    s = {"reads": lambda: synth.make_config(1, n_roots=20), "protein": lambda: synth.make_config(4, n_roots=400),
         "wide": _wide}[name]()
    data, off = to_device(s)
    with mj.Context(0) as ctx:
        ref = [t.cpu().numpy() for t in ctx.join(data, off, mj.params(s.K, T=s.T, flags=mj.MJ_FLAG_DEDUP_SORT))]
        want = ctx.stats()
    p = mj.params(s.K, T=s.T)
    joined, failed = 0, 0
    try:
        for nth in range(1, 60):
            with mj.Context(0) as ctx:
                lib.mj_inject_alloc_failure(nth)
                try:
                    got = ctx.join(data, off, p)
                    joined += 1
                except mj.MinJoinError as e:
                    assert e.status == -3
                    got = None
                    failed += 1
                lib.mj_inject_alloc_failure(0)
                for out in (got, ctx.join(data, off, p)):   # and again with allocations working
                    if out is not None:
                        have = ctx.stats()
                        assert all(np.array_equal(a.cpu().numpy(), b) for a, b in zip(out, ref)), nth
                        assert all(want[k] == have[k] for k in KEYS), nth
    finally:
        lib.mj_inject_alloc_failure(0)
    general = 0   # what the general path allocates and cannot do without
    for nth in range(1, 60):
        with mj.Context(0) as ctx:
            lib.mj_inject_alloc_failure(nth)
            try:
                ctx.join(data, off, mj.params(s.K, T=s.T, flags=mj.MJ_FLAG_DEDUP_SORT))
            except mj.MinJoinError as e:
                assert e.status == -3
                general += 1
            lib.mj_inject_alloc_failure(0)
    assert joined > 0 and failed > 0
    assert failed <= general, (failed, general)
