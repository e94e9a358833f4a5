"""mj_candidates_copy after a plain join by strings: the candidates of
mj_candidates, whether the join's own list holds them all (no lower bounds) or
not, also after other calls, again, on another stream, and under stream capture."""
import ctypes

import numpy as np
import pytest

import synth
from gpu_util import to_device

pytestmark = pytest.mark.gpu


def _sets():
    rng = np.random.Generator(np.random.PCG64(3))
    text = [synth.PRINTABLE[rng.integers(0, 3, size=int(rng.integers(300, 330)))] for _ in range(600)]
    return {"all_listed": synth.make_config(1, n_roots=30),
            # three letters (grams of six symbols), more candidates than joins without bounds have
            "bounded": synth.from_strings([t.tobytes() for t in text], K=4, T=100)}


def _copy(lib, ctx, m, stream=None):
    import torch
    out = [torch.full((m,), -1, dtype=torch.int32, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    assert lib.mj_candidates_copy(ctypes.c_void_p(ctx._h.value), out[0].data_ptr(), out[1].data_ptr(),
                                  stream.cuda_stream if stream else None) == 0
    return out


@pytest.mark.parametrize("name", ["all_listed", "bounded"])
@pytest.mark.parametrize("between", [None, "partition", "verify", "stream", "capture"])
def test_candidates_after_a_join(name, between):
    import paper_1810_08833_gb300 as mj
    import torch
    lib = mj.library()
    s = _sets()[name]
    data, off = to_device(s)
    p = mj.params(s.K, T=s.T)
    other, o2 = to_device(synth.make_config(4, n_roots=30))
    with mj.Context(0) as ctx:
        want = [t.cpu().numpy() for t in ctx.candidates(data, off, p)]
    with mj.Context(0) as ctx:
        for _ in range(2):
            ref = [t.cpu().numpy() for t in ctx.join(data, off, p)]
            st = ctx.stats()
            m = st["n_candidates"]
            assert m == want[0].shape[0] > (1 << 15 if name == "bounded" else 0)
            stream = torch.cuda.Stream()
            if between == "partition":
                ctx.partition(other, o2, mj.params(40, T=40))
            elif between == "verify":
                i = torch.arange(0, 100, dtype=torch.int32, device="cuda")
                ctx.verify(data, off, i, i.flip(0).contiguous(), s.K)
            if between == "capture":
                out = [torch.full((m,), -1, dtype=torch.int32, device="cuda") for _ in range(2)]
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.graph(graph, stream=stream):
                    got = lib.mj_candidates_copy(ctypes.c_void_p(ctx._h.value), out[0].data_ptr(),
                                                 out[1].data_ptr(), stream.cuda_stream)
                assert got == 0
                torch.cuda.synchronize()
                assert (out[0] == -1).all()   # captured, not run
                graph.replay()
            else:
                out = _copy(lib, ctx, m, stream if between == "stream" else None)
            torch.cuda.synchronize()
            for _ in range(2):   # and once more, from the list made
                assert all(np.array_equal(a.cpu().numpy(), b) for a, b in zip(out, want))
                out = _copy(lib, ctx, m)
                torch.cuda.synchronize()
            if between is None:
                assert ctx.stats() == st   # the join's counters and times stay
                res = [torch.empty(ref[0].shape[0], dtype=torch.int32, device="cuda") for _ in range(3)]
                assert lib.mj_result_copy(ctypes.c_void_p(ctx._h.value), *[r.data_ptr() for r in res], None) == 0
                torch.cuda.synchronize()
                assert all(np.array_equal(a.cpu().numpy(), b) for a, b in zip(res, ref))


@pytest.mark.parametrize("name", ["all_listed", "bounded"])
def test_allocation_failures(name):
    """Any allocation of the pass made to fail: the general path's candidates, or
    MJ_ERR_OOM and the candidates at the next call."""
    import paper_1810_08833_gb300 as mj
    import torch
    lib = mj.library()
    s = _sets()[name]
    data, off = to_device(s)
    p = mj.params(s.K, T=s.T)
    with mj.Context(0) as ctx:
        want = [t.cpu().numpy() for t in ctx.candidates(data, off, p)]
    m = want[0].shape[0]
    statuses = set()
    try:
        for nth in range(1, 14):
            with mj.Context(0) as ctx:
                ctx.join(data, off, p)
                out = [torch.full((m,), -1, dtype=torch.int32, device="cuda") for _ in range(2)]
                args = (ctypes.c_void_p(ctx._h.value), out[0].data_ptr(), out[1].data_ptr(), None)
                for _ in range(2):
                    lib.mj_inject_alloc_failure(nth)
                    st = lib.mj_candidates_copy(*args)
                    lib.mj_inject_alloc_failure(0)
                    statuses.add(st)
                    assert st in (0, -3)
                    if st == 0:
                        break
                assert lib.mj_candidates_copy(*args) == 0
                torch.cuda.synchronize()
                assert all(np.array_equal(a.cpu().numpy(), b) for a, b in zip(out, want)), nth
    finally:
        lib.mj_inject_alloc_failure(0)
    assert 0 in statuses


def test_no_candidates_after_a_join_with_some():
    """Empty strings have no records and no candidates, whatever was joined before."""
    import paper_1810_08833_gb300 as mj
    import torch
    lib = mj.library()
    s = _sets()["bounded"]
    data, off = to_device(s)
    empty = torch.zeros(3, dtype=torch.int64, device="cuda")
    with mj.Context(0) as ctx:
        ctx.join(data, off, mj.params(s.K, T=s.T))
        assert ctx.join(data[:0], empty, mj.params(s.K, T=s.T))[0].shape[0] == 0
        assert ctx.stats()["n_candidates"] == 0
        out = torch.full((64,), -1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        assert lib.mj_candidates_copy(ctypes.c_void_p(ctx._h.value), out.data_ptr(), out.data_ptr(), None) == 0
        torch.cuda.synchronize()
        assert (out == -1).all()
