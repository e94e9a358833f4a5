"""Results and candidates into buffers that a kernel of word stores cannot take:
addresses that are no multiple of 4."""
import ctypes

import numpy as np
import pytest

import synth
from gpu_util import to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1, 2, 3])
@pytest.mark.parametrize("wanted", [(1, 1, 1), (0, 1, 0), (1, 0, 1)])
def test_unaligned_buffers(shift, wanted):
    import paper_1810_08833_gb300 as mj
    import torch
    lib = mj.library()
    s = synth.make_config(1, n_roots=20)
    data, off = to_device(s)
    with mj.Context(0) as ctx:
        want = [t.cpu().numpy() for t in ctx.join(data, off, mj.params(s.K, T=s.T))]
        cand = [t.cpu().numpy() for t in ctx.candidates(data, off, mj.params(s.K, T=s.T))]
        ctx.join(data, off, mj.params(s.K, T=s.T))
        for call, ref in ((lib.mj_result_copy, want), (lib.mj_candidates_copy, cand)):
            m = ref[0].shape[0]
            bufs = [torch.zeros(4 * m + 8, dtype=torch.uint8, device="cuda") for _ in ref]
            args = [b.data_ptr() + shift if w else None for b, w in zip(bufs, wanted)]
            torch.cuda.synchronize()
            assert call(ctypes.c_void_p(ctx._h.value), *args, None) == 0
            torch.cuda.synchronize()
            for b, w, r in zip(bufs, wanted, ref):
                raw = b.cpu().numpy()
                got = np.frombuffer(raw[shift:shift + 4 * m].tobytes(), dtype=np.int32)
                assert np.array_equal(got, r) if w else not raw.any()
                assert not raw[:shift].any() and not raw[shift + 4 * m:].any()
