"""Two contexts on two host threads: joins of different inputs side by side give
what they give one after the other (nothing that a launch sets for its kernel
may depend on the call's own sizes)."""
import threading

import numpy as np
import pytest

import synth
from gpu_util import to_device

pytestmark = pytest.mark.gpu


def _one_length(seed, n, L, K):
    rng = np.random.Generator(np.random.PCG64(seed))
    roots = [synth.PROTEIN[rng.integers(0, 20, size=L)] for _ in range(n // 2)]
    strs = [r.tobytes() for r in roots]
    for r in roots:
        c = r.copy()
        c[rng.integers(0, L)] = synth.PROTEIN[0]
        strs.append(c.tobytes())
    return synth.from_strings(strs, K=K, T=K)


def _side_by_side(inputs, calls, what="join"):
    """Runs Context.join (or another method) on every (set, params) of `inputs`
    in a thread and context of its own, `calls` times, and returns (errors,
    outputs that differ from a lone run)."""
    import paper_1810_08833_gb300 as mj
    import torch
    errors, wrong = [], []
    jobs = []
    for s, p in inputs:
        data, off = to_device(s)
        with mj.Context(0) as ctx:
            jobs.append((data, off, p, [t.cpu().numpy() for t in getattr(ctx, what)(data, off, p)]))
    torch.cuda.synchronize()
    gate = threading.Barrier(len(jobs))

    def work(data, off, p, want):
        try:
            stream = torch.cuda.Stream()
            with mj.Context(0) as ctx:
                gate.wait()
                for t in range(calls):
                    with torch.cuda.stream(stream):
                        out = getattr(ctx, what)(data, off, p, stream=stream)
                        if t % 16 == 0:
                            got = [x.cpu().numpy() for x in out]
                            if not all(np.array_equal(a, b) for a, b in zip(got, want)):
                                wrong.append(p.K)
        except Exception as e:
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors, wrong


def test_joins_with_windows_of_different_widths():
    """The window of a string pair kernel is a bitmap in shared memory: 20,000
    strings of one length need 2.5 KB, 300 need 40 bytes."""
    import paper_1810_08833_gb300 as mj
    sets = [_one_length(1, 20_000, 40, 3), _one_length(2, 300, 40, 3), _one_length(3, 2_000, 60, 4)]
    errors, wrong = _side_by_side([(s, mj.params(s.K, T=s.T)) for s in sets], calls=400)
    assert not errors and not wrong, (errors, wrong)


def test_anchors_with_halos_of_different_radii():
    """The anchor kernel's span follows the radius: strings of 12,000 symbols in
    6 partitions (radius 856) and strings of 60 in 10 (radius 2)."""
    import paper_1810_08833_gb300 as mj
    long = synth.random_set(5, n=40, min_len=11_000, max_len=12_000, K=6, T=6, families=4, rate=0.0003)
    short = synth.random_set(6, n=300, min_len=50, max_len=60, K=10, T=10, families=12, rate=0.02)
    sets = [(s, mj.params(s.K, T=s.T)) for s in (long, short)]
    errors, wrong = _side_by_side(sets * 3, calls=1500, what="partition")
    assert not errors and not wrong, (errors, wrong)
