"""The measured workloads of the MinJoin library: what a user calls, over the
range of sizes the library is used at.

Inputs are families of near-duplicate strings, drawn on the GPU from the seed,
with the shapes of the benchmark's synthetic workloads (see synth/): reads and
long noisy reads over ACGT, protein-like strings, text-like strings of Zipf
distributed words, and random bytes.  Every family is one random root and ten
mutated copies; the copies come in random order.

Kinds of calls:
    join        Context.join: the whole path on device buffers
    join_host   Context.join_host: the same from and to pinned host buffers
    learned     Context.join in learned mode with a trained network
    candidates  Context.candidates: partitions, filters, dedup
    partition   Context.partition: anchors and partition records
    verify      Context.verify: banded distances of given pairs
    network     Context.band_forward and band_grad: the band network alone
"""
import math

import numpy as np
import torch

import paper_1810_08833_gb300 as mj

COPIES = 10   # mutated copies per family
DEV = "cuda"

# alphabet, length distribution, edit rate of a copy (low, high), K and T of
# the workload, families of its full size
SHAPES = {
    "tiny":    dict(symbols="dna", lengths=("fixed", 500, 0), rate=(0.01, 0.01), K=10, T=10, roots=100),
    "reads":   dict(symbols="dna", lengths=("normal", 5000, 500), rate=(0.01, 0.04), K=100, T=100, roots=5000),
    "long":    dict(symbols="dna", lengths=("loguniform", 2000, 20000), rate=(0.05, 0.15), K=1000, T=200, roots=2000),
    "protein": dict(symbols="protein", lengths=("lognormal", 400, 0.462), rate=(0.02, 0.10), K=40, T=40, roots=40000),
    "text":    dict(symbols="text", lengths=("normal", 1500, 200), rate=(0.01, 0.08), K=75, T=75, roots=30000),
    "bytes":   dict(symbols="bytes", lengths=("lognormal", 700, 0.5), rate=(0.01, 0.08), K=60, T=60, roots=4000),
}


def listed():
    return [
        # a handful of short reads: the whole join is latency and launches
        dict(name="join_tiny", kind="join", shape="tiny", roots=100, K=10, T=10, repeats=1),
        # 50,000 reads at full size: many families, few false candidates
        dict(name="join_reads", kind="join", shape="reads", roots=5000, K=100, T=100, repeats=1),
        # long noisy reads: bands of a thousand rows
        dict(name="join_long", kind="join", shape="long", roots=2000, K=1000, T=200, repeats=1),
        # 400,000 protein-like strings: 200 M candidates of short strings
        dict(name="join_protein", kind="join", shape="protein", roots=40000, K=40, T=40, repeats=1),
        # 300,000 text-like strings, the benchmark's default workload
        dict(name="join_text", kind="join", shape="text", roots=30000, K=75, T=75, repeats=1),
        # a service's request: text from host buffers, partitioned twice for recall
        dict(name="host_text", kind="join_host", shape="text", roots=200, K=75, T=75, repeats=2),
        # learned first-pass bands on protein-like strings
        dict(name="learned_protein", kind="learned", shape="protein", roots=4000, K=40, T=40, repeats=1),
        # candidates only, for a caller with its own verifier
        dict(name="candidates_text", kind="candidates", shape="text", roots=3000, K=75, T=75, repeats=1),
        # partitions only, as a sharded join makes them before the exchange
        dict(name="partition_protein", kind="partition", shape="protein", roots=10000, K=40, T=40, repeats=1),
        # distances of given pairs, every pair with its own band
        dict(name="verify_bands", kind="verify", shape="bytes", roots=1000, K=60, pairs=100_000, bands=True),
        # distances at bands wider than a warp holds
        dict(name="verify_wide", kind="verify", shape="long", roots=12, K=4000, pairs=3_000, bands=False),
        # the band network: prediction and one gradient of a batch
        dict(name="network", kind="network", rows=65_536),
    ]


def draw(rng):
    """One more case: a kind, a shape, a size between a few families and the
    shape's full size (log-uniform), and K, T and repetitions as they vary."""
    kind = rng.choice(["join"] * 6 + ["join_host", "learned", "candidates", "partition", "verify", "verify", "network"])
    if kind == "network":
        return dict(kind=kind, rows=int(math.exp(rng.uniform(math.log(1024), math.log(1 << 19)))))
    shape = rng.choice(["tiny", "reads", "long", "protein", "text", "bytes"])
    s = SHAPES[shape]
    full = {"join": 0.5, "join_host": 0.1, "learned": 0.1, "candidates": 0.2, "partition": 0.5, "verify": 0.1}[kind]
    top = max(24.0, full * s["roots"])
    roots = int(math.exp(rng.uniform(math.log(12), math.log(top))))
    K = max(2, int(s["K"] * rng.uniform(0.5, 1.1)))
    if kind == "verify":
        if shape == "long" and rng.random() < 0.5:
            K *= 2   # wider than one warp's band
        pairs = int(math.exp(rng.uniform(math.log(200), math.log(4_000 if shape == "long" else 400_000))))
        return dict(kind=kind, shape=shape, roots=roots, K=K, pairs=pairs, bands=rng.random() < 0.5)
    T = K // 5 if shape == "long" else max(2, int(K * rng.choice([0.5, 0.75, 1.0])))
    repeats = 2 if kind != "learned" and rng.random() < 0.2 else 1
    return dict(kind=kind, shape=shape, roots=roots, K=K, T=T, repeats=repeats)


# ---------------------------------------------------------------- inputs

def _lengths(g, shape, n):
    how, a, b = SHAPES[shape]["lengths"]
    if how == "fixed":
        return torch.full((n,), a, dtype=torch.int64, device=DEV)
    if how == "normal":
        x = torch.randn(n, generator=g, device=DEV, dtype=torch.float64) * b + a
        return x.round().clamp(0.2 * a, 3 * a).long()
    if how == "loguniform":
        u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
        return torch.exp(math.log(a) + u * math.log(b / a)).round().long()
    x = torch.randn(n, generator=g, device=DEV, dtype=torch.float64) * b + math.log(a)
    return torch.exp(x).round().clamp(50, 5000).long()


def _symbols(shape):
    """(byte values, cumulative probabilities or None) of inserted and substituted symbols."""
    which = SHAPES[shape]["symbols"]
    if which == "dna":
        return torch.tensor(list(b"ACGT"), dtype=torch.uint8, device=DEV), None
    if which == "bytes":
        return torch.arange(256, device=DEV).to(torch.uint8), None
    if which == "text":
        return torch.arange(0x20, 0x7F, device=DEV).to(torch.uint8), None
    freq = np.random.Generator(np.random.PCG64(4)).dirichlet(np.full(20, 2.0))   # a proteome's, the same for all inputs
    return (torch.tensor(list(b"ACDEFGHIKLMNPQRSTVWY"), dtype=torch.uint8, device=DEV),
            torch.tensor(np.cumsum(freq), device=DEV, dtype=torch.float32))


def _draw_symbols(g, symbols, cdf, n):
    if cdf is None:
        return symbols[torch.randint(symbols.numel(), (n,), generator=g, device=DEV, dtype=torch.int32)]
    u = torch.rand(n, generator=g, device=DEV)
    return symbols[torch.searchsorted(cdf, u).clamp_(max=symbols.numel() - 1)]


def _word_stream(g, total):
    """A stream of at least `total` symbols of space-joined words, their ranks
    Zipf(1.1) over 50,000 random lowercase words of 2 to 12 letters (a
    language's vocabulary, the same for all inputs), and the words' start
    positions."""
    vocab = 50_000
    rng = np.random.Generator(np.random.PCG64(5))
    h_len = rng.integers(2, 13, size=vocab)
    letters = torch.from_numpy((97 + rng.integers(0, 26, size=int(h_len.sum()))).astype(np.uint8)).to(DEV)
    wlen = torch.from_numpy(h_len).to(DEV)
    wstart = torch.cumsum(wlen, 0) - wlen
    p = torch.arange(1, vocab + 1, device=DEV, dtype=torch.float64) ** -1.1
    cdf = torch.cumsum(p / p.sum(), 0).float()
    m = int(total / 3.0) + 1024   # a word and its space take at least three symbols
    ranks = torch.searchsorted(cdf, torch.rand(m, generator=g, device=DEV)).clamp_(max=vocab - 1)
    ends = torch.cumsum(wlen[ranks] + 1, 0)
    m = int(torch.searchsorted(ends, torch.tensor(total + 16, device=DEV))) + 1
    ranks, ends = ranks[:m], ends[:m]
    starts = ends - wlen[ranks] - 1
    word = torch.repeat_interleave(torch.arange(m, device=DEV), wlen[ranks] + 1)
    inword = torch.arange(word.numel(), device=DEV) - starts[word]
    r = ranks[word]
    stream = torch.where(inword < wlen[r], letters[(wstart[r] + inword).clamp_(max=letters.numel() - 1)],
                         torch.tensor(32, dtype=torch.uint8, device=DEV))
    return stream, starts


def _roots(g, shape, n, symbols, cdf):
    """Concatenated roots and their offsets."""
    lens = _lengths(g, shape, n)
    off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(lens, 0, out=off[1:])
    if SHAPES[shape]["symbols"] != "text":
        return _draw_symbols(g, symbols, cdf, int(off[-1])), off
    # every root starts at a word of the stream
    room = off[:-1] + 16 * torch.arange(n, device=DEV)
    stream, starts = _word_stream(g, int(off[-1]) + 16 * n)
    at = starts[torch.searchsorted(starts, room).clamp_(max=starts.numel() - 1)]
    where = torch.arange(int(off[-1]), device=DEV) + torch.repeat_interleave(at - off[:-1], lens)
    return stream[where.clamp_(max=stream.numel() - 1)], off


def _strings(shape, n_roots, seed, chunk=1 << 26):
    """(bytes, offsets, family of every string): COPIES mutated copies of every
    root, in random order.  A position is edited with its copy's rate; an edit
    inserts a symbol before it, deletes it or replaces it."""
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * seed + 17 * n_roots + len(shape))
    symbols, cdf = _symbols(shape)
    root, roff = _roots(g, shape, n_roots, symbols, cdf)
    n = n_roots * COPIES
    family = torch.randperm(n, generator=g, device=DEV) // COPIES
    lo, hi = SHAPES[shape]["rate"]
    rate = lo + (hi - lo) * torch.rand(n, generator=g, device=DEV)
    src_len = (roff[1:] - roff[:-1])[family]
    src_off = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(src_len, 0, out=src_off[1:])
    bounds = src_off.cpu().numpy()
    parts, lens, c0 = [], [], 0
    while c0 < n:
        c1 = max(c0 + 1, int(np.searchsorted(bounds, bounds[c0] + chunk, side="right")) - 1)
        L, total = src_len[c0:c1], int(bounds[c1] - bounds[c0])
        copy = torch.repeat_interleave(torch.arange(c0, c1, device=DEV), L, output_size=total)
        src = root[torch.arange(total, device=DEV) - (src_off[c0:c1] - bounds[c0] - roff[family[c0:c1]])[copy - c0]]
        u = torch.rand(total, generator=g, device=DEV) / rate[copy]   # below 1: edited, its third says how
        ins, dele, sub = u < 1 / 3, (u >= 1 / 3) & (u < 2 / 3), (u >= 2 / 3) & (u < 1)
        src = torch.where(sub, _draw_symbols(g, symbols, cdf, total), src)
        count = ins.to(torch.int32) + (~dele).to(torch.int32)
        end = torch.cumsum(count, 0)
        out = torch.empty(int(end[-1]) if total else 0, dtype=torch.uint8, device=DEV)
        keep = ~dele
        out[(end - 1)[keep]] = src[keep]                   # the kept symbol is the position's last
        out[(end - count)[ins]] = _draw_symbols(g, symbols, cdf, total)[ins]
        edges = torch.cat([torch.zeros(1, dtype=end.dtype, device=DEV), end])[(src_off[c0:c1 + 1] - bounds[c0])]
        lens.append(edges[1:] - edges[:-1])
        parts.append(out)
        c0 = c1
    offsets = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.cat(lens), 0, out=offsets[1:])
    data = torch.cat(parts)
    del parts, lens, root, rate, src_len, src_off
    torch.cuda.empty_cache()   # the library allocates its own device memory
    return data, offsets, family


def _pairs(family, m, seed):
    """m pairs: three in four of one family, the others of any two strings."""
    g = torch.Generator(device=DEV)
    g.manual_seed(7919 * seed + m)
    n = family.numel()
    by_family = torch.argsort(family, stable=True)
    i = torch.randint(n, (m,), generator=g, device=DEV)
    mate = by_family[family[i] * COPIES + torch.randint(COPIES, (m,), generator=g, device=DEV)]
    other = torch.randint(n, (m,), generator=g, device=DEV)
    j = torch.where(torch.rand(m, generator=g, device=DEV) < 0.75, mate, other)
    return i.int().contiguous(), j.int().contiguous()


def _params(case, **more):
    return mj.params(case["K"], T=case["T"], repeats=case["repeats"], **more)


def _trained(ctx, case, seed):
    """A band network trained on another, smaller instance of the workload."""
    data, off, _ = _strings(case["shape"], max(10, min(200, case["roots"] // 4)), seed + 5000)
    ctx.join(data, off, _params(case, flags=mj.MJ_FLAG_FEATURES))
    x, ed, _, _ = ctx.features()
    ctx.band_init(seed=5)
    if x.shape[0]:
        ctx.band_train(x, ed, K=case["K"], steps=100, batch=1024, lr=2e-3, tau=0.9, seed=13)
    torch.cuda.synchronize()


def _room(case):
    """Entries of the caller's output buffers: more than any input of the case gives."""
    n, family_pairs = case["roots"] * COPIES, case["roots"] * COPIES * (COPIES - 1) // 2
    if case["kind"] == "partition":
        return int(n * case["repeats"] * (1.35 * case["T"] + 20))
    if case["kind"] == "candidates":
        return family_pairs + n * n // 40 + 4096
    return 2 * family_pairs + 4096


def _kept(st, out):
    """The call's results in the caller's own buffers, which are larger (-1 behind the results)."""
    for buf, x in zip(st["out"], out):
        m = min(x.shape[0], buf.shape[0])
        buf[:m] = x[:m]
    return st["out"]


def prepare(case, seed):
    kind = case["kind"]
    ctx = mj.Context(0)
    st = {"ctx": ctx, "kind": kind}
    if kind in ("join", "learned", "candidates", "partition"):
        types = {"candidates": [torch.int32] * 2, "partition": [torch.int32] * 3 + [torch.int64]}
        st["out"] = [torch.full((_room(case),), -1, dtype=t, device=DEV) for t in types.get(kind, [torch.int32] * 3)]
    elif kind == "join_host":
        st["out"] = [torch.full((_room(case),), -1, dtype=torch.int32).pin_memory() for _ in range(3)]
    if kind == "network":
        x, y, w = _network(case, seed)
        ctx.band_init(seed=5)
        ctx.band_set_weights(w)
        st.update(x=torch.from_numpy(x).to(DEV), y=torch.from_numpy(y).to(DEV))
        return st
    if kind == "learned":
        _trained(ctx, case, seed)
    data, off, family = _strings(case["shape"], case["roots"], seed)
    if kind == "verify":
        i, j = _pairs(family, case["pairs"], seed)
        k = None
        if case["bands"]:   # a band per pair, from an earlier estimate of its distance
            g = torch.Generator(device=DEV)
            g.manual_seed(31 * seed + 1)
            k = torch.randint(case["K"] // 4, case["K"] + 1, (case["pairs"],), generator=g, device=DEV).int()
        st.update(data=data, off=off, i=i, j=j, k=k, K=case["K"])
        return st
    if kind == "join_host":
        st.update(h_data=data.cpu().pin_memory(), h_off=off.cpu().pin_memory(), p=_params(case))
        return st
    if kind == "learned":
        st["p"] = _params(case, verify_mode=mj.MJ_VERIFY_LEARNED)
    else:
        st["p"] = _params(case)
    st.update(data=data, off=off)
    return st


def run(st):
    kind, ctx = st["kind"], st["ctx"]
    if kind in ("join", "learned"):
        return _kept(st, ctx.join(st["data"], st["off"], st["p"]))
    if kind == "join_host":   # the results land in the caller's pinned buffers
        ctx.join_host(st["h_data"].numpy(), st["h_off"].numpy(), st["p"], out=tuple(b.numpy() for b in st["out"]))
        return st["out"]
    if kind == "candidates":
        return _kept(st, ctx.candidates(st["data"], st["off"], st["p"]))
    if kind == "partition":
        return _kept(st, ctx.partition(st["data"], st["off"], st["p"]))
    if kind == "verify":
        return ctx.verify(st["data"], st["off"], st["i"], st["j"], st["K"], k=st["k"])
    return (ctx.band_forward(st["x"]),) + tuple(ctx.band_grad(st["x"], st["y"], tau=0.9))


# ---------------------------------------------------------------- what a pass cannot do without

def _mean_length(shape):
    how, a, b = SHAPES[shape]["lengths"]
    if how == "loguniform":
        return (b - a) / math.log(b / a)
    return a * math.exp(b * b / 2) if how == "lognormal" else a


def work(case):
    """Bytes: the input once and the output once (an output pair is 12 bytes; a
    quarter of a family's pairs come out of a join).  Operations: 16 per
    32-row band word and column for every pair of one family, over the first
    K + 1 columns, which any verifier by dynamic programming needs to reject a
    pair (for pairs given: for all of them)."""
    if case["kind"] == "network":
        m, mlp = case["rows"], 8 * 64 + 64 * 64 + 64
        return {"bytes": m * (8 * 4 + 4 + 4) + 3 * 4801 * 4, "flops": 2 * m * mlp * 4}
    L = _mean_length(case["shape"])
    n = case["roots"] * COPIES
    family_pairs = case["roots"] * COPIES * (COPIES - 1) // 2
    inputs = n * L + 8 * (n + 1)
    cols = min(L, case["K"] + 1) * ((case["K"] + 32) // 32) * 16
    if case["kind"] == "verify":
        return {"bytes": inputs + 12 * case["pairs"], "flops": case["pairs"] * cols}
    parts = n * min(case["T"], L / 2) * case["repeats"]
    if case["kind"] == "partition":
        return {"bytes": inputs + 20 * parts, "flops": 0}
    if case["kind"] == "candidates":
        return {"bytes": inputs + 8 * family_pairs, "flops": 0}
    return {"bytes": inputs + 12 * family_pairs / 4, "flops": family_pairs * cols}


# ---------------------------------------------------------------- the same in 64 bits

def _network(case, seed):
    """Feature rows as joins make them (bounded, correlated), distances as a
    share of K, and weights of a network trained for a while."""
    r = np.random.default_rng(seed)
    m = case["rows"]
    c = r.geometric(0.15, m).astype(np.float64)
    pa, pb = r.normal(75, 8, m).clip(1), r.normal(75, 8, m).clip(1)
    n = r.normal(1500, 200, m).clip(1)
    x = np.stack([np.log2(1 + n) / 16, r.random(m), c / 76, pa / 76, pb / 76, c / np.minimum(pa, pb),
                  np.log2(1 + c) / 8, np.full(m, 75 / 175)], axis=1)
    y = np.minimum(1.0 + 1 / 75, r.gamma(4.0, 0.25, m))
    w = np.concatenate([r.normal(0, math.sqrt(2 / 8), 512), r.normal(0, 0.05, 64),
                        r.normal(0, math.sqrt(2 / 64), 4096), r.normal(0, 0.05, 64),
                        r.normal(0, 1 / 8, 64), [0.5]])
    return x.astype(np.float32), y.astype(np.float32), w.astype(np.float32)


def exact(case, seed):
    """Only the network computes with floating-point numbers."""
    if case["kind"] != "network":
        return None
    x, y, w = (a.astype(np.float64) for a in _network(case, seed))
    w1, b1, w2, b2, w3, b3 = np.split(w, np.cumsum([512, 64, 4096, 64, 64]))
    w1, w2, tau = w1.reshape(64, 8), w2.reshape(64, 64), float(np.float32(0.9))
    z1 = x @ w1.T + b1
    h1 = np.maximum(z1, 0)
    z2 = h1 @ w2.T + b2
    h2 = np.maximum(z2, 0)
    out = h2 @ w3 + b3
    r = y - out
    loss = float(np.where(r > 0, tau * r, (tau - 1) * r).mean())
    dy = np.where(r > 0, -tau, 1 - tau) / y.size
    d2 = np.where(h2 > 0, dy[:, None] * w3, 0)
    d1 = np.where(h1 > 0, d2 @ w2, 0)
    grad = np.concatenate([(d1.T @ x).ravel(), d1.sum(0), (d2.T @ h1).ravel(), d2.sum(0), h2.T @ dy, [dy.sum()]])
    return out, grad, loss
