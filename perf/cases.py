"""Performance cases: the work a user of the library has it do, through its public entry points.

Every family of jobs the library runs is here at the sizes it meets in use: the small call whose
latency counts, the ordinary one and the largest; odd sizes next to round ones; both k-means
precisions and shapes beyond the tensor-core path's; histograms whose bins fit a thread block and
histograms whose bins do not; one launch for one job and one launch for many.

A large result stays on the device (``Context.result_device``), where the next step of a GPU program
takes it; it is released when the next pass over the same state begins, as a loop over batches of
input does.  A small result comes back through the one-shot helpers, as a script calls them.

Inputs are made on the GPU with the distributions of the ``synth`` package: Zipf-distributed words,
photographs as clusters of colours over uniform noise, noisy lines, Gaussian mixtures, uniform or
skewed keys, uniform bases with runs of N.
"""
import collections
import math

import numpy as np
import torch

import paper_1309_0215_gb300 as mr

MIB = 1 << 20
DEV = "cuda"

# the job mix of a batch: kind, share (half word counts, three tenths histograms, a fifth regressions)
BATCH_MIX = (("wordcount", 0.5), ("hist", 0.3), ("linreg", 0.2))
BATCH_MIN, BATCH_MAX = 4096, 64 * MIB


def listed():
    return [
        # a short document, counted by a script: latency and launches
        {"name": "wordcount 48 KB", "kind": "wordcount", "bytes": 48_611, "vocab": 2000, "maxlen": 12, "oneshot": True},
        # the word count of the paper's size class, 50,000 distinct words
        {"name": "wordcount 16 MiB", "kind": "wordcount", "bytes": 16 * MIB, "vocab": 50_000, "maxlen": 12,
         "oneshot": False},
        # a corpus shard
        {"name": "wordcount 256 MB", "kind": "wordcount", "bytes": 255_999_983, "vocab": 50_000, "maxlen": 12,
         "oneshot": False},
        # the colour histogram of one Full HD photograph, by a script
        {"name": "histogram 1080p", "kind": "hist", "pixels": 1920 * 1080, "oneshot": True},
        # the benchmark step: a 1.5 GiB histogram and a 512 MiB regression run together
        {"name": "histogram + regression 2 GiB", "kind": "arrays", "pixels": 536_870_912, "pairs": 268_435_456},
        # k-means at the benchmark's shape on the tensor cores, ten rounds
        {"name": "k-means 4M x 64 bf16", "kind": "kmeans", "n": 4_000_000, "d": 64, "k": 256, "iters": 10,
         "precision": "bf16", "oneshot": False},
        # the default precision at an odd size, by a script: a table of 37 features
        {"name": "k-means 200K x 37 fp32", "kind": "kmeans", "n": 200_003, "d": 37, "k": 100, "iters": 10,
         "precision": "fp32", "oneshot": True},
        # a codebook of 512 words over 128-dimensional descriptors: wider than the tensor-core path takes
        {"name": "k-means 250K x 128 fp32", "kind": "kmeans", "n": 250_000, "d": 128, "k": 512, "iters": 5,
         "precision": "fp32", "oneshot": False},
        # the paper's histogram: 16 million unique keys, 256 million elements
        {"name": "keys 256M, 16M bins", "kind": "keys", "n": 268_435_456, "bins": 1 << 24, "skewed": False},
        # category counts with a skewed distribution: bins that fit a thread block
        {"name": "keys 60M, 10K bins skewed", "kind": "keys", "n": 60_000_001, "bins": 10_000, "skewed": True},
        # the paper's Bloom filter: 30 million 32-mers into 300 million bits
        {"name": "bloom 30M", "kind": "bloom", "n": 30_000_031, "bits": 300_000_000, "kmer": 32, "hashes": 7,
         "runs": 100},
        # many jobs in one launch, replayed over buffers that a program refills
        {"name": "batch of 60 jobs", "kind": "batch", "jobs": 60, "spread": 11},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["wordcount", "wordcount", "hist", "arrays", "kmeans", "kmeans", "kmeans", "keys", "keys",
                       "bloom", "batch"])
    if kind == "wordcount":
        n = _log(rng, 4096, 255_000_000)
        return {"kind": kind, "bytes": n, "vocab": _words(n, _log(rng, 1000, 100_000)), "maxlen": rng.choice([12, 12, 24]),
                "oneshot": n < 200_000}
    if kind == "hist":
        n = _log(rng, 10_000, 400_000_000)
        return {"kind": kind, "pixels": n, "oneshot": n < 4_000_000}
    if kind == "arrays":
        return {"kind": kind, "pixels": _log(rng, 30_000, 500_000_000), "pairs": _log(rng, 30_000, 260_000_000)}
    if kind == "kmeans":
        shape = rng.choice(["bf16", "fp32", "wide"])
        if shape == "wide":
            d, k = rng.randint(65, 256), rng.randint(64, 1024)
            n = min(_log(rng, 20_000, 400_000), int(1.6e10 / (d * k)))
            return {"kind": kind, "n": n, "d": d, "k": k, "iters": 5, "precision": "fp32", "oneshot": False}
        d, k = rng.randint(2, 64), rng.randint(8, 256)
        n = _log(rng, 65_536, 2_000_000) if shape == "bf16" else _log(rng, 10_000, 1_000_000)
        return {"kind": kind, "n": n, "d": d, "k": k, "iters": 10, "precision": shape, "oneshot": n < 250_000}
    if kind == "keys":
        bins = _log(rng, 300, 1 << 24)
        return {"kind": kind, "n": _log(rng, 1_000_000, 260_000_000), "bins": bins, "skewed": rng.random() < 0.4}
    if kind == "bloom":
        n = _log(rng, 100_000, 30_000_000)
        return {"kind": kind, "n": n, "bits": n * rng.randint(8, 16) + rng.randint(0, 63), "kmer": rng.randint(15, 32),
                "hashes": rng.randint(3, 10), "runs": rng.randint(0, 200)}
    return {"kind": kind, "jobs": rng.randint(16, 60), "spread": rng.randint(0, 1 << 20)}


# ------------------------------------------------------------------ inputs

def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1_000_003 + salt)
    return g


def _text(nbytes, vocab, maxlen, g):
    """Words of 3..maxlen letters, Zipf-distributed (s = 1) with every word of the vocabulary present,
    single spaces, a newline about every 14 words; filled with newlines after the last whole word.
    A word's length depends on its rank alone, so that texts of one size have results of one size."""
    rank = torch.arange(vocab, device=DEV)
    lens = 3 + ((rank * 2_654_435_761) >> 7) % (maxlen - 2)
    letters = torch.randint(97, 123, (vocab, maxlen), device=DEV, generator=g)
    code = torch.randperm(26 ** 3, device=DEV, generator=g)
    for ln in range(3, maxlen + 1):  # the first three letters tell the words of one length apart
        own = torch.nonzero(lens == ln).view(-1)
        c = code[:len(own)]
        letters[own, 0], letters[own, 1], letters[own, 2] = 97 + c // 676, 97 + c // 26 % 26, 97 + c % 26
    letters = letters.to(torch.uint8)
    w = 1.0 / (rank + 1).double()
    cdf = torch.cumsum(w, 0) / w.sum()
    mean = float((lens.double() * w).sum() / w.sum()) + 1.0

    def zipf(m):
        u = torch.rand(m, device=DEV, generator=g, dtype=torch.float64)
        return torch.searchsorted(cdf, u).clamp_(max=vocab - 1)

    head = torch.cat([rank, zipf(vocab // 2)])
    head = head[torch.randperm(len(head), device=DEV, generator=g)]
    out = torch.full((nbytes,), 10, device=DEV, dtype=torch.uint8)
    at = 0
    while at < nbytes:
        m = min(int((nbytes - at) / mean * 1.02) + 64, 16_000_000)
        r = torch.cat([head, zipf(m)]) if at == 0 else zipf(m)
        drawn = len(r)
        end = torch.cumsum(lens[r] + 1, 0) + at
        keep = end <= nbytes
        r, end = r[keep], end[keep]
        if not len(r):
            break
        ln = lens[r]
        start = end - ln - 1
        nl = torch.rand(len(r), device=DEV, generator=g) < 1 / 14
        out[end - 1] = torch.where(nl, 10, 32).to(torch.uint8)
        for j in range(maxlen):
            has = ln > j
            out[start[has] + j] = letters[r[has], j]
        at = int(end[-1])
        if len(r) < drawn:
            break
    return out


def _pixels(n, g):
    """RGB bytes: 70% uniform, the rest in eight clusters of colours (sigma 12)."""
    out = torch.randint(0, 256, (n, 3), device=DEV, generator=g, dtype=torch.uint8)
    centres = torch.randint(0, 256, (8, 3), device=DEV, generator=g).float()
    for a in range(0, n, 32_000_000):
        b = min(n, a + 32_000_000)
        which = torch.randint(0, 8, (b - a,), device=DEV, generator=g)
        near = torch.randn(b - a, 3, device=DEV, generator=g).mul_(12).add_(centres[which]).round_().clamp_(0, 255)
        own = torch.rand(b - a, 1, device=DEV, generator=g) < 0.3
        out[a:b] = torch.where(own, near.to(torch.uint8), out[a:b])
    return out.view(-1)


def _pairs(n, g):
    """int8 pairs: x uniform on [-40, 40], y = 3 x plus noise of sigma 4."""
    out = torch.empty(n, 2, device=DEV, dtype=torch.int8)
    for a in range(0, n, 64_000_000):
        b = min(n, a + 64_000_000)
        x = torch.randint(-40, 41, (b - a,), device=DEV, generator=g).float()
        y = (3 * x + torch.randn(b - a, device=DEV, generator=g).mul_(4).round_()).clamp_(-128, 127)
        out[a:b, 0] = x.to(torch.int8)
        out[a:b, 1] = y.to(torch.int8)
    return out.view(-1)


def _points(n, d, k, g):
    """A mixture of 256 Gaussians (means uniform on [-10, 10], unit variance) and k of its points."""
    means = torch.rand(256, d, device=DEV, generator=g) * 20 - 10
    x = torch.randn(n, d, device=DEV, generator=g)
    for a in range(0, n, 1_000_000):
        b = min(n, a + 1_000_000)
        x[a:b] += means[torch.randint(0, 256, (b - a,), device=DEV, generator=g)]
    init = x[torch.randperm(n, device=DEV, generator=g)[:k]].clone()
    return x, init


def _keys(n, bins, skewed, g):
    """Keys below `bins`: uniform, or with rank density 1 / (rank + 1)."""
    out = torch.empty(n, device=DEV, dtype=torch.int32)
    for a in range(0, n, 64_000_000):
        b = min(n, a + 64_000_000)
        if skewed:
            u = torch.rand(b - a, device=DEV, generator=g, dtype=torch.float64)
            rank = (torch.exp(u * math.log(bins + 1.0)) - 1.0).long().clamp_(0, bins - 1)
            out[a:b] = ((rank * 7919 + 13) % bins).to(torch.int32)  # popular keys lie anywhere in the range
        else:
            out[a:b] = torch.randint(0, bins, (b - a,), device=DEV, generator=g, dtype=torch.int32)
    return out


def _bases(n, runs, g):
    out = torch.tensor(list(b"ACGT"), device=DEV, dtype=torch.uint8)[torch.randint(0, 4, (n,), device=DEV, generator=g)]
    at = torch.randint(0, n, (max(runs, 1),), device=DEV, generator=g).tolist()
    ln = torch.randint(1, 1000, (max(runs, 1),), device=DEV, generator=g).tolist()
    for i in range(runs):
        out[at[i]:at[i] + ln[i]] = ord("N")
    return out


def _words(nbytes, most):
    """Distinct words of a text of this size."""
    return max(64, min(most, nbytes // 24))


def _batch_specs(case):
    """(kind, bytes) of each job: sizes spread evenly over the logarithm of the range, then shuffled."""
    rng = np.random.default_rng(case["spread"])
    m = case["jobs"]
    kinds, acc = [], 0.0
    for name, share in BATCH_MIX:
        acc += share * m
        while len(kinds) < int(acc + 0.5):
            kinds.append(name)
    q = (rng.permutation(m) + rng.random(m)) / m
    sizes = np.exp(math.log(BATCH_MIN) + q * math.log(BATCH_MAX / BATCH_MIN)).astype(np.int64)
    rec = {"wordcount": 1, "hist": 3, "linreg": 2}
    return [(kd, int(s) - int(s) % rec[kd]) for kd, s in zip(kinds, sizes)]


def _batch_inputs(case, seed):
    """Inputs lie back to back in one buffer per kind, as a server keeps them: they start at any byte."""
    specs = _batch_specs(case)
    pools = {"wordcount": torch.cat([_text(n, _words(n, 50_000), 12, _gen(seed, 10 + i))
                                     for i, (kd, n) in enumerate(specs) if kd == "wordcount"]),
             "hist": _pixels(sum(n for kd, n in specs if kd == "hist") // 3, _gen(seed, 2)),
             "linreg": _pairs(sum(n for kd, n in specs if kd == "linreg") // 2, _gen(seed, 3))}
    out, at = [], dict.fromkeys(pools, 0)
    for kd, n in specs:
        out.append((kd, pools[kd][at[kd]:at[kd] + n]))
        at[kd] += n
    return out


def _inputs(case, seed):
    g, kind = _gen(seed), case["kind"]
    if kind == "wordcount":
        return (_text(case["bytes"], case["vocab"], case["maxlen"], g),)
    if kind == "hist":
        return (_pixels(case["pixels"], g),)
    if kind == "arrays":
        return _pixels(case["pixels"], g), _pairs(case["pairs"], _gen(seed, 1))
    if kind == "kmeans":
        return _points(case["n"], case["d"], case["k"], g)
    if kind == "keys":
        return (_keys(case["n"], case["bins"], case["skewed"], g),)
    if kind == "bloom":
        return (_bases(case["n"], case["runs"], g),)
    return _batch_inputs(case, seed)


# --------------------------------------------------------------- the passes

class _Memory:
    """Device memory of a context's job, as torch sees it; the context lives as long as the tensor."""

    def __init__(self, ctx, address, nbytes):
        self.ctx = ctx
        self.__cuda_array_interface__ = {"shape": (nbytes,), "typestr": "|u1", "data": (address, False), "version": 3}


def _result(ctx, job):
    address, nbytes = ctx.result_device(job)
    return torch.as_tensor(_Memory(ctx, address, nbytes), device=DEV)


_KINDS = {"wordcount": mr.WORDCOUNT, "hist": mr.HIST_RGB8, "linreg": mr.LINREG_I8}
_PRECISION = {"fp32": mr.KM_FP32, "bf16": mr.KM_BF16_TC}


def prepare(case, seed):
    s = {"case": case, "in": _inputs(case, seed), "jobs": []}
    if not case.get("oneshot"):
        s["ctx"] = mr.Context()
    if case["kind"] == "batch":
        ctx = s["ctx"]
        # a context made under torch's default stream runs on a stream of its own, and a job's input
        # may not change while it runs: what torch has queued has to be done first
        torch.cuda.synchronize()
        s["jobs"] = [ctx.add_job(_KINDS[kd], t) for kd, t in s["in"]]
        ctx.run(mr.RUN_BATCHED)
        s["out"] = [_as_typed(kd, _result(ctx, j)) for (kd, _), j in zip(s["in"], s["jobs"])]
        s["out"] = {kd: [o for (k2, _), o in zip(s["in"], s["out"]) if k2 == kd] for kd in _KINDS}
    return s


def _as_typed(kind, raw):
    return raw if kind == "wordcount" else raw.view(torch.int64)


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "batch":
        state["ctx"].rerun()
        return state["out"]
    if case.get("oneshot"):
        if kind == "wordcount":
            return np.frombuffer(mr.wordcount(state["in"][0]), dtype=np.uint8)
        if kind == "hist":
            return mr.hist_rgb8(state["in"][0])
        x, init = state["in"]
        cent, assign, _ = mr.kmeans(x, init, case["iters"], _PRECISION[case["precision"]])
        return {"centroids": cent, "assignments": assign}
    ctx = state["ctx"]
    for j in state["jobs"]:
        ctx.release(j)
    state["jobs"] = []
    if kind == "arrays":
        px, xy = state["in"]
        state["jobs"] = [ctx.add_job(mr.HIST_RGB8, px), ctx.add_job(mr.LINREG_I8, xy)]
        ctx.run(mr.RUN_CONCURRENT)
        return {"bins": _result(ctx, state["jobs"][0]).view(torch.int64),
                "sums": _result(ctx, state["jobs"][1]).view(torch.int64)}
    if kind == "kmeans":
        x, init = state["in"]
        k, d = init.shape
        n = x.shape[0]
        job = ctx.add_job(mr.KMEANS_F32, x, km_dims=d, km_k=k, km_iters=case["iters"], km_init=init,
                          km_precision=_PRECISION[case["precision"]])
    elif kind == "keys":
        job = ctx.add_job(mr.HIST_U32, state["in"][0], hist_bins=case["bins"])
    elif kind == "bloom":
        job = ctx.add_job(mr.BLOOM_DNA, state["in"][0], bloom_kmer=case["kmer"], bloom_bits=case["bits"],
                          bloom_hashes=case["hashes"])
    else:
        job = ctx.add_job(_KINDS[kind], state["in"][0])
    state["jobs"] = [job]
    ctx.run(mr.RUN_PLAIN)
    raw = _result(ctx, job)
    if kind == "kmeans":
        return {"centroids": raw[:4 * k * d].view(torch.float32).view(k, d),
                "assignments": raw[4 * k * d:4 * k * d + 4 * n].view(torch.int32)}
    if kind in ("keys", "hist"):
        return raw.view(torch.int64)
    return raw


# --------------------------------------------------------------- the floors

def work(case):
    kind = case["kind"]
    if kind == "wordcount":
        # 24 bytes a record and about 8 bytes of key for each word of the vocabulary
        return {"bytes": case["bytes"] + 32 * case["vocab"], "flops": 0}
    if kind == "hist":
        return {"bytes": 3 * case["pixels"] + 768 * 8, "flops": 0}
    if kind == "arrays":
        return {"bytes": 3 * case["pixels"] + 2 * case["pairs"] + 768 * 8 + 40, "flops": 0}
    if kind == "kmeans":
        n, d, k = case["n"], case["d"], case["k"]
        return {"bytes": 4 * n * d + 8 * k * d + 4 * n, "flops": 2.0 * n * d * k * case["iters"]}
    if kind == "keys":
        return {"bytes": 4 * case["n"] + 8 * (case["bins"] + 1), "flops": 0}
    if kind == "bloom":
        return {"bytes": case["n"] + (case["bits"] + 7) // 8, "flops": 0}
    return {"bytes": sum(n for _, n in _batch_specs(case)), "flops": 0}


# ------------------------------------------------- the same results, plainly

def _exact_wordcount(text):
    raw = text.cpu().numpy().tobytes()
    if len(raw) > 64 * MIB:
        return None
    got = collections.Counter(raw.split())
    order = sorted(got.items(), key=lambda kv: (-kv[1], kv[0]))
    keys = b"".join(k for k, _ in order)
    rec = np.empty((len(order), 3), dtype=np.uint64)
    rec[:, 0] = [c for _, c in order]
    rec[:, 2] = [len(k) for k, _ in order]
    rec[:, 1] = np.concatenate([[0], np.cumsum(rec[:, 2])[:-1]]) if len(order) else 0
    head = np.array([len(order), len(keys)], dtype=np.uint64)
    return np.frombuffer(head.tobytes() + rec.tobytes() + keys, dtype=np.uint8)


def _exact_hist(px):
    px = px.view(-1, 3)
    return torch.cat([torch.bincount(px[:, c].contiguous(), minlength=256) for c in range(3)])


def _exact_linreg(xy):
    total = torch.zeros(5, device=DEV, dtype=torch.int64)
    v = xy.view(-1, 2)
    for a in range(0, len(v), 64_000_000):
        x, y = v[a:a + 64_000_000, 0].long(), v[a:a + 64_000_000, 1].long()
        total += torch.stack([x.sum(), y.sum(), (x * x).sum(), (y * y).sum(), (x * y).sum()])
    return total


def _exact_kmeans(case, x, init):
    n, d, k = case["n"], case["d"], case["k"]
    if 3.0 * n * d * k * case["iters"] > 6e12:
        return None
    c = init.double()
    assign = torch.empty(n, device=DEV, dtype=torch.int64)
    step = max(1, (1 << 27) // (k * 8))
    for _ in range(case["iters"]):
        sums = torch.zeros(k, d, device=DEV, dtype=torch.float64)
        for a in range(0, n, step):
            xa = x[a:a + step].double()
            dist = torch.zeros(len(xa), k, device=DEV, dtype=torch.float64)
            for j in range(d):
                dist += (xa[:, j:j + 1] - c[:, j]).square_()
            own = dist.argmin(1)
            assign[a:a + step] = own
            sums.index_add_(0, own, xa)
        count = torch.bincount(assign, minlength=k).unsqueeze(1)
        # the centroids of a round are FP32 values
        c = torch.where(count > 0, sums / count.clamp(min=1), c).float().double()
    return {"centroids": c, "assignments": assign.int()}


def _shift_right(v, s):
    return (v >> s) & ((1 << (64 - s)) - 1)


def _wrap(v):
    return v - (1 << 64) if v >= 1 << 63 else v


def _mix(z):
    z = (z ^ _shift_right(z, 30)) * _wrap(0xBF58476D1CE4E5B9)
    z = (z ^ _shift_right(z, 27)) * _wrap(0x94D049BB133111EB)
    return z ^ _shift_right(z, 31)


def _mod(v, m):
    return (_shift_right(v, 1) % m * 2 + (v & 1)) % m  # v as an unsigned number


def _exact_bloom(case, seq):
    m, length = case["bits"], case["kmer"]
    code = torch.full((256,), -1, device=DEV, dtype=torch.int64)
    for i, b in enumerate(b"ACGT"):
        code[b] = i
    v = code[seq.int()]
    n = len(v) - length + 1
    win = torch.zeros(n, device=DEV, dtype=torch.int64)
    ok = torch.ones(n, device=DEV, dtype=torch.bool)
    for j in range(length):
        part = v[j:j + n]
        ok &= part >= 0
        win = win * 4 + part
    win = win[ok]
    pos, step = _mod(_mix(win), m), 1 + _mod(_mix(win ^ _wrap(0x9E3779B97F4A7C15)), m - 1)
    bits = torch.zeros((m + 7) // 8 * 8, device=DEV, dtype=torch.uint8)
    for _ in range(case["hashes"]):
        bits[pos] = 1
        pos = (pos + step) % m
    weight = (1 << torch.arange(8, device=DEV)).to(torch.uint8)
    return (bits.view(-1, 8) * weight).sum(1).to(torch.uint8)


def exact(case, seed):
    given, kind = _inputs(case, seed), case["kind"]
    if kind == "wordcount":
        return _exact_wordcount(given[0])
    if kind == "hist":
        return _exact_hist(given[0])
    if kind == "arrays":
        return {"bins": _exact_hist(given[0]), "sums": _exact_linreg(given[1])}
    if kind == "kmeans":
        return _exact_kmeans(case, *given)
    if kind == "keys":
        return torch.cat([sum(torch.bincount(p, minlength=case["bins"]) for p in given[0].split(64_000_000)),
                          torch.zeros(1, device=DEV, dtype=torch.int64)])
    if kind == "bloom":
        return _exact_bloom(case, given[0])
    plain = {"wordcount": _exact_wordcount, "hist": _exact_hist, "linreg": _exact_linreg}
    return {kd: [plain[kd](t) for k2, t in given if k2 == kd] for kd in _KINDS}
