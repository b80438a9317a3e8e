"""GPU parity: large-key histogram and Bloom-filter build against the oracle.

Both are integer/bit work, so every result must equal the oracle's bytes.
Cases cover the three containers of the histogram (shared-memory local
arrays of one CTA, local arrays spread over a thread-block cluster, the global
array), key ranges from 1 bin to 16M bins, out-of-range keys,
skewed keys, ragged lengths and unaligned device pointers; for the Bloom
filter, window lengths 1..32, filter sizes that are not powers of two, runs
of non-ACGT bytes and sequences shorter than one window; plus the full-size
workloads (256M keys over 16M bins; 30M windows into 300M bits)."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


def _dev(a, offset_bytes=0):
    """Device copy of a uint8/uint32 array starting offset_bytes into a buffer."""
    import torch
    raw = np.array(a, copy=True, order="C").view(np.uint8)  # a writable copy for torch
    buf = torch.zeros(raw.size + offset_bytes + 16, dtype=torch.uint8, device="cuda")
    if raw.size:
        buf[offset_bytes: offset_bytes + raw.size] = torch.from_numpy(raw).cuda()
    return buf[offset_bytes: offset_bytes + raw.size]


@pytest.mark.parametrize("nbins", [1, 100, 4096, 20000, 1 << 20, 1 << 24])
@pytest.mark.parametrize("container", ["auto", "smem", "global"])
def test_hist_u32_matches_oracle(mr, nbins, container):
    cmap = {"auto": mr.C_AUTO, "smem": mr.C_SMEM_ARRAY, "global": mr.C_GLOBAL_ARRAY}
    if container == "smem" and nbins > 40000:
        pytest.skip("local arrays of this many bins do not fit one CTA")
    n = 3_000_001  # ragged: not a multiple of any tile
    keys = synth.keys_u32(n, nbins + nbins // 8 + 1, seed=nbins)  # about 1 key in 9 out of range
    got = mr.hist_u32(_dev(keys), nbins, container=cmap[container])
    assert np.array_equal(got, oracle.hist_u32(keys, nbins))


def _cluster_max_bins():
    import torch
    return 8 * (torch.cuda.get_device_properties(0).shared_memory_per_block_optin // 4) - 1


@pytest.mark.parametrize("nbins", [1, 7, 8, 40, 70_000, 300_000, "max"])
def test_hist_u32_cluster_container(mr, nbins):
    """Local arrays spread over a thread-block cluster's distributed shared
    memory (a container the caller picks): slice boundaries, the out-of-range
    bin and the largest bin count the cluster holds, against the oracle and
    against the automatically chosen container."""
    if nbins == "max":
        nbins = _cluster_max_bins()
    n = 2_000_003
    keys = synth.keys_u32(n, nbins + nbins // 8 + 1, seed=nbins + 5)
    got = mr.hist_u32(_dev(keys), nbins, container=mr.C_CLUSTER_ARRAY)
    assert np.array_equal(got, oracle.hist_u32(keys, nbins))
    if nbins > 60_000:
        assert np.array_equal(mr.hist_u32(_dev(keys), nbins), got)  # C_AUTO


def test_hist_u32_cluster_container_skewed_unaligned_and_bad_args(mr):
    sk = synth.keys_u32(3_000_001, 200_000, skewed=True, seed=8)
    got = mr.hist_u32(_dev(sk, 4), 200_000, container=mr.C_CLUSTER_ARRAY)
    assert np.array_equal(got, oracle.hist_u32(sk, 200_000))
    c = mr.Context()
    keys = synth.keys_u32(1000, 100, seed=2)
    with pytest.raises(mr.MRError):
        c.add_job(mr.HIST_U32, keys, hist_bins=_cluster_max_bins() + 1, container=mr.C_CLUSTER_ARRAY)
    with pytest.raises(mr.MRError):
        c.add_job(mr.HIST_RGB8, np.zeros(30, dtype=np.uint8), container=mr.C_CLUSTER_ARRAY)
    with pytest.raises(mr.MRError):
        c.add_job(mr.WORDCOUNT, b"a b", container=mr.C_CLUSTER_ARRAY)
    c.close()


@pytest.mark.parametrize("offset", [4, 8, 12])
def test_hist_u32_unaligned_and_tiny(mr, offset):
    for n in (0, 1, 3, 5, 33, 1000):
        keys = synth.keys_u32(n, 50, seed=n + offset)
        for c in (mr.C_SMEM_ARRAY, mr.C_GLOBAL_ARRAY):
            got = mr.hist_u32(_dev(keys, offset), 40, container=c)
            assert np.array_equal(got, oracle.hist_u32(keys, 40)), (n, offset, c)


def test_hist_u32_skewed_and_constant(mr):
    sk = synth.keys_u32(5_000_000, 1 << 24, skewed=True, seed=3)
    for c in (mr.C_GLOBAL_ARRAY, mr.C_AUTO):
        assert np.array_equal(mr.hist_u32(_dev(sk), 1 << 24, container=c), oracle.hist_u32(sk, 1 << 24))
    const = np.full(2_000_003, 77, dtype=np.uint32)
    for c in (mr.C_SMEM_ARRAY, mr.C_GLOBAL_ARRAY):
        got = mr.hist_u32(_dev(const), 1000, container=c)
        assert got[77] == const.size and int(got.sum()) == const.size


def test_hist_u32_host_input_and_bad_args(mr):
    keys = synth.keys_u32(100_000, 5000, seed=1)
    assert np.array_equal(mr.hist_u32(keys, 5000), oracle.hist_u32(keys, 5000))
    c = mr.Context()
    with pytest.raises(mr.MRError):
        c.add_job(mr.HIST_U32, keys, hist_bins=0)
    with pytest.raises(mr.MRError):
        c.add_job(mr.HIST_U32, keys.view(np.uint8)[:7], hist_bins=10)  # not whole keys
    with pytest.raises(mr.MRError):
        c.add_job(mr.HIST_U32, keys, hist_bins=1 << 24, container=mr.C_SMEM_ARRAY)
    c.close()


def test_hist_u32_full_size(mr):
    """The paper's Histogram: 256M keys over 16M bins (global array in L2)."""
    keys = synth.keys_u32(256 << 20, 1 << 24)
    got = mr.hist_u32(_dev(keys), 1 << 24)
    assert int(got.sum()) == keys.size
    assert np.array_equal(got, oracle.hist_u32(keys, 1 << 24))


@pytest.mark.parametrize("L", [1, 5, 16, 31, 32])
@pytest.mark.parametrize("m,h", [(2, 1), (97, 3), (1_000_003, 7), (1 << 22, 32)])
def test_bloom_matches_oracle(mr, L, m, h):
    seq = synth.dna(200_000 + L, seed=L, n_runs=20, max_run=300)
    got = mr.bloom_dna(_dev(seq), L, m, h)
    assert np.array_equal(got, oracle.bloom_dna(seq, L, m, h))


@pytest.mark.parametrize("offset", [1, 3, 7])
def test_bloom_edges(mr, offset):
    cases = [b"", b"ACG", b"ACGT", b"ACGTNACGTN", b"acgtACGTACGTACGT", b"A" * 100, b"ACGT\n" * 50,
             bytes(synth.dna(8192 * 3 + 17, seed=offset))]
    for raw in cases:
        seq = np.frombuffer(raw, dtype=np.uint8)
        for L in (4, 32):
            got = mr.bloom_dna(_dev(seq, offset), L, 10_007, 5)
            assert np.array_equal(got, oracle.bloom_dna(raw, L, 10_007, 5)), (raw[:20], L)


def test_bloom_full_size(mr):
    """The paper's Bloom Filter build: 30M k-mers into 300M bits, 7 hashes."""
    L = 32
    seq = synth.dna(30_000_000 + L - 1)
    got = mr.bloom_dna(_dev(seq), L, 300_000_000, 7)
    assert np.array_equal(got, oracle.bloom_dna(seq, L, 300_000_000, 7))


def _part_keys(kind, n, nbins, seed):
    rng = np.random.default_rng(seed)
    if kind == "skewed":
        return synth.keys_u32(n, nbins, seed=seed, skewed=True)
    if kind == "one":
        return np.full(n, nbins // 3, dtype=np.uint32)
    keys = rng.integers(0, nbins + nbins // 8 + 2, n, dtype=np.uint32)  # about one key in nine out of range
    if kind == "sorted":
        keys.sort()
    if kind == "outside":
        keys[rng.random(n) < 0.7] = 0xFFFFFFFF
    return keys


@pytest.mark.parametrize("n,nbins", [
    (1 << 24, 58_112),            # two ranges of bins
    ((1 << 24) + 4_099, 65_535),  # the last bin and the out-of-range bin share a range
    ((1 << 24) + 5, 65_536),      # the out-of-range bin has a range of its own
    (1 << 22, 1 << 20),           # the fewest keys; 33 ranges, buckets smaller than a range
    (20_000_003, 5_000_000),
])
@pytest.mark.parametrize("kind", ["uniform", "skewed", "one", "sorted", "outside"])
@pytest.mark.parametrize("offset", [0, 12])
def test_hist_u32_partitioned(mr, n, nbins, kind, offset):
    """Jobs large enough for partitioned counting: the oracle's counts, and the
    same bytes as the global array's atomics (which a pinned container keeps)."""
    keys = _part_keys(kind, n, nbins, seed=n % 1000 + nbins)
    dev = _dev(keys, offset)
    got = mr.hist_u32(dev, nbins)
    assert np.array_equal(got, oracle.hist_u32(keys, nbins))
    assert np.array_equal(got, mr.hist_u32(dev, nbins, container=mr.C_GLOBAL_ARRAY))


def test_hist_u32_partitioned_rounds_and_budget(mr):
    """More keys than one round groups (the second round's counts add to the
    first's), and a context with an HBM budget, which keeps the global array."""
    import torch
    n, nbins = (1 << 28) + 70_001, 1_000_000
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    keys = torch.randint(0, nbins + 10, (n,), device="cuda", generator=g, dtype=torch.int32)
    torch.cuda.synchronize()
    want = torch.bincount(keys.clamp(max=nbins), minlength=nbins + 1).cpu().numpy().astype(np.uint64)
    assert np.array_equal(mr.hist_u32(keys, nbins), want)
    ctx = mr.Context(hbm_budget=64 << 20)
    j = ctx.add_job(mr.HIST_U32, keys, hist_bins=nbins)
    assert ctx.bytes_in_use < 16 << 20
    ctx.run()
    assert np.array_equal(np.frombuffer(ctx.fetch(j), dtype=np.uint64), want)
    ctx.close()


@pytest.mark.parametrize("n,L,m,h", [
    (2_396_776, 32, 20_000_003, 7),     # 2^24 positions and a few
    (16_777_217, 2, 97, 1),             # one range of four words, 8,192 windows a chunk
    (2_400_001, 15, (1 << 20) + 1, 7),  # a second range of one bit
    (530_001, 20, 1 << 22, 32),         # the most hashes
    (3_400_007, 31, 1 << 29, 5),        # the most ranges
])
@pytest.mark.parametrize("offset", [0, 1, 3])
def test_bloom_partitioned(mr, n, L, m, h, offset):
    """Filters with enough positions to be grouped by ranges of bits: the
    oracle's bytes (runs of N, a sequence that starts at any byte)."""
    seq = synth.dna(n, seed=n + L, n_runs=50, max_run=3000)
    assert np.array_equal(mr.bloom_dna(_dev(seq, offset), L, m, h), oracle.bloom_dna(seq, L, m, h))


def test_bloom_partitioned_rounds_and_budget(mr):
    """More positions than one round groups, against a context with an HBM
    budget, which sets every bit with an atomicOr on the global array."""
    n, L, m, h = 17_000_031, 21, 400_000_007, 32
    seq = _dev(synth.dna(n, seed=9, n_runs=300, max_run=1000))
    import torch
    torch.cuda.synchronize()
    ctx = mr.Context(hbm_budget=1 << 30)
    j = ctx.add_job(mr.BLOOM_DNA, seq, bloom_kmer=L, bloom_bits=m, bloom_hashes=h)
    ctx.run()
    want = np.frombuffer(ctx.fetch(j), dtype=np.uint8)
    ctx.close()
    assert np.array_equal(mr.bloom_dna(seq, L, m, h), want)


@pytest.mark.parametrize("L,h", [(32, 7), (32, 5), (17, 6), (21, 9), (20, 10), (25, 12), (11, 27), (32, 32)])
@pytest.mark.parametrize("offset", [0, 1, 3])
def test_bloom_partitioned_windows_and_scratch(mr, L, h, offset):
    """The grouped path, seen to be taken by its scratch: at most 4.4 bytes a
    position whatever the number of hashes (chunks of whole warps of windows),
    windows of all lengths up to 32 at any start, runs of N."""
    import torch
    m = 20_000_003
    n = ((1 << 24) + 300_000) // h + L
    seq = synth.dna(n, seed=h + L, n_runs=50, max_run=3000)
    dev = _dev(seq, offset)
    torch.cuda.synchronize()
    with mr.Context() as ctx:
        j = ctx.add_job(mr.BLOOM_DNA, dev, bloom_kmer=L, bloom_bits=m, bloom_hashes=h)
        scratch = ctx.bytes_in_use - (m + 7) // 8
        assert 3.9 <= scratch / ((n - L + 1) * h) <= 4.4
        ctx.run()
        assert np.array_equal(np.frombuffer(ctx.fetch(j), dtype=np.uint8), oracle.bloom_dna(seq, L, m, h))


@pytest.mark.parametrize("n,nbins", [(1 << 22, 1 << 20), ((1 << 24) + 4_099, 65_535)])
def test_hist_u32_partitioned_scratch(mr, n, nbins):
    """The grouped path is seen to be taken, by its 2 bytes a key and its tables."""
    keys = synth.keys_u32(n, nbins, seed=4)
    dev = _dev(keys, 4)
    with mr.Context() as ctx:
        j = ctx.add_job(mr.HIST_U32, dev, hist_bins=nbins)
        assert 2.0 <= (ctx.bytes_in_use - 8 * (nbins + 1)) / n <= 2.2
        ctx.run()
        assert np.array_equal(np.frombuffer(ctx.fetch(j), dtype=np.uint64), oracle.hist_u32(keys, nbins))


@pytest.mark.parametrize("n,nbins", [
    (1 << 26, 1 << 20),            # several units a range, cut at equal numbers of keys
    ((1 << 26) + 4_099, 1 << 24),  # one unit a range, its keys in four chunks
    (1 << 24, 60_000),             # two ranges, pieces in parts
    ((1 << 28) + 70_001, 300_000),  # the second round adds to the first
])
@pytest.mark.parametrize("kind", ["sorted", "sorted, the end not", "sequence", "reversed", "blocks", "constant",
                                  "half constant"])
def test_hist_u32_partitioned_keys_in_lumps(mr, n, nbins, kind):
    """Keys whose ranges fill whole chunks, or one range all of them; sorted ones
    repeat enough to take the global array, in one round or both."""
    import torch
    g = torch.Generator(device="cuda")
    g.manual_seed(n % 1000)
    if kind in ("sequence", "reversed"):
        keys = torch.arange(n, device="cuda", dtype=torch.int32).remainder_(nbins + 3)
        if kind == "reversed":
            keys = keys.flip(0).contiguous()
    elif kind == "blocks":  # 100,000 keys of one range at a time, in any order
        at = torch.randint(0, max(nbins - 1000, 1), (n // 100_000 + 1,), device="cuda", generator=g, dtype=torch.int32)
        keys = at.repeat_interleave(100_000)[:n] + torch.randint(0, 1000, (n,), device="cuda", generator=g, dtype=torch.int32)
    else:
        keys = torch.randint(0, nbins + 9, (n,), device="cuda", generator=g, dtype=torch.int32)
        if kind == "sorted":
            keys = keys.sort()[0]
        elif kind == "sorted, the end not":
            keys[: n - 70_000] = keys[: n - 70_000].sort()[0]
        else:
            keys[: n if kind == "constant" else n // 2] = nbins // 3
    torch.cuda.synchronize()
    want = torch.bincount(keys.clamp(max=nbins), minlength=nbins + 1).cpu().numpy().astype(np.uint64)
    assert np.array_equal(mr.hist_u32(keys, nbins), want)


@pytest.mark.parametrize("m,h", [(1_000_003, 7), (300_000_007, 5)])
@pytest.mark.parametrize("valid", [0, 40, 100_000, 1_000_000])
def test_bloom_partitioned_few_windows(mr, m, h, valid):
    """Sequences of which nearly all is N: ranges without a position, and ranges
    whose positions come from a few chunks."""
    seq = np.full(5_000_003, ord("N"), dtype=np.uint8)
    if valid:
        seq[3_000_001: 3_000_001 + valid] = synth.dna(valid, seed=valid)
    assert np.array_equal(mr.bloom_dna(_dev(seq, 1), 30, m, h), oracle.bloom_dna(seq, 30, m, h))
