"""GPU: contexts on different host threads, whose launches interleave.

A kernel's limit of dynamic shared memory is shared by all of them, so a thread
with small jobs must not lower it for a thread with large ones."""
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _jobs(mr):
    """(kind, device input, job parameters): shapes whose kernels need little and
    much shared memory."""
    for n, d, k, iters in [(2_000, 64, 256, 6), (1_500, 3, 2, 6), (1_200, 96, 300, 4), (900, 300, 40, 4),
                           (1_300, 16, 1_200, 4)]:
        x, _, _ = synth.kmeans_points(n, d, 8, seed=n)
        yield mr.KMEANS_F32, _dev(x), dict(km_dims=d, km_k=k, km_iters=iters, km_init=_dev(synth.kmeans_init(x, k, seed=n)))
    for n, nbins in [(1 << 22, 1 << 20), (1 << 22, 1 << 22), (50_000, 40_000), (50_000, 100)]:
        keys = synth.keys_u32(n, nbins, seed=nbins)
        yield mr.HIST_U32, _dev(keys.view(np.int32)), dict(hist_bins=nbins)
    for m in (1 << 28, 1 << 20):
        yield mr.BLOOM_DNA, _dev(synth.dna(2_400_031, seed=3)), dict(bloom_kmer=20, bloom_bits=m, bloom_hashes=7)


def test_contexts_on_threads_of_other_shapes(mr):
    import torch
    jobs = list(_jobs(mr))
    torch.cuda.synchronize()

    def run(ctx, job):
        kind, data, kw = job
        j = ctx.add_job(kind, data, **kw)
        ctx.run()
        out = ctx.fetch(j)
        ctx.release(j)
        return out

    with mr.Context(use_torch_allocator=False) as ctx:
        want = [run(ctx, job) for job in jobs]
    errors = []

    def work(t):
        try:
            with mr.Context(use_torch_allocator=False) as ctx:
                for r in range(80):
                    i = (r + 2 * t) % len(jobs)
                    if run(ctx, jobs[i]) != want[i]:
                        errors.append((t, r, "another result"))
        except Exception as e:
            errors.append((t, repr(e)))

    threads = [threading.Thread(target=work, args=(t,)) for t in range(5)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
