"""Calls at the limits of what the library takes: other streams than the usual ones, arrays of
every origin, read sets and memory that leave the ordinary case. Every comparison is of whole
numbers, so exact."""
import mmap

import numpy as np
import pytest

import synth
from test_gpu_parity import assert_same, gpu, oracle_for, run_gpu, to_dev  # noqa: F401

pytestmark = pytest.mark.gpu

PER_THREAD_STREAM = 2  # cudaStreamPerThread


def counted(rs, stream=None, **kw):
    """A finalized handle of the read set."""
    import torch
    from paper_1705_11147_gb300 import KmerAnalysis, make_params
    p = dict(rs.meta["params"])
    p.pop("bloom_fpr", None)
    p.update(kw)
    reads = to_dev(torch, rs)
    torch.cuda.synchronize()
    ka = KmerAnalysis(make_params(**p, max_bases=rs.n_bases, max_reads=rs.n_reads, expected_distinct=rs.n_bases), stream=stream)
    ka.count(*reads)
    ka.finalize()
    return ka


def mapped(shape, dtype):
    """An array on pages that nothing has touched."""
    n = int(np.prod(shape)) * np.dtype(dtype).itemsize
    return np.frombuffer(mmap.mmap(-1, max(n, 1)), dtype, int(np.prod(shape))).reshape(shape)


def host_query(ka, keys, fresh):
    from paper_1705_11147_gb300 import capi
    n = len(keys)
    out = [(mapped if fresh else np.ones)(shape, dtype) for shape, dtype in (((n,), np.uint32), ((n, 8), np.uint32), ((n, 2), np.uint8))]
    assert capi.load().kmer_analysis_query(ka.handle, keys.ctypes.data, n, *(a.ctypes.data for a in out), 0) == 0
    return out


@pytest.mark.parametrize("stream", [None, PER_THREAD_STREAM])
def test_host_answers(gpu, stream):
    """Lookups from and to host arrays on fresh and on written pages, from one answer to 152 MB of
    them, other keys each time, against the same lookups on the device. cudaStreamPerThread names
    another stream in every thread: the copies have to stay with the thread that launched the lookups."""
    rs = synth.workload("plain_1m", scale=0.3)
    with counted(rs) as ref, counted(rs, stream=stream) as ka:
        have = ref.copy_result().keys
        rng = np.random.default_rng(5)
        for n in (1, 999, 30_000, 250_000, 850_000, 4_000_000):
            for fresh in (True, False, True):
                keys = have[rng.integers(0, len(have), n)]
                keys[rng.random(n) < 0.3, 0] ^= np.uint64(5)
                want = [x.cpu().numpy() for x in ref.query(gpu.from_numpy(keys.view(np.int64)).cuda())]
                for w, g in zip(want, host_query(ka, keys, fresh)):
                    np.testing.assert_array_equal(w.view(g.dtype), g, err_msg=f"{n} fresh={fresh}")


def spent(ka, reads, what):
    """Milliseconds in the counting kernels of one pass over the reads, the least of three."""
    best = float("inf")
    ka.set_profiling(True)
    for _ in range(3):
        ka.reset()
        ka.timings(reset=True)
        ka.count(*reads)
        ka.finalize()
        t = ka.timings(reset=True)
        best = min(best, sum(t[f"ms_{w}"] for w in what))
    return best


@pytest.mark.parametrize("k", [31, 63])
def test_reads_shorter_than_k(gpu, k):
    """Short reads add no windows: with so many of them that n_bases - (k - 1) * n_reads is about 0,
    the records are the long reads' own, and the sub-buckets are as many as for the long reads
    alone (with one or two of them every record would be counted several times as slowly)."""
    from paper_1705_11147_gb300 import KmerAnalysis, make_params
    rng = np.random.default_rng(8)
    genome = rng.integers(0, 4, 2_000_000).astype(np.uint8)
    n, length, short = 20_000, 1000, 12
    starts = rng.integers(0, len(genome) - length, n)
    long = np.frombuffer(b"ACGT", np.uint8)[genome[starts[:, None] + np.arange(length)]]
    m = n * (length - k + 1) // (k - 1 - short) // n * n
    each = m // n  # short reads behind every long one
    row = np.concatenate([long, np.full((n, each * short), ord("C"), np.uint8)], axis=1)
    lens = np.tile(np.array([length] + [short] * each), n)
    p = dict(k=k, min_depth=2, min_ext_count=2, qual_threshold=20, partitions=4, expected_distinct=5_000_000, expected_keys=2_500_000,
             max_bases=row.size, max_reads=len(lens))
    sets = [(row.reshape(-1), lens), (long.reshape(-1), np.full(n, length))]
    got, ms = [], []
    for seq, ln in sets:
        offs = np.concatenate([[0], np.cumsum(ln)]).astype(np.int64)
        reads = (gpu.from_numpy(seq.copy()).cuda(), gpu.full((seq.size,), 70, dtype=gpu.uint8, device="cuda"), gpu.from_numpy(offs).cuda())
        assert seq.size <= p["max_bases"]
        with KmerAnalysis(make_params(**p)) as ka:
            ms.append(spent(ka, reads, ("pass", "recount")))
            got.append(ka.copy_result().sorted())
    assert_same(*got)
    assert len(got[0]) > 1_000_000
    assert ms[0] < 2.5 * ms[1], ms


def hot_reads(n, unit, other, seed):
    """n reads of 150 bases, every third from a tandem array of one 171-base unit, the others random."""
    rng = np.random.default_rng(seed)
    array = np.tile(rng.integers(0, 4, unit).astype(np.uint8), 3)
    genome = rng.integers(0, 4, other).astype(np.uint8)
    hot = np.arange(n) % 3 == 0
    at = np.where(hot, rng.integers(0, unit, n), rng.integers(0, other - 150, n))[:, None] + np.arange(150)
    codes = np.where(hot[:, None], array[np.minimum(at, len(array) - 1)], genome[at])
    return readset_of(np.frombuffer(b"ACGT", np.uint8)[codes].reshape(-1), np.arange(n + 1) * 150)


def readset_of(seq, offsets, **params):
    return synth.ReadSet(seq.copy(), np.full(len(seq), 70, np.uint8), offsets.astype(np.uint64), {"params": params})


@pytest.mark.parametrize("n", [2_000, 9_000, 30_000, 120_000])
@pytest.mark.parametrize("k", [31, 63])
def test_hot_keys_of_small_samples(gpu, n, k):
    """Hot k-mers in few segments, in as many as there are warps, and in more, against the oracle."""
    rs = hot_reads(n, 171, 20_000, n)
    for depth, bloom in ((1, False), (2, True)):
        rs.meta["params"] = dict(k=k, min_depth=depth, min_ext_count=2, qual_threshold=20)
        assert_same(run_gpu(gpu, rs, use_bloom=bloom, partitions=3), oracle_for(rs), f"depth {depth}")


def test_hot_keys_use_all_warps(gpu):
    """A third of a small sample's windows from 171 k-mers: counted in less than three times the time of
    as many windows without them (a single warp for a bucket's few segments: five times)."""
    from paper_1705_11147_gb300 import KmerAnalysis, make_params
    ms = []
    for unit in (171, 60_000):
        rs = hot_reads(40_000, unit, 120_000, 3)
        with KmerAnalysis(make_params(k=31, min_depth=2, partitions=2, max_bases=rs.n_bases, max_reads=rs.n_reads,
                                      expected_distinct=500_000)) as ka:
            ms.append(spent(ka, to_dev(gpu, rs), ("pass",)))
    assert ms[0] < 3 * ms[1], ms


def test_finalize_after_graphs(gpu):
    """Every batch graph that has been in the process makes allocations from the library's pool on a
    busy stream slower: a pass of another handle takes as long as before them, but for one such
    allocation (with ten it took 35 us longer for each graph)."""
    import time
    from paper_1705_11147_gb300 import BatchGraph, KmerAnalysis, make_params
    rs = synth.workload("plain_1m", scale=0.3)
    reads = to_dev(gpu, rs)
    kw = dict(k=33, min_depth=2, max_bases=rs.n_bases, max_reads=rs.n_reads, expected_distinct=4_000_000, partitions=4)

    def passes():
        with KmerAnalysis(make_params(**kw)) as a, KmerAnalysis(make_params(**kw)) as b, KmerAnalysis(make_params(**kw)) as c:
            us = []
            for i in range(60):
                ka = (a, b, c)[i % 3]
                t = time.perf_counter()
                ka.reset()
                ka.count(*reads)
                ka.finalize()
                us.append((time.perf_counter() - t) * 1e6)
            return float(np.median(us[20:]))

    before = passes()
    small = [synth.workload("plain_1m", scale=0.05 * (1 + i % 4)) for i in range(12)]
    for _ in range(8):
        handles = [KmerAnalysis(make_params(k=31, min_depth=2, max_bases=s.n_bases, max_reads=s.n_reads, partitions=4,
                                            expected_distinct=s.n_bases // 4, expected_keys=s.n_bases // 10)) for s in small]
        graph = BatchGraph(handles, [to_dev(gpu, s) for s in small])
        graph.replay()
        assert all(int(r.n) > 0 for r in graph.results())
        del handles, graph
    after = passes()
    assert after - before < 120, (before, after)
