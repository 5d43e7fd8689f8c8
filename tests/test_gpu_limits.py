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


def device_reads(gpu, n, length, unit, other, seed, quality=70):
    """n reads of `length` bases on the device: every third from a tandem array of one `unit`, the others
    from a random genome of `other` bases."""
    g = gpu.Generator(device="cuda").manual_seed(seed)
    codes = gpu.randint(0, 4, (other,), generator=g, device="cuda", dtype=gpu.uint8)
    array = gpu.randint(0, 4, (unit,), generator=g, device="cuda", dtype=gpu.uint8).repeat(length // unit + 2)
    letters = gpu.tensor(list(b"ACGT"), dtype=gpu.uint8, device="cuda")
    seq = gpu.empty((n, length), dtype=gpu.uint8, device="cuda")
    span = gpu.arange(length, device="cuda")
    for a in range(0, n, 200_000):
        b = min(n, a + 200_000)
        at = gpu.randint(0, other - length, (b - a,), generator=g, device="cuda")
        hot = gpu.arange(a, b, device="cuda") % 3 == 0
        row = codes[at[:, None] + span]
        row[hot] = array[(at[hot] % unit)[:, None] + span]
        seq[a:b] = letters[row.long()]
    offsets = gpu.arange(n + 1, device="cuda") * length
    return seq.view(-1), gpu.full((n * length,), quality, dtype=gpu.uint8, device="cuda"), offsets


def same_result(gpu, a, b):
    """Two finalized handles hold the same records (in any order)."""
    got = []
    for ka in (a, b):
        keys, counts, ext, codes = ka.copy_result_device()
        order = gpu.argsort(keys[:, 0], stable=True)
        order = order[gpu.argsort(keys[order, 1], stable=True)]
        got.append([x[order] for x in (keys, counts, ext, codes)])
    for x, y in zip(*got):
        assert gpu.equal(x, y)
    assert int(a.result_info.n_uu) == int(b.result_info.n_uu)
    assert int(a.result_info.valid_windows) == int(b.result_info.valid_windows)


@pytest.mark.parametrize("bloom", [True, False])
def test_groups_of_buckets(gpu, bloom):
    """More than 2 GiB of records, hot k-mers among them: counted in groups of buckets, by finalize (sizes
    from the bucket totals), by finalize_to_host and in a graph (groups of a fixed number of
    buckets), as in one table; and with no valid window at all."""
    from paper_1705_11147_gb300 import BatchGraph, KmerAnalysis, host_result_buffers, make_params
    reads = device_reads(gpu, 950_000, 150, 171, 1_500_000, 5)
    kw = dict(k=51, min_depth=2 if bloom else 1, use_bloom=bloom, max_bases=reads[0].numel(), max_reads=950_000, expected_distinct=4_000_000,
              expected_keys=3_000_000)
    assert reads[0].numel() * 16 > 2 << 30
    with KmerAnalysis(make_params(**kw, partitions=1)) as one, KmerAnalysis(make_params(**kw, partitions=8)) as ka:
        one.count(*reads)
        one.finalize()
        assert int(one.result_info.n) > 1_400_000
        ka.count(*reads)
        ka.finalize()
        same_result(gpu, one, ka)
        ka.reset()
        ka.count(*reads)
        res = ka.finalize_to_host(host_result_buffers(4_000_000, pinned=True)).sorted()
        np.testing.assert_array_equal(res.keys, one.copy_result().sorted().keys)
        same_result(gpu, one, ka)
        graph = BatchGraph([ka], [reads])
        graph.replay()
        graph.results()
        same_result(gpu, one, ka)
        del graph
        ka.set_stream(gpu.cuda.current_stream())
        ka.reset()
        none = gpu.full_like(reads[0], ord("N"))
        ka.count(none, reads[1], reads[2])
        assert int(ka.finalize().n) == 0 and int(ka.result_info.valid_windows) == 0
        assert not ka.query(one.copy_result_device()[0])[0].any()


@pytest.mark.parametrize("k,bloom", [(31, True), (51, True), (51, False)])
def test_more_keys_than_slots(gpu, k, bloom):
    """A table with fewer slots than keys: KMA_EFULL, and the handle counts again after reset."""
    from paper_1705_11147_gb300 import KmerAnalysis, capi, make_params
    reads = device_reads(gpu, 40_000, 150, 171, 2_000_000, 6)
    few = device_reads(gpu, 300, 150, 171, 1_000, 7)
    kw = dict(k=k, min_depth=2 if bloom else 1, use_bloom=bloom, max_bases=reads[0].numel(), max_reads=40_000, expected_distinct=2_000_000)
    for slots in (50_000, 200_000):
        with KmerAnalysis(make_params(**kw, partitions=4, table_capacity=slots)) as ka, KmerAnalysis(make_params(**kw, partitions=1)) as one:
            ka.count(*reads)
            with pytest.raises(capi.KmaError) as e:
                ka.finalize()
            assert e.value.code == capi.KMA_EFULL
            for h in (ka, one):
                h.reset()
                h.count(*few)
                h.finalize()
            same_result(gpu, one, ka)


LITTLE_MEMORY = """
import sys
import torch as gpu
from test_gpu_limits import device_reads, same_result
from paper_1705_11147_gb300 import KmerAnalysis, finalize_batch, host_result_buffers, make_params
from paper_1705_11147_gb300.capi import KMA_ENOMEM, KmaError
k, keys, leave, host = (int(x) for x in sys.argv[1:])
out = host_result_buffers(4_000_000, pinned=True)
few = device_reads(gpu, 2_000, 150, 171, 10_000, 9)
small, alone = (KmerAnalysis(make_params(k=k, min_depth=2, max_bases=300_000, max_reads=2_000, expected_distinct=100_000, partitions=2))
                for _ in range(2))
for h in (small, alone):
    h.count(*few)
alone.finalize()
reads = device_reads(gpu, 600_000, 150, 171, 1_500_000, 5)
kw = dict(k=k, min_depth=2, max_bases=reads[0].numel(), max_reads=600_000, expected_distinct=4_000_000)
ka = KmerAnalysis(make_params(**kw, expected_keys=keys, partitions=8))
one = KmerAnalysis(make_params(**kw, expected_keys=3_000_000, partitions=1))
one.count(*reads)
one.finalize()
ka.count(*reads)
gpu.cuda.synchronize()
gpu.cuda.empty_cache()
free = gpu.cuda.mem_get_info()[0]
held = gpu.empty(free - (leave << 20), dtype=gpu.uint8, device="cuda")
if host == 1:
    n = ka.finalize_to_host(out)
elif host == 2:
    try:
        finalize_batch([small, ka])
        raise AssertionError("there was enough memory")
    except KmaError as e:
        assert e.code == KMA_ENOMEM
    del held
    gpu.cuda.empty_cache()
    finalize_batch([small, ka])
    assert small.result_info.table_keys == alone.result_info.table_keys
    assert small.timings()["first_sightings"] == alone.timings()["first_sightings"]
    same_result(gpu, alone, small)
else:
    n = ka.finalize()
held = None
gpu.cuda.empty_cache()
same_result(gpu, one, ka)
if host == 1:
    w, g = one.copy_result().sorted(), n.sorted()
    assert (w.keys == g.keys).all() and (w.counts == g.counts).all() and (w.ext == g.ext).all() and (w.codes == g.codes).all()
print("same")
"""


def little_memory(*args):
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([root, os.path.join(root, "tests")]))
    r = subprocess.run([sys.executable, "-c", LITTLE_MEMORY, *map(str, args)], cwd=root, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same" in r.stdout, r.stderr[-2000:]


@pytest.mark.parametrize("k,leave", [(51, 1500), (31, 700)])
def test_little_memory_for_the_sorts(gpu, k, leave):
    """Not enough memory for the sorted copy of all records at once: smaller groups of buckets."""
    little_memory(k, 3_000_000, leave, 0)


@pytest.mark.parametrize("k,keys,leave,host", [(51, 40_000_000, 1500, 0), (51, 40_000_000, 2470, 0), (51, 3_000_000, 240, 1)])
def test_little_memory_for_the_records(gpu, k, keys, leave, host):
    """No memory for the output that the table was sized for (2.4 GB), or none for the sorts beside it:
    the records are brought out when their number is known."""
    little_memory(k, keys, leave, host)


def test_finalize_again(gpu):
    """A batch whose second handle finds no memory can be finalized when there is: the first one's
    figures are not added up twice."""
    little_memory(51, 3_000_000, 90, 2)


@pytest.mark.parametrize("partitions", [1, 4])
@pytest.mark.parametrize("reason", ["reads", "long"])
def test_refused_host_reads(gpu, partitions, reason):
    """A call that does not fit, by its number of reads or by one read longer than the staging buffer
    behind others, counts none of its reads, also when it is copied in pieces."""
    from paper_1705_11147_gb300 import KmerAnalysis, capi, make_params
    rng = np.random.default_rng(4)
    seq = np.frombuffer(b"ACGT", np.uint8)[rng.integers(0, 4, 30_000_000)]
    qual = np.full(len(seq), 70, np.uint8)
    offsets = np.arange(0, len(seq) + 1, 50, dtype=np.uint64)
    if reason == "long":
        offsets = np.concatenate([offsets[:400_000], [np.uint64(len(seq))]])
    kw = dict(k=31, min_depth=1, use_bloom=False, max_bases=30_000_000, max_reads=1000, expected_distinct=200_000, expected_keys=100_000,
              staging_bytes=9_000_000 if reason == "long" else 0, partitions=partitions)
    with KmerAnalysis(make_params(**kw)) as ka:
        with pytest.raises(capi.KmaError) as e:
            ka.count(seq, qual, offsets)
        assert e.value.code == (capi.KMA_EINVAL if reason == "long" else capi.KMA_EFULL)
        ka.count(seq[:500], qual[:500], offsets[:11])
        info = ka.finalize()
        assert int(info.valid_windows) == 200 and int(info.n) == 200
