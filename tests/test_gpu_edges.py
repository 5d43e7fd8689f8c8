"""Edges of the partitioned counter's two sorts and its shared-memory tables, of the vector paths
of the FASTQ parser and the lookups, of the summaries' merge and of the contigs' list ranking:
each against the CPU oracle. Every comparison is of whole numbers, so exact."""
import numpy as np
import pytest

import oracle
import synth
from test_gpu_parity import (_check_contigs, _check_heavy_summary, _to_fastq, assert_same, gpu, oracle_for,  # noqa: F401
                             readset, run_gpu)

pytestmark = pytest.mark.gpu

TILE = 8192  # window starts per scatter tile


def one_read(n, seed, alphabet="ACGT"):
    rng = np.random.default_rng(seed)
    return "".join(np.array(list(alphabet))[rng.integers(0, len(alphabet), n)])


def oracle_absent(keys, k):
    """Keys of random k-mers that are not among `keys`."""
    have = {(int(a), int(b)) for a, b in keys}
    rng = np.random.default_rng(13)
    out = [(int(rng.integers(0, 1 << min(2 * k, 62))), int(rng.integers(0, 1 << (2 * k - 64))) if 2 * k > 64 else 0) for _ in range(2000)]

    def canonical(key):
        x, y = key[0] | key[1] << 64, 0
        for i in range(k):
            y |= (3 - (x >> 2 * i & 3)) << 2 * (k - 1 - i)
        x = min(x, y)
        return x & (1 << 64) - 1, x >> 64
    return np.array([q for q in out if canonical(q) not in have], np.uint64)


def both(gpu, rs, what, **kw):
    """Partitioned and oracle, with and without the minimum of two sightings."""
    for depth in (1, 2, 3):
        for bloom in ((False,) if depth == 1 else (False, True)):
            rs.meta["params"].update(min_depth=depth)
            assert_same(run_gpu(gpu, rs, use_bloom=bloom, **kw), oracle_for(rs), f"{what} depth={depth} bloom={bloom}")


@pytest.mark.parametrize("k,canonical", [(1, True), (21, True), (31, True), (32, False), (33, True), (62, False), (63, True)])
def test_tile_edges(gpu, k, canonical):
    """Reads that end one position before, at and after the ends of scatter tiles and of the arena
    words, and a single window."""
    for n in (k, 63, 64, 65, TILE - 2, TILE - 1, TILE, TILE + 1, 2 * TILE + 65):
        if n < k:
            continue
        r = one_read(n, n + k)
        rs = readset([r, r[: n // 2], r], k=k, min_ext_count=2, qual_threshold=20, canonical=canonical)
        both(gpu, rs, f"k={k} n={n}", partitions=3)


@pytest.mark.parametrize("threshold", [0, 20, 41, 300])
def test_packing(gpu, threshold):
    """Reads and qualities that start at different bytes of a 16-byte piece, reads of every length
    from none to more than a word, and thresholds that all, some and no qualities reach."""
    from paper_1705_11147_gb300 import KmerAnalysis, make_params
    rng = np.random.default_rng(11)
    lens = list(range(0, 70)) + [0] * 70 + [1, 2] * 40 + [63, 64, 65, 127, 128, 129, 20_000]
    reads = [one_read(n, 70 + n, "ACGTACGTacgtNx") for n in lens] * 2
    quals = ["".join(chr(33 + x) for x in rng.integers(0, 42, len(r))) for r in reads]
    rs = readset(reads, quals, k=5, min_depth=1, min_ext_count=1, qual_threshold=threshold)
    want = oracle_for(rs)
    for a, b in ((0, 0), (1, 1), (3, 8), (15, 0), (0, 15), (7, 6)):
        seq, qual = (gpu.zeros(rs.n_bases + 16, dtype=gpu.uint8, device="cuda")[o:o + rs.n_bases] for o in (a, b))
        seq.copy_(gpu.from_numpy(rs.seq))
        qual.copy_(gpu.from_numpy(rs.qual))
        with KmerAnalysis(make_params(max_bases=rs.n_bases, max_reads=rs.n_reads, expected_distinct=rs.n_bases, use_bloom=False,
                                      **rs.meta["params"])) as ka:
            ka.count(seq, qual, gpu.from_numpy(rs.offsets.astype(np.int64)).cuda())
            ka.finalize()
            assert_same(ka.copy_result().sorted(), want, (a, b))


@pytest.mark.parametrize("k", [31, 33])
@pytest.mark.parametrize("kind", ["one key", "few keys", "crowded", "distinct", "mixed"])
def test_sub_bucket_shapes(gpu, k, kind):
    """Sub-buckets that overflow (one key more than 2^16 times, a few hot keys), whose keys are all
    repeated (every record goes to the second table) or all distinct, and a mix of them."""
    reads = []
    if kind in ("one key", "mixed"):
        reads += ["A" * 1500] * 50
    if kind in ("few keys", "mixed"):
        unit = one_read(171, 5)
        reads += [(unit * 6)[i:i + 700] for i in range(0, 300, 3)] * 2
    if kind in ("crowded", "mixed"):
        g = one_read(40_000, 6)
        reads += [g] * 4
    if kind in ("distinct", "mixed"):
        reads += [one_read(20_000, 100 + i) for i in range(8)]
    rs = readset(reads, k=k, min_ext_count=2, qual_threshold=20)
    both(gpu, rs, f"{kind} k={k}", partitions=4)
    both(gpu, rs, f"{kind} k={k}, a few buckets", partitions=64)


@pytest.mark.parametrize("k", [25, 51])
def test_more_records_than_room(gpu, k):
    """More records than the output arrays are first given: they are compacted from the table."""
    rs = readset([one_read(3000, 300 + i) for i in range(20)], k=k, min_ext_count=2, qual_threshold=20)
    rs.meta["params"].update(min_depth=1)
    want = oracle_for(rs)
    for load in (0.05, 0.9):
        assert_same(run_gpu(gpu, rs, use_bloom=False, partitions=8, load_factor=load, table_capacity=1 << 17), want, load)


@pytest.mark.parametrize("k", [31, 51])
@pytest.mark.parametrize("partitions", [2, 7, 64])
def test_table_of_ranges(gpu, k, partitions):
    """The table that is made a sub-bucket's range at a time, roomy and nearly full (keys that find no
    slot in their range, go round a partition's end or into the next group's slots), in one group of
    buckets and in eight: every key is found in it, and no other."""
    from paper_1705_11147_gb300 import KmerAnalysis, make_params
    rs = readset([one_read(3000, 500 + i) for i in range(20)], k=k, min_ext_count=1, qual_threshold=20, min_depth=1)
    want = oracle_for(rs)
    absent = oracle_absent(want.keys, k)
    for slots in (1.02, 1.2, 12.0):
        for to_host in (False, True):
            # the partitions' shares of the keys differ by a few standard deviations
            room = int(len(want) * slots) + int(6 * np.sqrt(len(want) * partitions))
            with KmerAnalysis(make_params(max_bases=rs.n_bases, max_reads=rs.n_reads, use_bloom=False, partitions=partitions,
                                          table_capacity=room, **rs.meta["params"])) as ka:
                for _ in range(2):  # also over the table of a sample before
                    ka.reset()
                    ka.count(rs.seq, rs.qual, rs.offsets)
                    if to_host:
                        n = len(want) + 5
                        ka.finalize_to_host((np.empty((n, 2), np.uint64), np.empty(n, np.uint32), np.empty((n, 8), np.uint32),
                                             np.empty((n, 2), np.uint8)))
                    else:
                        ka.finalize()
                    counts, ext, codes = ka.query(want.keys)
                    assert np.array_equal(counts, want.counts) and np.array_equal(ext, want.ext)
                    assert np.array_equal(codes, want.codes)
                    assert not ka.query(absent)[0].any()


@pytest.mark.parametrize("partitions", [1, 6])
def test_no_reads(gpu, partitions):
    """A handle without a window, after one with some: an empty result and an empty table."""
    from paper_1705_11147_gb300 import KmerAnalysis, make_params
    rs = readset([one_read(500, 6)] * 2, k=31, min_depth=2, min_ext_count=1, qual_threshold=20)
    keys = oracle_for(rs).keys
    with KmerAnalysis(make_params(max_bases=rs.n_bases, max_reads=rs.n_reads, partitions=partitions, **rs.meta["params"])) as ka:
        for some in (False, True, False):
            ka.reset()
            if some:
                ka.count(rs.seq, rs.qual, rs.offsets)
            assert ka.finalize().n == (len(keys) if some else 0)
            assert ka.query(keys)[0].astype(bool).all() == some and ka.query(keys)[0].any() == some


@pytest.mark.parametrize("n_parts", [2, 7])
def test_batches_and_owners(gpu, n_parts):
    """Several count calls (slabs of scatter tiles) and the owner filter: the parts' records add up."""
    rs = synth.random_reads(seed=8, n_reads=4000, min_len=0, max_len=200, alphabet=b"ACGTACGTACGTN", q_lo=10, q_hi=40)
    rs.meta["params"] = dict(k=31, min_depth=1, min_ext_count=2, qual_threshold=20)
    want = oracle_for(rs)
    got = [run_gpu(gpu, rs, use_bloom=False, partitions=5, batches=9, n_parts=n_parts, part=p) for p in range(n_parts)]
    rows = np.concatenate([np.column_stack([g.keys, g.counts.astype(np.uint64), g.ext.astype(np.uint64)]) for g in got])
    rows = rows[np.lexsort((rows[:, 0], rows[:, 1]))]
    ref = np.column_stack([want.keys, want.counts.astype(np.uint64), want.ext.astype(np.uint64)])
    assert np.array_equal(rows, ref[np.lexsort((ref[:, 0], ref[:, 1]))])


@pytest.mark.parametrize("k", [31, 63])
def test_partitioned_as_one_table(gpu, k):
    """The rule that takes a sample to partitions: the same records as one table for any number of
    them, device and host input, and into host arrays."""
    rs = synth.random_reads(seed=9, n_reads=3000, min_len=30, max_len=260, alphabet=b"ACGTACGTACGTACGTacgtN", q_lo=10, q_hi=40)
    rs = synth.ReadSet(np.concatenate([rs.seq, rs.seq]), np.concatenate([rs.qual, rs.qual]),
                       np.concatenate([rs.offsets, rs.offsets[1:] + rs.offsets[-1]]))
    rs.meta["params"] = dict(k=k, min_depth=2, min_ext_count=2, qual_threshold=20)
    one = run_gpu(gpu, rs, partitions=1)
    assert_same(one, oracle_for(rs), "one table")
    for parts in (2, 3, 16, 100, 1000):
        assert_same(run_gpu(gpu, rs, partitions=parts, device_inputs=parts % 2 == 0, batches=parts % 3 + 1), one, parts)


@pytest.mark.parametrize("shift", [0, 1, 7, 15])
@pytest.mark.parametrize("final_newline", [True, False])
def test_fastq_alignment(gpu, shift, final_newline):
    """Text that starts at any address and ends at any byte of a 16-byte piece or a chunk."""
    from paper_1705_11147_gb300 import parse_fastq
    for extra in range(0, 17, 2 if shift else 1):
        n = 40
        lens = [0, 1, 7, 8, 9, 15, 16, 17, 127, 128, 129, 255 + extra] + [100 + i for i in range(n)] + [65_400 - 30 * extra]
        reads = [one_read(m, 1000 + m, "ACGTN") for m in lens]
        text = "".join(f"@r{i}\n{r}\n+\n{'I' * len(r)}\n" for i, r in enumerate(reads))
        text += "@last\nACGT\n+\nIIII" + ("\n" if final_newline else "")
        raw = np.frombuffer(text.encode(), np.uint8)
        buf = gpu.zeros(len(raw) + 64, dtype=gpu.uint8, device="cuda")
        buf[:] = ord("\n")  # newlines around the text must not be seen
        buf[16 + shift:16 + shift + len(raw)] = gpu.from_numpy(raw.copy()).cuda()
        got = [x.cpu().numpy() for x in parse_fastq(buf[16 + shift:16 + shift + len(raw)])]
        for a, b in zip(got, oracle.parse_fastq(text.encode())):
            assert np.array_equal(a, b), (shift, extra)


@pytest.mark.parametrize("partitions", [1, 6])
def test_query_slices(gpu, partitions):
    """Keys and answers at addresses that the wide accesses cannot take, against those they can."""
    from paper_1705_11147_gb300 import KmerAnalysis, make_params
    r = one_read(5000, 77)
    rs = readset([r, r, r[100:400]], k=31, min_depth=2, min_ext_count=2, qual_threshold=20)
    with KmerAnalysis(make_params(max_bases=rs.n_bases, max_reads=rs.n_reads, expected_distinct=rs.n_bases, partitions=partitions,
                                  **rs.meta["params"])) as ka:
        ka.count(rs.seq, rs.qual, rs.offsets)
        ka.finalize()
        want = ka.copy_result()
        keys = np.concatenate([want.keys, want.keys ^ np.uint64(5)])
        n = len(keys)
        flat = gpu.zeros(2 * n + 1, dtype=gpu.int64, device="cuda")
        flat[1:] = gpu.from_numpy(keys.view(np.int64).reshape(-1)).cuda()
        aligned = flat[1:].clone().view(n, 2)
        a = ka.query(aligned)
        for key_off, ext_off, code_off in ((1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 1)):
            q = flat[1:].view(n, 2) if key_off else aligned
            out = (gpu.empty(n, dtype=gpu.int32, device="cuda"),
                   gpu.empty(8 * n + 1, dtype=gpu.int32, device="cuda")[ext_off:8 * n + ext_off].view(n, 8),
                   gpu.empty(2 * n + 1, dtype=gpu.uint8, device="cuda")[code_off:2 * n + code_off].view(n, 2))
            for x, y in zip(a, ka.query(q, out)):
                assert gpu.equal(x, y)
        assert np.array_equal(a[0][:len(want)].cpu().numpy().view(np.uint32), want.counts)
        assert np.array_equal(a[1][:len(want)].cpu().numpy().view(np.uint32), want.ext)


def test_query_host_arrays(gpu):
    """Host arrays of lookups below, at and above the size that is copied by several threads, and two
    calls at once: as with device arrays."""
    import threading

    from paper_1705_11147_gb300 import KmerAnalysis, make_params
    r = one_read(5000, 78)
    rs = readset([r, r], k=31, min_depth=2, min_ext_count=2, qual_threshold=20)
    edge = (8 << 20) // 38
    with KmerAnalysis(make_params(max_bases=rs.n_bases, max_reads=rs.n_reads, expected_distinct=rs.n_bases,
                                  **rs.meta["params"])) as ka:
        ka.count(rs.seq, rs.qual, rs.offsets)
        ka.finalize()
        found = ka.copy_result().keys
        for n in (1, edge, edge + 1, 700_001):
            keys = found[np.random.default_rng(n).integers(0, len(found), n)]
            keys[::3] ^= np.uint64(9)
            want = [x.cpu().numpy() for x in ka.query(gpu.from_numpy(keys.view(np.int64)).cuda())]
            got = [None, None]

            def look(i):
                got[i] = ka.query(keys)

            threads = [threading.Thread(target=look, args=(i,)) for i in range(2 if n > edge else 1)]
            [t.start() for t in threads]
            [t.join() for t in threads]
            for answer in got[:len(threads)]:
                for x, y in zip(answer, want):
                    assert np.array_equal(x.view(y.dtype), y), n


@pytest.mark.parametrize("partitions", [1, 5])
def test_host_pieces(gpu, partitions):
    """Host reads that are copied in pieces, one read longer than a piece among them."""
    piece = 8 << 20
    reads = [one_read(n, 60 + i) for i, n in enumerate((1, piece + 5, 40, piece - 45, 200, 3, piece // 2))]
    rs = readset(reads, k=31, min_depth=1, min_ext_count=1, qual_threshold=20)
    kw = dict(use_bloom=False, partitions=partitions)
    assert_same(run_gpu(gpu, rs, device_inputs=False, **kw), run_gpu(gpu, rs, **kw), "pieces")


@pytest.mark.parametrize("k", [31, 51])
def test_summary_merge(gpu, k):
    """Fewer and more keys than a summary holds, one key above all, the all-A key."""
    from paper_1705_11147_gb300 import estimate_distinct
    for reads in (["A" * 40_000], ["A" * 30_000, one_read(300_000, 3)], [one_read(64 * 20, 4)] * 400, [one_read(1_500_000, 5)]):
        rs = readset(reads, k=k)
        est = estimate_distinct(rs.seq, rs.qual, rs.offsets, k=k)
        _check_heavy_summary(est, rs, k)


@pytest.mark.parametrize("k", [21, 51])
def test_contig_lengths(gpu, k):
    """Chains of one vertex, around the jumps of one launch, long ones, and cycles."""
    reads = [one_read(k + n, 50 + n) for n in (0, 1, 2, 15, 16, 17, 31, 33, 1000)] + [one_read(30_000, 51)]
    for n in (5, 40, 700):  # a circle
        c = one_read(n + k, 900 + n)
        reads.append(c + c[:k])
    _check_contigs(gpu, readset([r for r in reads for _ in range(2)]), k)
    _check_contigs(gpu, readset([one_read(k, 52)] * 2), k)
