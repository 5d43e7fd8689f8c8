"""Calls at the limits of what the library takes: other streams than the usual ones, arrays of
every origin, read sets and memory that leave the ordinary case. Every comparison is of whole
numbers, so exact."""
import mmap

import numpy as np
import pytest

import synth
from test_gpu_parity import gpu, to_dev  # noqa: F401

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
