"""Host-side sizing rules (kmer_analysis_plan), no GPU needed."""
import pytest


@pytest.fixture(scope="module")
def plan():
    from paper_1705_11147_gb300 import build, make_params
    from paper_1705_11147_gb300 import plan as p
    build.build()
    return lambda **kw: p(make_params(**kw))


@pytest.mark.parametrize("bloom,enough", [(True, 1_200_000), (False, 4_000_000)])
def test_small_samples_stay_in_one_table(plan, bloom, enough):
    """Partitions are for samples with enough windows to pay for the sorts' kernels, or a table that
    costs more than those to clear and to scan; up to 32 MB of filter and table there are none."""
    kw = dict(k=25, use_bloom=bloom, min_depth=2 if bloom else 1, expected_distinct=200_000)
    mb = 1 << 20
    for max_bases, table, parted in ((enough - 1, 64 * mb, False), (enough, 64 * mb, True), (enough - 1, 500 * mb, False),
                                     (50_000, 513 * mb, True), (enough, 20 * mb, False), (100 * enough, 20 * mb, False)):
        got = plan(max_bases=max_bases, table_capacity=table // 64, **kw).partitions
        assert (got > 1) == parted, (max_bases, table)
