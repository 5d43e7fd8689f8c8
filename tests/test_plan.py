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


@pytest.mark.parametrize("kw,gb", [
    (dict(k=51, max_bases=120_000_000, expected_distinct=40_000_000, expected_keys=6_000_000), 4.45),
    (dict(k=51, max_bases=250_000_000, expected_distinct=100_000_000, expected_keys=8_000_000), 7.27),
    (dict(k=31, max_bases=30_000_000, expected_distinct=8_000_000, expected_keys=1_500_000), 1.86),
    (dict(k=51, max_bases=6_000_000_000, expected_distinct=2_100_000_000, expected_keys=300_000_000), 157.1)])
def test_planned_bytes(plan, kw, gb):
    """What a partitioned handle is planned with stays near one copy of the records (17 or 9 bytes a base,
    the filter and the table: the given figure). A serving loop admits its jobs by it."""
    assert plan(**kw).device_bytes < 1.4e9 * gb
