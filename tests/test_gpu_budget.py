"""Device memory: a call that fails for want of memory keeps none of it."""
import numpy as np
import pytest

import datagen
import oracle
from gpu_util import amplicon, assert_same_result

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_reads", [400, 20_000])  # counted by sorting, by hashing
def test_a_failed_allocation_leaks_nothing(hsk, n_reads):
    """Whichever allocation of a call fails, the context holds as much after a
    later good call as one that never failed."""
    reads, offs = datagen.random_reads(7, n_reads, 150, 150)
    with hsk.Context() as ctx:
        ctx.count(reads, offs, 31, 17, 1, 1000)
        want = ctx.allocated()
    failed = 0
    for i in range(60):
        with hsk.Context() as ctx:
            ctx.fail_alloc_after(i)
            try:
                ctx.count(reads, offs, 31, 17, 1, 1000)
                break
            except hsk.HskError as e:
                assert e.code == hsk.HSK_ENOMEM
            failed += 1
            ctx.fail_alloc_after(-1)
            ctx.count(reads, offs, 31, 17, 1, 1000)
            assert ctx.allocated() == want, f"allocation {i}"
    assert failed > 15


@pytest.mark.parametrize("budget_mb", [176, 180])
def test_a_budget_for_the_sorting_path_is_enough(hsk, budget_mb):
    """Partitions that the hash count cannot take are gathered beside the
    originals; where the budget has no room for that, the sorting path alone
    counts the job."""
    reads, offs = amplicon(12_000_000, 1)
    want = oracle.count(reads, offs, 55, 1, 1000)
    with hsk.Context(hbm_budget=budget_mb << 20) as ctx:
        assert_same_result(ctx.count(reads, offs, 55, 21, 1, 1000), want, f"{budget_mb} MB")
        assert ctx.allocated() <= budget_mb << 20


def test_occurrences_within_a_budget_for_the_sorting_path(hsk):
    """The arrays that only the count needs make room for the occurrence lists."""
    reads, offs = amplicon(12_000_000, 1)
    want = oracle.count_ext(reads, offs, 55, 2, 1000)
    with hsk.Context(hbm_budget=218 << 20) as ctx:
        res, off, rd, ps = ctx.count_ext(reads, offs, 55, 21, 2, 1000)
    assert np.array_equal(res.kmers, want.kmers) and np.array_equal(res.counts, want.counts)
    assert np.array_equal(off, want.occ_offsets)
    assert np.array_equal(rd, want.occ_read) and np.array_equal(ps, want.occ_pos)
