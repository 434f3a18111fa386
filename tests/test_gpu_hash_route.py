"""Which jobs and packs are counted by hashing (hsk_debug_hash_stats): the tuned
parameters that concern the sorting path do not decide it."""
import numpy as np
import pytest

import oracle
from gpu_util import ACGT, assert_same_result, bases, reads_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("group_div", [1, 2, 3, 6])
@pytest.mark.parametrize("k,m", [(31, 17), (55, 21)])
def test_packs_hash_whatever_group_div(hsk, k, m, group_div):
    """Sets on either side of what one bucket holds on each path."""
    sizes = [60_000, 349_500, 393_300, 450_000, 516_300, 524_400, 1_100_000, 1_300_000]
    jobs = [reads_of(bases(max(2000, n // 8), i), n // 150, 150, 0.002, 50 + i) + (k, m, 2, 1000)
            for i, n in enumerate(sizes)]
    wants = [oracle.count(r, o, k, 2, 1000) for r, o, *_ in jobs]
    with hsk.Context() as ctx:
        ctx.tune_set(slots=1, group_div=group_div)
        for i, (g, w) in enumerate(zip(ctx.count_batch(jobs), wants)):
            assert_same_result(g, w, f"group_div={group_div} set {i}")
        st, packs = ctx.pack_stats(), ctx.hash_stats()["packs"]
    assert st["sets"] == len(jobs) and st["failed_passes"] == 0 and st["alone"] == 0, st
    assert packs == st["passes"] > 0, (packs, st)


@pytest.mark.parametrize("k,m,most", [(31, 17, 256 * 3072), (55, 21, 256 * 4032)])
@pytest.mark.parametrize("around", [-1, 0, 1])
def test_either_side_of_the_largest_job(hsk, k, m, most, around):
    """A context's own n_buckets (here one) limits the bases the hash count takes."""
    n = most + around
    template = bases(300_000, k)
    reads = ACGT[np.tile(template, n // template.size + 1)[:n]]
    offs = np.array([0, n // 3, n], np.uint64)
    want = oracle.count(reads, offs, k, 1, 1000)
    with hsk.Context(n_buckets=1) as ctx:
        assert_same_result(ctx.count(reads, offs, k, m, 1, 1000), want, f"{n} bases")
        assert (ctx.hash_stats()["partitions"] > 0) == (around <= 0)


def test_a_tuned_bucket_shift_does_not_end_the_hash_path(hsk):
    """256 buckets (a shift of 4) have partitions for 201 M windows: a larger job
    takes more buckets instead of the sorting path.  Checked against the radix sort."""
    reads, offs = reads_of(bases(8_000_000, 1), 840_000, 250, 0.001, 2)
    with hsk.Context() as ctx:
        ctx.tune_set(plain_bucket_shift=4)
        got = ctx.count(reads, offs, 31, 17, 2, 1000)
        assert ctx.hash_stats()["partitions"] == 512 << 8
    with hsk.Context(local_sort=False) as ctx:
        assert_same_result(got, ctx.count(reads, offs, 31, 17, 2, 1000))
