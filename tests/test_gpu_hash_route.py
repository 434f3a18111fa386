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


@pytest.mark.parametrize("k,m", [(31, 17), (32, 16), (21, 11), (31, 31)])
def test_scatter_in_two_halves(hsk, k, m):
    """The descriptors from both ends of their array, with room for all, for all
    but a few (both ends meet, and the walk runs again) and for none."""
    reads, offs = reads_of(bases(200_000, 1), 20_000, 150, 0.002, 2)
    want = oracle.count(reads, offs, k, 1, 1000)
    with hsk.Context() as ctx:
        n = ctx.count(reads, offs, k, m, 1, 1000).n_supermers
    for room in (None, n + 1, n, n - 1, n // 2, 1, 0):
        for one_scatter in (0, 1 << 19):
            with hsk.Context() as ctx:
                ctx.debug_limit("one_scatter", one_scatter)
                if room is not None:
                    ctx.debug_limit("descriptors", room)
                got = ctx.count(reads, offs, k, m, 1, 1000)
                assert got.n_supermers == n and ctx.hash_stats()["partitions"] > 0
                assert_same_result(got, want, f"k={k} room {room} of {n}")


@pytest.mark.parametrize("k,m,lo,hi", [(31, 17, 2, 1000), (55, 21, 1, 3)])
def test_occurrences_through_wide_composites(hsk, k, m, lo, hi):
    """Index and position in two words, as past 64 bits of them."""
    reads, offs = reads_of(bases(60_000, 1), 6000, 150, 0.002, 2)
    want = oracle.count_ext(reads, offs, k, lo, hi)
    with hsk.Context() as ctx:
        for bits in (64, 30, 0):
            ctx.debug_limit("composite_bits", bits)
            res, off, rd, ps = ctx.count_ext(reads, offs, k, m, lo, hi)
            assert np.array_equal(res.kmers, want.kmers) and np.array_equal(res.counts, want.counts), bits
            assert np.array_equal(off, want.occ_offsets), bits
            assert np.array_equal(rd, want.occ_read) and np.array_equal(ps, want.occ_pos), bits
        with pytest.raises(hsk.HskError):
            ctx.debug_limit("composite_bits", 65)


@pytest.mark.parametrize("k,m", [(31, 17), (55, 21)])
def test_a_large_set_among_hundreds(hsk, k, m):
    """More sets than the output's second digit is kept for, one of them with
    ranges that do not fit an SM: the pack's pairs take the radix passes."""
    jobs = [reads_of(bases(1500, i), 20, 150, 0.0, 1000 + i) + (k, m, 1, 1000) for i in range(300)]
    jobs.insert(100, reads_of(bases(4_300_000, 7), 29_000, 150, 0.0, 8) + (k, m, 1, 1000))
    wants = [oracle.count(r, o, k, 1, 1000) for r, o, *_ in jobs]
    assert max(w.counts.size for w in wants) > 256 * 6144
    with hsk.Context(hist_len=256) as ctx:
        ctx.tune_set(slots=1)
        got = ctx.count_batch(jobs)
        st, packs = ctx.pack_stats(), ctx.hash_stats()["packs"]
    assert st["passes"] == packs == 1 and st["sets"] == 301 and st["failed_passes"] == 0 and st["alone"] == 0, st
    for i, (g, w) in enumerate(zip(got, wants)):
        assert np.array_equal(g.kmers, w.kmers) and np.array_equal(g.counts, w.counts), f"set {i}"
        assert (g.n_windows, g.n_distinct, g.max_count) == (w.n_windows, w.n_distinct, w.max_count), f"set {i}"
