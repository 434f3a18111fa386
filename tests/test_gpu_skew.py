"""Reads crowded around a few minimizers (deep amplicons, low complexity):
their fine partitions hold far more records or distinct k-mers than an SM's
table, next to partitions that hold few.  Every result is the CPU oracle's."""
import numpy as np
import pytest

import oracle
from gpu_util import ACGT, amplicon, assert_same_result, bases, join, low_score_mmer, reads_of

pytestmark = pytest.mark.gpu


def poly(unit, n):
    return np.tile(np.array(["ACGT".index(c) for c in unit], np.uint8), n // len(unit) + 1)[:n]


@pytest.mark.parametrize("k,m", [(31, 17), (55, 21), (12, 12)])
@pytest.mark.parametrize("length", [60, 150, 5000])
def test_low_complexity_reads(hsk, k, m, length):
    """Runs longer than a record, tiles with one minimizer, and errors."""
    reads, offs = join(reads_of(poly("A", 6000), 300_000 // length, length, 0.0, 1),
                       reads_of(poly("AT", 6000), 300_000 // length, length, 0.002, 2),
                       reads_of(poly("ACG", 6000), 300_000 // length, length, 0.01, 3),
                       reads_of(bases(20_000, 4), 300_000 // length, length, 0.005, 5))
    want = oracle.count(reads, offs, k, 1, 1 << 30)
    with hsk.Context() as ctx:
        assert_same_result(ctx.count(reads, offs, k, m, 1, 1 << 30), want, f"k={k} length={length}")


def _stage_ms(ctx, stage, reads, offs, k, m):
    ctx.profile()
    best = 1e9
    for _ in range(5):
        ctx.count(reads, offs, k, m, 2, 1000, copy=False)
        best = min(best, ctx.profile_read()[0][stage])
    return best


def test_walk_is_as_fast_on_one_minimizer(hsk):
    """Records counted at one address must not queue there: the walk over reads
    of one base against the same number of random reads (six times as long with
    an atomic per record, less than twice without)."""
    n = 250_000
    crowd, offs = reads_of(poly("A", 1000), n, 150, 0.0, 1)
    spread, _ = reads_of(bases(2_000_000, 2), n, 150, 0.0, 3)
    with hsk.Context() as ctx:
        a, b = (_stage_ms(ctx, 1, r, offs, 31, 17) for r in (crowd, spread))
    assert a < 3 * b, (a, b)


def crowd(n, m, side, seed):
    """n reads, each with its own `side` bases on both sides of one m-mer that no
    other scores below, so that all their k-mers of m + side bases share it."""
    low = low_score_mmer(np.random.default_rng(seed), m)
    x = np.empty((n, m + 2 * side), np.uint8)
    x[:, :side], x[:, side + m:] = (bases(n * side, seed + i).reshape(n, side) for i in (1, 2))
    x[:, side: side + m] = low
    return ACGT[x].reshape(-1), np.arange(n + 1, dtype=np.uint64) * np.uint64(x.shape[1])


@pytest.mark.parametrize("k,m", [(31, 17), (55, 21), (32, 16), (33, 17)])
@pytest.mark.parametrize("lo,hi", [(1, 1 << 30), (2, 50)])
def test_partitions_cut_into_slices(hsk, k, m, lo, hi):
    """Partitions of more records than one CTA should walk: of few distinct
    k-mers, of more than its table holds, of distinct ones only; and one of few
    records that overfills the second table.  With a low limit on the slices' pairs
    the same partitions go on to the sorting path."""
    spread = reads_of(bases(50_000, 1), 10_000, 150, 0.002, 2)
    few = reads_of(poly("A", 1000), 30_000, 150, 0.0, 3)
    many = reads_of(bases(120, 4), 60_000, 120, 0.01, 5)
    for label, sets in (("few", (spread, few)), ("many", (many, spread, few)),
                        ("distinct", (few, crowd(40_000, m, k - m, 6), spread)),
                        ("alone", (crowd(40_000, m, k - m, 6), spread)),
                        ("rejected", (crowd(1500, m, k - m, 7), spread))):
        reads, offs = join(*sets)
        want = oracle.count(reads, offs, k, lo, hi)
        with hsk.Context() as ctx:
            for _ in range(2):
                assert_same_result(ctx.count(reads, offs, k, m, lo, hi), want, f"k={k} {label}")
            s = ctx.hash_stats()
            assert s["heavy"] > 0 and s["sorted"] == 0 and (s["overfull"] > 0 or label != "rejected"), (label, s)
            assert label != "many" or s["pairs"] > 20_000, s  # slices that outgrew the table
            ctx.debug_limit("pairs", 4000)
            assert_same_result(ctx.count(reads, offs, k, m, lo, hi), want, f"k={k} {label}, sorted")
            t = ctx.hash_stats()
            assert t["sorted"] == (s["heavy"] if s["pairs"] > 4000 else 0), (label, s, t)


@pytest.mark.parametrize("around", [-1, 0, 1])
@pytest.mark.parametrize("k,m,most", [(31, 17, 16384), (55, 21, 6144)])
def test_either_side_of_a_heavy_partition(hsk, k, m, most, around):
    """Exactly so many records, all in one partition: reads of a full record (two
    when they cross a 1024-window tile), then reads of one k-mer."""
    per = (60 if k <= 32 else 124) - k + 1
    length, at, n_rec, lens = per + k - 1, 0, 0, []
    while n_rec < most + around:
        full = n_rec + 2 <= most + around
        lens.append(length if full else k)
        n_rec += (at + per - 1) // 1024 - at // 1024 + 1 if full else 1
        at += lens[-1]
    offs = np.cumsum([0] + lens).astype(np.uint64)
    reads = np.full(at, ord("A"), np.uint8)
    want = oracle.count(reads, offs, k, 1, 1 << 30)
    with hsk.Context() as ctx:
        assert_same_result(ctx.count(reads, offs, k, m, 1, 1 << 30), want, f"{most + around}")
        s = ctx.hash_stats()
    assert s["heavy"] == (1 if around > 0 else 0) and s["heavy"] + s["overfull"] == 1, s


@pytest.mark.parametrize("k,m", [(31, 17), (55, 21)])
def test_heavy_partitions_of_packed_sets(hsk, k, m):
    """The same k-mers are heavy in several sets of a pack, and counted for each."""
    spread = reads_of(bases(300_000, 1), 20_000, 150, 0.002, 2)
    jobs = [spread] + [join(reads_of(poly("A", 1000), 30_000 + 1000 * i, 150, 0.002 * i, 3 + i),
                            reads_of(bases(30_000, 9), 3000, 150, 0.0, 20 + i)) for i in range(4)] + [spread]
    wants = [oracle.count(r, o, k, 2, 1 << 20) for r, o in jobs]
    for limit in (None, 100):
        with hsk.Context() as ctx:
            ctx.tune_set(slots=1)
            if limit:
                ctx.debug_limit("pairs", limit)
            for _ in range(2):
                for i, (g, w) in enumerate(zip(ctx.count_batch([(r, o, k, m, 2, 1 << 20) for r, o in jobs]), wants)):
                    assert_same_result(g, w, f"k={k} set {i}")
            st = ctx.pack_stats()
        assert st["sets"] == 2 * len(jobs) and st["failed_passes"] == 0, st
        assert st["alone"] == (8 if limit else 0), st


@pytest.mark.parametrize("k,m,sizes", [(31, 17, (1023, 1024, 1025, 4000, 6143, 6144, 6145, 8192, 8193)),
                                       (55, 21, (255, 256, 257, 2048, 4095, 4096, 4097, 8192, 8193))])
@pytest.mark.parametrize("prefix", [9, 11, 13, 16])
def test_output_keys_that_share_their_top_bits(hsk, k, m, sizes, prefix):
    """So many k-mers with one prefix (of 18 to 32 bits) next to others: bins on
    either side of what is ranked, ranges on either side of what fits an SM."""
    sets = [reads_of(bases(30_000, 1), 4000, 150, 0.0, 2)]
    for i, n in enumerate(sizes):
        x = bases(n * k, 10 + i).reshape(n, k)
        x[:, :prefix] = [0, 0, 1 + i % 3] + [i // 3] * 2 + [3] * (prefix - 5)  # below the reverse complement's start
        sets.append((ACGT[x].reshape(-1), np.arange(n + 1, dtype=np.uint64) * np.uint64(k)))
    for some in ([sets[0]] + sets[1:4], sets):
        reads, offs = join(*some)
        want = oracle.count(reads, offs, k, 1, 1000)
        with hsk.Context() as ctx:
            assert_same_result(ctx.count(reads, offs, k, m, 1, 1000), want, f"k={k} prefix {prefix}")


def test_output_order_of_crowded_keys_is_not_quadratic(hsk):
    """S6 on the variants of an amplicon's k-mers against as many k-mers of random
    reads (fifteen times as long when every key is ranked in its bin)."""
    crowd = amplicon(12_000_000, 1)
    spread = reads_of(bases(1_000_000, 2), 60_000, 150, 0.0, 3)
    with hsk.Context() as ctx:
        ctx.profile()
        ms = []
        for reads, offs in (crowd, spread):
            best = 1e9
            for _ in range(5):
                n = ctx.count(reads, offs, 55, 21, 1, 1000, copy=False).extra["n_pairs"]
                best = min(best, ctx.profile_read()[0][6])
            ms.append(best / n)
    assert ms[0] < 8 * ms[1], ms
