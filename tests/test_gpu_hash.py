"""Counting by on-chip hashing (k_hash.cu) against the CPU oracle: key widths
at their edges, partitions that overfill the table, equal records on both
strands, and jobs on either side of the smallest size it takes."""
import numpy as np
import pytest

import datagen
import oracle
from gpu_util import assert_same_result

pytestmark = pytest.mark.gpu


def _join(strs):
    offs = np.zeros(len(strs) + 1, np.uint64)
    offs[1:] = np.cumsum([len(s) for s in strs])
    return np.frombuffer("".join(strs).encode(), np.uint8).copy(), offs


@pytest.mark.parametrize("k,m", [(12, 10), (21, 11), (31, 17), (32, 16), (33, 17), (55, 21), (63, 32), (64, 21)])
@pytest.mark.parametrize("coverage", [1.5, 40.0])
def test_key_widths_and_coverages(hsk, k, m, coverage):
    rs = datagen.batched_set(datagen.derive_seed(k, m), int(4_500_000 / coverage), coverage)
    for lo, hi in ((1, 1 << 30), (2, 20)):
        want = oracle.count(rs.reads, rs.offsets, k, lo, hi)
        with hsk.Context() as ctx:
            assert_same_result(ctx.count(rs.reads, rs.offsets, k, m, lo, hi), want, f"k={k} lo={lo}")


def _fmix32(h):
    h = np.asarray(h, np.uint32).copy()
    with np.errstate(over="ignore"):
        h ^= h >> np.uint32(16)
        h *= np.uint32(0x85EBCA6B)
        h ^= h >> np.uint32(13)
        h *= np.uint32(0xC2B2AE35)
        h ^= h >> np.uint32(16)
    return h


def _low_score_mmer(rng, m, seed):
    """An m-mer whose score is the least of 200,000 random ones."""
    c = rng.integers(0, 4, size=(200_000, m))
    w = (np.uint64(1) << (2 * np.arange(m - 1, -1, -1)).astype(np.uint64))
    f = (c.astype(np.uint64) * w).sum(1, dtype=np.uint64)
    r = ((3 - c[:, ::-1]).astype(np.uint64) * w).sum(1, dtype=np.uint64)
    v = np.minimum(f, r)
    s = _fmix32((v & np.uint64(0xFFFFFFFF)).astype(np.uint32) ^ (v >> np.uint64(32)).astype(np.uint32) ^
                np.uint32(seed & 0xFFFFFFFF))
    return "".join("ACGT"[x] for x in c[int(np.argmin(s))])


@pytest.mark.parametrize("k,m,n", [(31, 17, 500), (31, 17, 900), (31, 17, 20_000), (55, 21, 150), (55, 21, 3_000)])
def test_partitions_that_overfill_the_table(hsk, k, m, n):
    """n reads around one low-scoring m-mer: up to k - m + 1 distinct k-mers
    each, nearly all in one partition -- within the first table, within the
    larger one, and in neither (then the sorting path takes the partition)."""
    rng = np.random.default_rng(n + k)
    mm = _low_score_mmer(rng, m, hsk.DEFAULT_SEED)
    side = k - m
    acgt = np.array(list("ACGT"))
    strs = ["".join(rng.choice(acgt, side)) + mm + "".join(rng.choice(acgt, side)) for _ in range(n)]
    strs += ["".join(rng.choice(acgt, 300)) for _ in range(600)]
    comp = str.maketrans("ACGT", "TGCA")
    strs += [s.translate(comp)[::-1] for s in strs[:: 3]]  # the other strand of every third read
    reads, offs = _join(strs)
    want = oracle.count(reads, offs, k, 1, 1000)
    with hsk.Context() as ctx:
        for _ in range(2):
            assert_same_result(ctx.count(reads, offs, k, m, 1, 1000), want, f"n={n}")


@pytest.mark.parametrize("n_reads", [545, 546, 547])
def test_either_side_of_the_smallest_size(hsk, n_reads):
    """150-base reads have 120 31-mers: 65,400 to 65,640 windows around 2^16."""
    reads, offs = datagen.random_reads(n_reads, n_reads, 150, 150)
    want = oracle.count(reads, offs, 31, 1, 1000)
    with hsk.Context() as ctx:
        assert_same_result(ctx.count(reads, offs, 31, 17, 1, 1000), want, f"{n_reads} reads")


@pytest.mark.parametrize("k", [31, 55])
def test_one_record_many_times(hsk, k):
    """Repeated reads make a few records with thousands of copies (more than a
    batch holds) next to unique ones."""
    rng = np.random.default_rng(k)
    acgt = np.array(list("ACGT"))
    rep = "".join(rng.choice(acgt, 130))
    strs = [rep] * 5000 + ["".join(rng.choice(acgt, 200)) for _ in range(500)] + ["A" * 3000]
    reads, offs = _join(strs)
    want = oracle.count(reads, offs, k, 1, 1 << 30)
    with hsk.Context() as ctx:
        assert_same_result(ctx.count(reads, offs, k, 17, 1, 1 << 30), want, "repeats")


@pytest.mark.parametrize("k,m", [(31, 17), (55, 21)])
@pytest.mark.parametrize("copies", [2, 4, 6, 8, 60])
def test_few_entries_left_after_the_first_round(hsk, k, m, copies):
    """Every read `copies` times: a batch of records holds ever fewer distinct
    k-mers, so that about 300 down to none of them share a slot at first (the
    last 64 are settled by one warp)."""
    rng = np.random.default_rng(100 * k + copies)
    reads = ["".join("ACGT"[x] for x in rng.integers(0, 4, 2000)) for _ in range(max(1, 120 // copies))]
    r, o = _join(reads * copies)
    with hsk.Context() as ctx:
        assert_same_result(ctx.count(r, o, k, m, 1, 1 << 30), oracle.count(r, o, k, 1, 1 << 30), f"{copies} copies")


def test_chunks_and_small_histogram(hsk):
    rs = datagen.batched_set(datagen.derive_seed(9, 9), 400_000, 12.0)
    want = oracle.count(rs.reads, rs.offsets, 31, 1, 5, hist_len=7)
    with hsk.Context(hist_len=7, max_chunk_kmers=900_000) as ctx:
        got = ctx.count(rs.reads, rs.offsets, 31, 17, 1, 5)
    assert got.n_chunks > 3
    assert_same_result(got, want, "chunks")


@pytest.mark.parametrize("k,m", [(31, 17), (21, 11), (55, 21), (64, 32)])
def test_large_packs_are_counted_by_hashing(hsk, k, m):
    """Packed passes of several million bases: sets of very different sizes
    (among them empty ones and one of a single repeated read) and filters that
    keep everything or little; each result is the oracle's for the set alone."""
    rng = np.random.default_rng(k)
    jobs = []
    for i in range(20):
        g = int(np.exp(rng.uniform(np.log(3_000), np.log(400_000))))
        rs = datagen.batched_set(datagen.derive_seed(k, i), g, float(rng.uniform(5, 30)))
        jobs.append((rs.reads, rs.offsets))
    jobs.insert(3, (np.zeros(0, np.uint8), np.zeros(1, np.uint64)))
    jobs.insert(7, _join(["ACGT" * 30] * 3000))
    jobs.insert(9, _join(["N" * 5000, "A" * 20000]))
    for lo, hi in ((1, 1 << 30), (2, 1000)):
        wants = [oracle.count(r, o, k, lo, hi) for r, o in jobs]
        with hsk.Context() as ctx:
            ctx.tune_set(slots=1)
            for _ in range(2):
                got = ctx.count_batch([(r, o, k, m, lo, hi) for r, o in jobs])
                for i, (a, b) in enumerate(zip(got, wants)):
                    assert_same_result(a, b, f"k={k} lo={lo} set {i}")
            assert ctx.pack_stats()["failed_passes"] == 0
