"""Helpers shared by the GPU tests (device tensors from numpy, key decoding)."""
import numpy as np


def dev(a, dtype=None):
    import torch
    t = torch.from_numpy(np.ascontiguousarray(a))
    if dtype is not None:
        t = t.to(dtype)
    return t.cuda()


def dev_u64(a):
    import torch
    return dev(np.ascontiguousarray(a, dtype=np.uint64).view(np.int64), torch.int64)


def host_u64(t):
    return t.cpu().numpy().view(np.uint64)


def empty_dev(n, dtype):
    import torch
    return torch.zeros(max(int(n), 1), dtype=dtype, device="cuda")


def as_int_keys(kmers, key_words):
    """Python ints of a key array ((n,) or (n, 2) {lo, hi})."""
    if key_words == 1:
        return [int(x) for x in kmers]
    return [int(r[0]) | (int(r[1]) << 64) for r in kmers]


def assert_same_result(got, want, label=""):
    assert got.n_windows == want.n_windows, (label, got.n_windows, want.n_windows)
    assert got.n_distinct == want.n_distinct, (label, got.n_distinct, want.n_distinct)
    assert got.max_count == want.max_count, (label, got.max_count, want.max_count)
    assert got.key_words == want.key_words
    assert got.kmers.shape == want.kmers.shape, (label, got.kmers.shape, want.kmers.shape)
    assert np.array_equal(got.kmers, want.kmers), label
    assert np.array_equal(got.counts, want.counts), label
    assert np.array_equal(got.hist, want.hist), label


ACGT = np.frombuffer(b"ACGT", np.uint8)


def reads_of(template, n_reads, length, err, seed):
    """n_reads reads of `length` bases from either strand of a template, with
    substitutions at rate err; (ASCII bases, offsets)."""
    rng = np.random.default_rng(seed)
    start = rng.integers(0, len(template) - length + 1, n_reads)
    x = template[start[:, None] + np.arange(length)]
    flip = rng.random(n_reads) < 0.5
    x[flip] = 3 - x[flip, ::-1]
    hit = rng.random(x.shape, dtype=np.float32) < err
    x = np.where(hit, (x + rng.integers(1, 4, x.shape, dtype=np.uint8)) & 3, x)
    return ACGT[x].reshape(-1), np.arange(n_reads + 1, dtype=np.uint64) * np.uint64(length)


def join(*sets):
    at = np.cumsum([0] + [int(o[-1]) for _, o in sets])
    offs = [o[:-1] + np.uint64(a) for (_, o), a in zip(sets, at)] + [np.array([at[-1]], np.uint64)]
    return np.concatenate([r for r, _ in sets]), np.concatenate(offs)


def bases(n, seed):
    return np.random.default_rng(seed).integers(0, 4, n, dtype=np.uint8)


def amplicon(n_bases, seed, err=0.01):
    return reads_of(bases(400, seed), n_bases // 400, 400, err, seed + 1)


def low_score_mmer(rng, m, seed=0x9E3779B97F4A7C15):
    """The base codes of an m-mer whose score (the minimizers' hash) is the least
    of 200,000 random ones."""
    c = rng.integers(0, 4, size=(200_000, m), dtype=np.uint8)
    w = (np.uint64(1) << (2 * np.arange(m - 1, -1, -1)).astype(np.uint64))
    v = np.minimum((c.astype(np.uint64) * w).sum(1, dtype=np.uint64),
                   ((3 - c[:, ::-1]).astype(np.uint64) * w).sum(1, dtype=np.uint64))
    h = (v & np.uint64(0xFFFFFFFF)).astype(np.uint32) ^ (v >> np.uint64(32)).astype(np.uint32) ^ np.uint32(seed & 0xFFFFFFFF)
    for shift, mul in ((16, 0x85EBCA6B), (13, 0xC2B2AE35), (16, 1)):
        h ^= h >> np.uint32(shift)
        h = (h.astype(np.uint64) * np.uint64(mul) & np.uint64(0xFFFFFFFF)).astype(np.uint32)
    return c[int(np.argmin(h))]
