"""Output order (S6) of the on-chip range sort at its capacities: ranges that
share their top digit or top two digits and hold up to, just over and far over
one on-chip sort, and few pairs in many ranges."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same_result

pytestmark = pytest.mark.gpu


def _reads(k, n_same, prefix, n_random, seed):
    """n_same reads of one k-mer starting with `prefix`, n_random reads of 1000 bases."""
    rng = np.random.default_rng(seed)
    acgt = np.frombuffer(b"ACGT", np.uint8)
    same = acgt[rng.integers(0, 4, size=(n_same, k))]
    same[:, : len(prefix)] = np.frombuffer(prefix, np.uint8)
    rest = acgt[rng.integers(0, 4, size=(n_random, 1000))]
    lens = np.concatenate([np.full(n_same, k), np.full(n_random, 1000)])
    offs = np.zeros(lens.size + 1, np.uint64)
    offs[1:] = np.cumsum(lens)
    return np.concatenate([same.reshape(-1), rest.reshape(-1)]), offs


@pytest.mark.parametrize("k,m", [(12, 9), (31, 17), (55, 21)])
@pytest.mark.parametrize("n_same,prefix", [(0, b"A"), (4000, b"AAAA"), (5000, b"AAAACCC"), (4096, b"AAAAAAAA"),
                                           (4200, b"AAAAAAAA"), (6300, b"AAAAAAAA"), (8100, b"AAAAAAAA"),
                                           (9000, b"AAAAAAAA"), (20000, b"AAAAAAAAAA")])
def test_ranges_at_the_capacity(hsk, k, m, n_same, prefix):
    if k == 12 and n_same > 4000:
        pytest.skip("12-mers with that prefix are few")
    reads, offs = _reads(k, n_same, prefix, 120, n_same + k)
    want = oracle.count(reads, offs, k, 1, 1 << 20)
    with hsk.Context() as ctx:
        for _ in range(2):
            assert_same_result(ctx.count(reads, offs, k, m, 1, 1 << 20), want, f"k={k} {n_same} {prefix}")


@pytest.mark.parametrize("k,m,n_random", [(31, 17, 900), (31, 17, 2600), (55, 21, 1700)])
def test_second_digit_pass_and_groups(hsk, k, m, n_random):
    """More pairs than one on-chip sort per top digit: groups of sub-ranges."""
    reads, offs = _reads(k, 1000, b"ACG", n_random, n_random)
    want = oracle.count(reads, offs, k, 1, 1 << 20)
    with hsk.Context() as ctx:
        assert_same_result(ctx.count(reads, offs, k, m, 1, 1 << 20), want, f"k={k}")
