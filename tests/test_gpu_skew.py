"""Reads crowded around a few minimizers (deep amplicons, low complexity):
their fine partitions hold far more records or distinct k-mers than an SM's
table, next to partitions that hold few.  Every result is the CPU oracle's."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same_result, bases, join, reads_of

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
