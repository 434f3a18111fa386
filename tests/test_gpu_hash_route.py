"""Which jobs and packs are counted by hashing (hsk_debug_hash_stats): the tuned
parameters that concern the sorting path do not decide it."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_same_result, bases, reads_of

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
