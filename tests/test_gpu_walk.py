"""The S2 walk at the edges of its decomposition: window lengths around the
powers of two and past a lane's 32 scores, m-mers around 16 bases, runs longer
than a record, and data that ends inside a tile."""
import numpy as np
import pytest

import datagen
import oracle
from gpu_util import assert_same_result, dev, dev_u64, empty_dev, host_u64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [4, 16, 17, 32])
@pytest.mark.parametrize("w", [1, 2, 3, 8, 15, 16, 17, 31, 32, 33, 34, 35, 48, 61])
def test_window_minima(hsk, m, w):
    k = m + w - 1
    if k > 64:
        pytest.skip("k > 64")
    import torch
    reads, offs = datagen.random_reads(100 * m + w, 40, 0, 900, p_invalid=0.003, invalid=b"N")
    tail = np.frombuffer(b"ACGT" * 30 + b"A" * 300 + b"CA" * 90, np.uint8)
    reads = np.concatenate([reads, tail])
    offs = np.concatenate([offs, [offs[-1] + tail.size]]).astype(np.uint64)
    n = reads.size
    pos, key, mh, _ = oracle.windows(reads, offs, k, m)
    with hsk.Context() as ctx:
        valid, keys, mins = empty_dev(n, torch.uint8), empty_dev(2 * n, torch.int64), empty_dev(n, torch.int64)
        ctx.stage_windows(dev(reads), dev_u64(offs), k, m, valid, keys, mins)
        gv = np.nonzero(valid.cpu().numpy()[:n])[0]
        assert np.array_equal(gv.astype(np.uint64), pos)
        assert np.array_equal(host_u64(keys)[: 2 * n].reshape(n, 2)[gv], key)
        assert np.array_equal(host_u64(mins)[:n][gv], mh)


@pytest.mark.parametrize("n", [1023, 1024, 1025, 2047, 3000])
def test_long_runs_and_tile_ends(hsk, n):
    """One minimizer over whole tiles (more than a record's k-mers a run)."""
    strs = ["A" * n, "AC" * (n // 2), "A" * 40 + "N" + "A" * (n - 41)]
    offs = np.zeros(len(strs) + 1, np.uint64)
    offs[1:] = np.cumsum([len(s) for s in strs])
    reads = np.frombuffer("".join(strs).encode(), np.uint8).copy()
    for k, m in ((31, 17), (55, 21)):
        want = oracle.count(reads, offs, k, 1, 1 << 20)
        with hsk.Context() as ctx:
            assert_same_result(ctx.count(reads, offs, k, m, 1, 1 << 20), want, f"n={n} k={k}")
