"""S1's 16-byte units (k_encode.cu) against the oracle: every byte value, ends
inside a unit, and inputs that start off a 16-byte boundary."""
import numpy as np
import pytest

import oracle
from gpu_util import dev, dev_u64, empty_dev, host_u64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [0, 1, 8, 15])
@pytest.mark.parametrize("n", [1, 15, 16, 17, 31, 33, 63, 65, 1023, 4096, 4111])
def test_ragged_ends_and_unaligned_starts(hsk, n, shift):
    import torch
    rng = np.random.default_rng(n + shift)
    raw = rng.choice(np.frombuffer(b"ACGT", np.uint8), n + shift)
    other = rng.random(n + shift) < 0.1
    raw[other] = rng.integers(0, 256, int(other.sum()), dtype=np.uint8)
    if n >= 1023:
        raw[shift:shift + 256] = np.arange(256, dtype=np.uint8)
    reads = raw[shift:].copy()
    code, inv = oracle.encode(reads)
    with hsk.Context() as ctx:
        pk = empty_dev((n + 31) // 32 + 4, torch.int64)
        iv = empty_dev((n + 63) // 64 + 4, torch.int64)
        st = empty_dev((n + 63) // 64 + 4, torch.int64)
        ctx.stage_encode(dev(raw)[shift:], dev_u64(np.array([0, n], np.uint64)), pk, iv, st)
        pk, iv = host_u64(pk), host_u64(iv)
    g = np.arange(n)
    assert np.array_equal(((pk[g // 32] >> (62 - 2 * (g % 32)).astype(np.uint64)) & np.uint64(3)).astype(np.uint8), code)
    assert np.array_equal(((iv[g // 64] >> (63 - g % 64).astype(np.uint64)) & np.uint64(1)).astype(np.uint8), inv)
