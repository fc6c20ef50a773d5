"""Sorts whose parts are hard for the last step: keys in fewer bits than it has bins (the values decide, over the
bits in which they differ), and sets whose first sample misses nearly every key, so that the second round's parts
are larger than a block sorts at once and are merged in global memory."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _check(lib, k, levels=21, off=None):
    u, i = (np.uint64, np.int64) if levels == 21 else (np.uint32, np.int32)
    kin = torch.from_numpy(k.astype(u).view(i)).cuda()
    kout, perm = torch.empty_like(kin), torch.empty(k.size, dtype=torch.int32, device="cuda")
    if off is None:
        lib.cstone_sort(kin, kout, perm, lib.Workspace(), levels=levels)
        want = np.argsort(k, kind="stable")
    else:
        lib.cstone_sort_segmented(kin, kout, perm, torch.from_numpy(off).cuda(), lib.Workspace())
        want = np.lexsort((np.arange(k.size), k, np.repeat(np.arange(off.size - 1), np.diff(off))))
    assert np.array_equal(perm.cpu().numpy().view(np.uint32), want.astype(np.uint32))
    assert np.array_equal(kout.cpu().numpy().view(u), k.astype(u)[want])


@pytest.mark.parametrize("n", [1025, 2560, 2561, 60_001, 786_433, 2_000_003])
@pytest.mark.parametrize("values", [1, 2, 33, 1000])
def test_keys_of_few_bits(lib, n, values):
    rng = np.random.default_rng(n + values)
    k = rng.integers(0, values, n, dtype=np.uint64)
    _check(lib, k)
    _check(lib, k + np.uint64((1 << 62) - values // 2))
    _check(lib, k + np.uint64(77), levels=10)
    off = np.array([0, n // 3, n // 3 + 40, n - 3000 if n > 9000 else n // 2, n], np.int64)
    _check(lib, k, off=off)


@pytest.mark.parametrize("n", [2_000_003, 8_000_003])  # merges of chunks of 8192: none and one; one and two
def test_first_sample_misses_the_set(lib, n):
    full = -(-n // 1536)
    parts = max(min(int(np.sqrt(np.float32(full))) + 1, 256), min(-(-full // 384), 512))
    ns = parts * min(32, 8192 // parts)
    e = np.arange(ns, dtype=np.uint64)
    lo, hi = e * np.uint64(n) // np.uint64(ns), (e + np.uint64(1)) * np.uint64(n) // np.uint64(ns)
    with np.errstate(over="ignore"):
        x = e.astype(np.uint32)  # the sample's integer hash of e
        x = (x ^ np.uint32(61)) ^ (x >> np.uint32(16))
        x = x * np.uint32(9)
        x = x ^ (x >> np.uint32(4))
        x = x * np.uint32(0x27D4EB2D)
        x = x ^ (x >> np.uint32(15))
    k = np.random.default_rng(n).integers(1 << 40, 1 << 63, n, dtype=np.uint64)
    k[(lo + x.astype(np.uint64) % (hi - lo)).astype(np.int64)] = e
    _check(lib, k)
