"""Sorts whose parts are hard for the last step: keys in fewer bits than it has bins (the values decide, over the
bits in which they differ)."""
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
