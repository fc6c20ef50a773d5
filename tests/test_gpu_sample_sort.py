"""The sample sort behind cstone_sort and cstone_sort_segmented at the sizes where its path changes
(digit passes up to 1024 keys, one block up to 2560, one round of splitting up to 786,432, two above)
and on key sets that are hard to split, bit for bit against a stable sort."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SMALL, TARGET, PARTS = 2560, 1536, 512  # pairs sorted by one block, mean part, most parts of a bucket


def _kinds(rng, n):
    top = np.uint64((1 << 63) - 1)
    yield "uniform", rng.integers(0, 1 << 63, n, dtype=np.uint64)
    c = rng.integers(0, 1 << 63, 9, dtype=np.uint64)
    tight = (c[rng.integers(0, 9, n)] + rng.integers(0, 1 << 14, n, dtype=np.uint64)) & top
    yield "tight clumps beside sparse keys", np.where(rng.random(n) < 0.5, tight, rng.integers(0, 1 << 63, n, dtype=np.uint64))
    yield "few distinct", rng.integers(0, 1 << 63, 3, dtype=np.uint64)[rng.integers(0, 3, n)]
    yield "fifty of each", rng.integers(0, max(1, n // 50), n, dtype=np.uint64) << np.uint64(13)
    yield "all equal", np.full(n, (1 << 62) + 5, np.uint64)
    yield "descending", np.sort(rng.integers(0, 1 << 63, n, dtype=np.uint64))[::-1].copy()


def _check(lib, k, alias=False, levels=21):
    dt = (np.uint64, np.int64) if levels == 21 else (np.uint32, np.int32)
    kin = torch.from_numpy(k.astype(dt[0]).view(dt[1])).cuda()
    kout = kin if alias else torch.empty_like(kin)
    perm = torch.empty(k.size, dtype=torch.int32, device="cuda")
    lib.cstone_sort(kin, kout, perm, lib.Workspace(), levels=levels)
    want = np.argsort(k, kind="stable")
    assert np.array_equal(perm.cpu().numpy().view(np.uint32), want.astype(np.uint32))
    assert np.array_equal(kout.cpu().numpy().view(dt[0]), k.astype(dt[0])[want])


@pytest.mark.parametrize("n", [1024, 1025, SMALL, SMALL + 1, 4 * SMALL + 11, TARGET * PARTS, TARGET * PARTS + 1, 2_500_003])
def test_sizes_and_kinds(lib, n):
    for _, k in _kinds(np.random.default_rng(n), n):
        _check(lib, k)


@pytest.mark.parametrize("n", [1, 900, SMALL + 1, 1_000_003])
def test_30_bit_keys(lib, n):
    rng = np.random.default_rng(n)
    for k in (rng.integers(0, 1 << 30, n), rng.integers(0, max(1, n // 3000), n) << 7):
        _check(lib, k.astype(np.uint64), levels=10)


@pytest.mark.parametrize("n", [1000, SMALL, 50_001, 900_001])
def test_output_may_be_the_input(lib, n):
    _check(lib, np.random.default_rng(n).integers(0, 1 << 40, n, dtype=np.uint64), alias=True)


def test_part_that_the_sample_missed(lib):
    """Every sampled key is small and all others are large: the last part holds nearly the whole set and
    is sorted by merges."""
    n = 100_001
    np_parts = -(-n // TARGET)
    ns = np_parts * 32
    e = np.arange(ns, dtype=np.uint64)
    lo, hi = e * np.uint64(n) // np.uint64(ns), (e + np.uint64(1)) * np.uint64(n) // np.uint64(ns)
    with np.errstate(over="ignore"):
        x = e.astype(np.uint32)  # the sample's integer hash of e (the set starts at 0)
        x = (x ^ np.uint32(61)) ^ (x >> np.uint32(16))
        x = x * np.uint32(9)
        x = x ^ (x >> np.uint32(4))
        x = x * np.uint32(0x27D4EB2D)
        x = x ^ (x >> np.uint32(15))
    pos = lo + x.astype(np.uint64) % (hi - lo)
    k = np.random.default_rng(1).integers(1 << 40, 1 << 63, n, dtype=np.uint64)
    k[pos.astype(np.int64)] = e
    _check(lib, k)


def test_segments_of_all_sizes(lib):
    rng = np.random.default_rng(8)
    sizes = np.array([0, 1, 31, SMALL, SMALL + 1, 0, 20_000, TARGET * PARTS + 5, 777, 100_000, 0])
    off = np.concatenate([[0], np.cumsum(sizes)])
    n = int(off[-1])
    for _, k in _kinds(rng, n):
        kin = torch.from_numpy(k.view(np.int64)).cuda()
        kout, perm = torch.empty_like(kin), torch.empty(n, dtype=torch.int32, device="cuda")
        lib.cstone_sort_segmented(kin, kout, perm, torch.from_numpy(off).cuda(), lib.Workspace())
        seg = np.repeat(np.arange(sizes.size), sizes)
        want = np.lexsort((np.arange(n), k, seg))
        assert np.array_equal(perm.cpu().numpy().view(np.uint32), want.astype(np.uint32))
        assert np.array_equal(kout.cpu().numpy().view(np.uint64), k[want])
