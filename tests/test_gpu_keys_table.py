"""Hilbert keys on both sides of 2^22 particles, where the table of two levels gives way to the one of three (for
30-bit keys it reaches two levels too far, which the key drops), against the oracle: single sets with aligned and
odd arrays, with multipole records, and batches whose tiles lie in several sets."""
import numpy as np
import pytest
import torch

from _gpu_util import dev, u32, u64

pytestmark = pytest.mark.gpu

EDGE = 1 << 22


@pytest.fixture(scope="module")
def particles(oracle):
    from paper_2307_06345_gb300 import workloads as w
    x, y, z = w.plummer(EDGE + 1, 77)
    box = oracle.bounding_cube(x, y, z)
    return (x, y, z), box, {lv: oracle.keys(x, y, z, box, 1, levels=lv) for lv in (21, 10)}


def _shifted(a, shift):
    t = torch.empty(a.numel() + shift, dtype=a.dtype, device="cuda")[shift:]
    return t.copy_(a)


@pytest.mark.parametrize("levels", [21, 10])
@pytest.mark.parametrize("n", [EDGE - 1, EDGE, EDGE + 1])
def test_single_set(lib, particles, levels, n):
    pos, box, want = particles
    dt, host = (torch.int64, u64) if levels == 21 else (torch.int32, u32)
    for shift in (0, 1):  # 16-byte accesses, and arrays that do not allow them
        p = [_shifted(dev(c[:n]), shift) for c in pos]
        k = torch.empty(n + shift, dtype=dt, device="cuda")[shift:]
        lib.cstone_keys(*p, dev(box), lib.HILBERT, k, levels=levels)
        assert np.array_equal(host(k).astype(np.uint64), want[levels][:n]), shift
        k.zero_()
        rec, ws = torch.empty(lib.records_size(n), dtype=torch.uint8, device="cuda"), lib.Workspace()
        lib.cstone_keys_records(*p, torch.ones(n, device="cuda"), dev(box), lib.HILBERT, k, rec, ws, levels=levels)
        assert ws.status() == lib.OK
        assert np.array_equal(host(k).astype(np.uint64), want[levels][:n]), shift


@pytest.mark.parametrize("n", [EDGE - 1, EDGE + 1])
def test_batch_of_straddling_sets(lib, oracle, particles, n):
    pos, box, want = particles
    # large sets, sets smaller than a tile of 1024, empty ones; every third in a box of its own
    sizes = [1_500_001, 5, 0, 1023, 700_333, 1, 1, 0, 900_000, 2047, 513]
    sizes.append(n - sum(sizes))
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    boxes = np.array([box if s % 3 else box * np.array([1, 1, 1, 1.5]) for s in range(len(sizes))])
    k = torch.empty(n, dtype=torch.int64, device="cuda")
    lib.cstone_keys_batched(*(dev(c[:n]) for c in pos), dev(off), dev(boxes), lib.HILBERT, k, lib.Workspace())
    got = u64(k)
    for s, size in enumerate(sizes):
        a, b = off[s], off[s + 1]
        ref = want[21][a:b] if s % 3 else oracle.keys(*(c[a:b] for c in pos), boxes[s], 1)
        assert np.array_equal(got[a:b], ref), s
