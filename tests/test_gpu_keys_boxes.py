"""Keys of boxes and coordinates off the common path, against the oracle: boxes with one axis or all far from
the origin (the shared fixed-point frame does not hold, an axis' own may), particles outside the box, on the
borders of cells, and at the extremes of the format."""
import numpy as np
import pytest
import torch

from _gpu_util import dev, u32, u64

pytestmark = pytest.mark.gpu

BOXES = {  # corner, side
    "unit": ((0.0, 0.0, 0.0), 1.0),
    "one axis far": ((0.0, 0.0, 1e6), 1.0),
    "two axes far": ((-3e7, 0.25, 1e6), 1.0),
    "all far": ((1e9, -1e9, 1e9), 1.0),
    "beyond any bound": ((1e15, 0.0, -1.0), 1.0),
    "edge of the bound": ((float(1 << 13), 0.0, float(-(1 << 14))), 1.0),
    "small and off": ((30.0, 1e-3, -7.0), 1e-5),
    "tiny": ((0.0, -1e-290, 1e-291), 1e-290),
    "huge": ((-1e300, 1e299, 0.0), 3e300),
}


def _particles(rng, n, corner, side):
    c = []
    for lo in corner:
        x = lo + side * rng.random(n)
        k = n // 8
        x[:k] = lo + side * (rng.integers(0, (1 << 21) + 1, k) / (1 << 21))  # cell borders
        x[k:2 * k] = lo + side * rng.uniform(-3.0, 4.0, k)  # in and around the box
        x[2 * k:2 * k + 8] = [np.inf, -np.inf, 0.0, -0.0, 5e-324, -5e-324, 1.7e308, -1.7e308]
        c.append(rng.permutation(x))
    return c


@pytest.mark.parametrize("name", BOXES)
@pytest.mark.parametrize("levels", [21, 10])
def test_single_set(lib, oracle, name, levels):
    corner, side = BOXES[name]
    box = np.array([*corner, side])
    for n in (1, 33, 40_001):
        x, y, z = _particles(np.random.default_rng(n), max(n, 64), corner, side)
        x, y, z = x[:n], y[:n], z[:n]
        for curve in (lib.MORTON, lib.HILBERT):
            k = torch.empty(n, dtype=torch.int64 if levels == 21 else torch.int32, device="cuda")
            lib.cstone_keys(dev(x), dev(y), dev(z), dev(box), curve, k, levels=levels)
            got = u64(k) if levels == 21 else u32(k).astype(np.uint64)
            assert np.array_equal(got, oracle.keys(x, y, z, box, curve, levels=levels)), (n, curve)


# sets of a tile of 1024 particles on average or more, and of fewer: looked up by tile, and by particle
@pytest.mark.parametrize("sizes", [(5, 1023, 0, 1024, 3000, 1, 2, 700, 4097), (5, 1023, 0, 1024, 2000, 1, 2, 64, 1100)])
@pytest.mark.parametrize("curve", [0, 1])
def test_sets_with_boxes_of_their_own(lib, oracle, curve, sizes):
    rng = np.random.default_rng(curve)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    parts = [[c[:n] for c in _particles(rng, max(n, 64), *BOXES[b])] for n, b in zip(sizes, BOXES)]
    x, y, z = (np.concatenate([p[d] for p in parts]) for d in range(3))
    boxes = np.array([[*BOXES[b][0], BOXES[b][1]] for b in BOXES])
    k = torch.empty(x.size, dtype=torch.int64, device="cuda")
    lib.cstone_keys_batched(dev(x), dev(y), dev(z), dev(off), dev(boxes), curve, k, lib.Workspace())
    want = np.concatenate([oracle.keys(*p, b, curve) for p, b in zip(parts, boxes) if p[0].size])
    assert np.array_equal(u64(k), want)


@pytest.mark.parametrize("name", ["unit", "one axis far", "small and off"])
def test_records_take_the_same_keys(lib, oracle, name):
    corner, side = BOXES[name]
    box, n = np.array([*corner, side]), 10_007
    rng = np.random.default_rng(3)
    x, y, z = (lo + side * rng.random(n) for lo in corner)
    k = torch.empty(n, dtype=torch.int64, device="cuda")
    rec, ws = torch.empty(lib.records_size(n), dtype=torch.uint8, device="cuda"), lib.Workspace()
    lib.cstone_keys_records(dev(x), dev(y), dev(z), torch.ones(n, device="cuda"), dev(box), 1, k, rec, ws)
    assert ws.status() == lib.OK
    assert np.array_equal(u64(k), oracle.keys(x, y, z, box, 1))
    # the fixed-point coordinates: x * 2^F truncated, F the widest frame of the box
    big = max(abs(v) for v in (min(corner), max(corner), max(corner) + 2 * side))
    F = 61 - int(np.floor(np.log2(big))) - 1
    got = rec.view(torch.int64).view(-1, 4)[:n, :3].cpu().numpy()
    want = [[int(v * 2.0 ** F) for v in p] for p in zip(x, y, z)]
    assert np.array_equal(got, np.array(want, dtype=np.int64))
