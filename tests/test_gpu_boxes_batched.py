"""Bounding cubes of batches where their kernel changes its loads: sets of two particles per thread (8192), odd
first and last particles, and arrays that are not aligned for 16-byte loads, against the oracle."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

SIZES = (0, 1, 2, 8191, 8192, 8193, 8194, 0, 8195, 1, 20_001, 12_288, 3)


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("rotate", range(3))
def test_sets_around_the_pairs(lib, oracle, shift, rotate):
    sizes = SIZES[rotate:] + SIZES[:rotate]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    rng = np.random.default_rng(rotate)
    # the extremes lie at the ends of the sets, where a pair could be left out
    c = rng.normal(size=(3, off[-1]))
    for s, n in enumerate(sizes):
        for d in range(3 if n else 0):
            c[d, off[s] if d % 2 else off[s + 1] - 1] = rng.choice([-9.0, 9.0]) + d
    held = [torch.from_numpy(np.concatenate([np.zeros(shift), v])).cuda()[shift:] for v in c]
    boxes = torch.empty((len(sizes), 4), dtype=torch.float64, device="cuda")
    lib.cstone_bbox_batched(*held, torch.from_numpy(off).cuda(), boxes)
    got = boxes.cpu().numpy()
    for s, n in enumerate(sizes):
        part = [np.ascontiguousarray(v[off[s]:off[s + 1]]) for v in c]
        want = oracle.bounding_cube(*part) if n else np.array([0.0, 0.0, 0.0, 1.0])
        assert np.array_equal(got[s], want), (s, n)
