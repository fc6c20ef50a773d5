"""One focused pass around the number of focus tiles (eight) up to which every lane takes its own distances, from
an empty focus on, against the oracle's decision, scan and rebalance."""
import numpy as np
import pytest
import torch

from _gpu_util import dev, u32, u64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels", [21, 10])
@pytest.mark.parametrize("curve", [0, 1])
def test_pass_with_a_few_tiles(lib, oracle, levels, curve):
    from paper_2307_06345_gb300 import workloads as w
    x, y, z = w.clumps(30_000, 5, n_clumps=25)
    P, _ = oracle.sort(oracle.keys(x, y, z, oracle.bounding_cube(x, y, z), curve, levels=levels))
    K = oracle.canonical_leaves(P, 8, levels=levels)
    nl = K.size - 1
    N = oracle.histogram(P, K)
    kd = dev(K if levels == 21 else K.astype(np.uint32))
    unit = (1 << (3 * levels)) >> 9  # a node of level 3
    seen = set()
    # ranges of such nodes that start and end inside their parents
    for a, b in [(0, 0), (9, 10), (10, 12), (13, 18), (11, 17), (9, 16), (9, 17), (9, 18), (9, 20), (9, 72), (3, 509)]:
        f = (a * unit, b * unit)
        tiles = len(oracle.focus_tiles(*f, levels=levels)) if b > a else 0
        seen.add(tiles)
        for theta, ncrit in ((0.35, 4), (1.2, 32)):
            out = torch.empty(8 * nl + 2, dtype=torch.int64 if levels == 21 else torch.int32, device="cuda")
            nl2, changed = lib.cstone_rebalance_focus(kd, dev(N), nl, ncrit, *f, theta, curve, out, lib.Workspace(),
                                                      levels=levels)
            O = oracle.focus_decision(K, N, ncrit, *f, theta, curve, levels=levels)
            K2 = oracle.rebalance(K, O, oracle.exclusive_scan(O), levels=levels)
            got = u64(out) if levels == 21 else u32(out).astype(np.uint64)
            assert nl2 == K2.size - 1 and changed == bool((O[:nl] != 1).any()), (f, theta)
            assert np.array_equal(got[: nl2 + 1], K2), (f, theta)
    assert {0, 1, 2, 7, 8, 9} <= seen, seen
