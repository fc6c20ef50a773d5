"""The linked tree and the node counts that come with it, on both sides of the tile size's limit (2^18 leaves):
against the sum over the children that cstone_upsweep_counts makes, and a batch's sets against single builds."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _points(n, kind, seed):
    rng = np.random.default_rng(seed)
    if kind == "uniform":
        p = rng.random((3, n))
    elif kind == "tight":  # a deep chain of single children beside a few far particles
        p = 0.3 + 1e-7 * rng.standard_normal((3, n))
        p[:, :: max(n // 50, 1)] = rng.random((3, p[:, :: max(n // 50, 1)].shape[1]))
    else:  # half uniform, half in clumps
        p = rng.random((3, n))
        c = rng.random((3, 20))
        half = n // 2
        p[:, :half] = c[:, rng.integers(0, 20, half)] + 1e-3 * rng.standard_normal((3, half))
    return [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in np.clip(p, 0.0, 0.999999)]


@pytest.mark.parametrize("levels", [21, 10])
@pytest.mark.parametrize("n,ncrit,kind", [(2, 1, "uniform"), (9, 1, "uniform"), (1200, 1, "tight"), (5000, 1, "clumps"),
                                          (400_000, 1, "clumps"), (60_000, 1, "tight"), (2_500_000, 2, "uniform")])
def test_counts_of_the_linked_tree(lib, levels, n, ncrit, kind):
    x, y, z = _points(n, kind, n)
    t = lib.build_octree(x, y, z, curve=0, ncrit=ncrit, levels=levels)
    nl, nn = t["n_leaves"], t["NK"].numel()
    want = torch.full((nn,), -1, dtype=torch.int32, device="cuda")
    lib.cstone_upsweep_counts(t["leaf_counts"], nl, t["leaf_to_node"], t["CO"], t["LO"], want, None, None, levels)
    assert torch.equal(t["node_counts"], want) and int(want[0]) == n
    # children: the eight nodes from CO on carry the parent's key with one more digit
    inner = torch.nonzero(t["CO"] > 0).reshape(-1)
    assert inner.numel() == (nn - 1) // 8
    c = t["CO"][inner].long()
    for d in range(8):
        assert torch.equal(t["NK"][c + d], 8 * t["NK"][inner] + d)
    if nn > 1:
        assert torch.equal(t["parent"][: (nn - 1) // 8], inner.int())


@pytest.mark.parametrize("sizes,ncrit", [((700, 0, 1, 12_000, 9), 4), ((300_000, 5, 0, 150_001, 64, 1), 2)])
def test_batched_sets_equal_single_builds(lib, sizes, ncrit):
    parts = [_points(s, k, 7 + i) if s else [torch.empty(0, dtype=torch.float64, device="cuda")] * 3
             for i, (s, k) in enumerate(zip(sizes, ("clumps", "uniform", "tight", "uniform", "clumps", "uniform")))]
    x, y, z = (torch.cat([p[a] for p in parts]).contiguous() for a in range(3))
    off = torch.tensor(np.concatenate([[0], np.cumsum(sizes)]), dtype=torch.int64, device="cuda")
    box = torch.tensor([0.0, 0.0, 0.0, 1.0], dtype=torch.float64, device="cuda")
    boxes = box.repeat(len(sizes), 1).contiguous()
    out = lib.build_octrees_batched(x, y, z, off, curve=1, ncrit=ncrit, boxes=boxes)
    for s, n in enumerate(sizes):
        if n == 0:
            continue
        one = lib.build_octree(*parts[s], curve=1, ncrit=ncrit, box=box)
        a, b = out["node_offsets_host"][s], out["node_offsets_host"][s + 1]
        assert torch.equal(out["NK"][a:b], one["NK"])
        assert torch.equal(out["node_counts"][a:b], one["node_counts"])
        co = out["CO"][a:b]
        assert torch.equal(torch.where(co > 0, co - a, co), one["CO"])


@pytest.mark.parametrize("shift", [0, 1])
def test_batched_boxes_of_odd_ranges(lib, shift):
    """Sets that start and end at odd and even particles, from arrays on and off 16-byte boundaries."""
    sizes = [1, 1, 2, 3, 0, 4, 5, 8193, 8192, 1, 100_001]
    n = sum(sizes)
    rng = np.random.default_rng(3)
    xyz = [torch.from_numpy(rng.standard_normal(n + shift)).cuda()[shift:] for _ in range(3)]
    off = torch.tensor(np.concatenate([[0], np.cumsum(sizes)]), dtype=torch.int64, device="cuda")
    out = lib.build_octrees_batched(*xyz, off, curve=0, ncrit=32)
    for s, size in enumerate(sizes):
        a, b = int(off[s]), int(off[s + 1])
        lo = [float(c[a:b].min()) if size else 0.0 for c in xyz]
        side = max(float(c[a:b].max()) - v for c, v in zip(xyz, lo)) if size else 1.0
        want = lo + [side if side > 0.0 else 1.0]
        assert out["boxes"][s].tolist() == want, s
