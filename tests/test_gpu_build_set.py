"""build_octree (two C calls) against the single entry points in order: every array identical, for both
key lengths, with and without a box, masses and a warm start, and when the leaf capacity is too small."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("levels", [21, 10])
@pytest.mark.parametrize("n,ncrit", [(1, 1), (1000, 16), (4096, 5000), (70001, 8), (3_000_000, 8)])
@pytest.mark.parametrize("boxed,masses,cap", [(False, True, 0), (True, False, 0), (True, True, 1)])
def test_build_octree_equals_single_calls(lib, levels, n, ncrit, boxed, masses, cap):
    rng = np.random.default_rng(n + levels)
    x, y, z = (torch.from_numpy(rng.random(n) ** k).cuda() for k in (1, 2, 3))
    m = torch.from_numpy(rng.random(n, dtype=np.float32)).cuda() if masses else None
    box = torch.tensor([0.0, 0.0, 0.0, 1.0], dtype=torch.float64, device="cuda") if boxed else None
    small = lib.OctreeBuffers.allocate(n, cap, "cuda", levels) if cap else None
    got = lib.build_octree(x, y, z, curve=1, ncrit=ncrit, box=box, masses=m, buffers=small, levels=levels)

    b = lib.OctreeBuffers.allocate(n, lib.leaf_capacity(n, ncrit), "cuda", levels)
    if box is None:
        lib.cstone_bbox(x, y, z, b.box, b.ws)
        box = b.box
    if masses:
        records = torch.empty(lib.records_size(n), dtype=torch.uint8, device="cuda")
        lib.cstone_keys_records(x, y, z, m, box, 1, b.keys, records, lib.Workspace("cuda"), None, levels)
    else:
        lib.cstone_keys(x, y, z, box, 1, b.keys, None, levels)
    lib.cstone_sort(b.keys, b.sorted_keys, b.perm, b.ws, None, levels)
    nl, iters = lib.cstone_build_leaves(b.sorted_keys, ncrit, b.leaves, b.counts, b.offsets, 0, 64, b.ws, None, levels)
    t = b.tree_buffers(nl)
    nn = lib.n_nodes(nl)
    lib.cstone_link_tree(b.leaves, nl, t["NK"], t["CO"], t["LO"], t["leaf_to_node"], t["parent"], b.ws, None, levels)
    lib.cstone_upsweep_counts(b.counts, nl, t["leaf_to_node"], t["CO"], t["LO"], t["counts"], b.ws, None, levels)
    assert (got["n_leaves"], got["iters"]) == (nl, iters)
    want = {"keys": b.keys, "sorted_keys": b.sorted_keys, "perm": b.perm, "leaves": b.leaves[: nl + 1],
            "NK": t["NK"][:nn], "CO": t["CO"][:nn], "LO": t["LO"], "node_counts": t["counts"][:nn],
            "leaf_to_node": t["leaf_to_node"][:nl]}
    if masses:
        want["mass"] = torch.empty(nn, dtype=torch.float32, device="cuda")
        want["com"] = torch.empty(3 * nn, dtype=torch.float64, device="cuda")
        want["quad"] = torch.empty(6 * nn, dtype=torch.float32, device="cuda")
        lib.cstone_upsweep_multipoles_records(records, b.perm, n, b.offsets, nl, t["leaf_to_node"], t["CO"], t["LO"],
                                              box, want["mass"], want["com"], want["quad"], b.ws, None, levels)
    for k in want:
        assert torch.equal(got[k].reshape(-1), want[k].reshape(-1)), k

    warm = lib.build_octree(x, y, z, curve=1, ncrit=ncrit, box=box, levels=levels, warm_leaves=got["leaves"].clone())
    assert warm["n_leaves"] == nl
    assert torch.equal(warm["leaves"], want["leaves"]) and torch.equal(warm["NK"], want["NK"])


@pytest.mark.parametrize("levels", [21, 10])
def test_masses_of_no_particles(lib, levels):
    """A build of no particles with masses clears the error word of the records' workspace, as any other."""
    none = torch.empty(0, dtype=torch.float64, device="cuda")
    b = lib.OctreeBuffers.allocate(0, 64, "cuda", levels)
    b.records = torch.empty(lib.records_size(0), dtype=torch.uint8, device="cuda")
    b.rws = lib.Workspace("cuda")
    b.rws.get(256).fill_(255)
    got = lib.build_octree(none, none, none, masses=none.float(), buffers=b, levels=levels)
    assert b.rws.status() == lib.OK
    assert got["n_leaves"] == 1 and got["node_counts"].tolist() == [0]
    assert got["mass"].tolist() == [0.0] and not got["quad"].any()
