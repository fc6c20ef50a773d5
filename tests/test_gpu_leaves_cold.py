"""The one-sweep cold build of the leaf array (cstone_build_leaves from the root) at the edges of its
tiles (2048 positions) and of its range of N_crit (up to 1024; the loop above), against the oracle's
f / g iteration: keys, counts, first particles, passes, and the capacity it asks for."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _keys(rng, n, kind, levels):
    end = 1 << (3 * levels)
    if kind == "uniform":
        k = rng.integers(0, end, n, dtype=np.uint64)
    elif kind == "clustered":
        c = rng.integers(0, end - (1 << 12), 5, dtype=np.uint64)
        k = np.where(rng.random(n) < 0.7, c[rng.integers(0, 5, n)] + rng.integers(0, 1 << 12, n, dtype=np.uint64),
                     rng.integers(0, end, n, dtype=np.uint64))
    elif kind == "corners":
        k = np.array([0, end - 1, end // 2, end // 2 - 1, 7], np.uint64)[rng.integers(0, 5, n)]
    else:
        k = np.full(n, end // 3, np.uint64)
    return np.sort(k)


def _build(lib, P, ncrit, cap, levels=21, max_iters=64):
    dt, t = ((np.int64, torch.int64), (np.int32, torch.int32))[levels == 10]
    d = torch.from_numpy(P.astype(np.uint64 if levels == 21 else np.uint32).view(dt)).cuda()
    K = torch.zeros(cap + 1, dtype=t, device="cuda")
    N = torch.zeros(cap, dtype=torch.int32, device="cuda")
    off = torch.zeros(cap + 1, dtype=torch.int32, device="cuda")
    nl, it = lib.cstone_build_leaves(d, ncrit, K, N, off, 0, max_iters, levels=levels)
    un = np.uint64 if levels == 21 else np.uint32
    return (K[: nl + 1].cpu().numpy().view(un).astype(np.uint64), N[:nl].cpu().numpy().view(np.uint32),
            off[: nl + 1].cpu().numpy().view(np.uint32), it)


@pytest.mark.parametrize("levels", [21, 10])
@pytest.mark.parametrize("ncrit", [0, 1, 3, 64, 1000, 1024, 1025])
def test_every_edge(lib, oracle, ncrit, levels):
    rng = np.random.default_rng(ncrit + levels)
    for n in (0, 1, 2, 2046, 2047, 2048, 2049, 4095, 4096, 9001):
        for kind in ("uniform", "clustered", "corners", "equal"):
            P = _keys(rng, n, kind, levels)
            K_ref, N_ref, it_ref = oracle.build_leaves(P, ncrit, levels=levels)
            K, N, off, it = _build(lib, P, ncrit, max(8, K_ref.size), levels)
            assert np.array_equal(K, K_ref) and np.array_equal(N, N_ref) and it == it_ref, (n, kind)
            assert np.array_equal(off, np.concatenate([[0], np.cumsum(N_ref)])), (n, kind)


@pytest.mark.parametrize("max_iters", [3, 64])
def test_capacity_and_passes(lib, oracle, max_iters):
    """A failed build says what the loop says: the leaves after the pass that did not fit, unless the
    passes end before it."""
    P = _keys(np.random.default_rng(2), 30_000, "uniform", 21)
    K, _, passes = oracle.build_leaves(P, 8)
    LO = oracle.link(K)["LO"].astype(np.int64)
    internal = (LO[2:] - LO[1:-1]) // 8
    after = 1 + 7 * np.cumsum(internal)  # leaves after pass 0, 1, ...
    for cap in (7, 60, 500, int(K.size) - 2):
        over = int(np.argmax(after > cap))
        with pytest.raises(lib.CstoneError) as e:
            _build(lib, P, 8, cap, max_iters=max_iters)
        if over < max_iters:
            assert e.value.status == lib.ERR_CAPACITY and e.value.required == after[over]
        else:
            assert e.value.status == lib.ERR_NOT_CONVERGED
    if max_iters < passes:
        with pytest.raises(lib.CstoneError) as e:
            _build(lib, P, 8, K.size, max_iters=max_iters)
        assert e.value.status == lib.ERR_NOT_CONVERGED


@pytest.mark.parametrize("sizes", [(0, 0), (0, 5, 0, 0, 4000, 1, 0), (2048, 2048), (2047, 1, 2048, 3, 0), tuple(range(60))])
@pytest.mark.parametrize("ncrit", [1, 16, 700])
def test_batched_sets(lib, oracle, sizes, ncrit):
    rng = np.random.default_rng(len(sizes))
    P = [_keys(rng, n, ("clustered", "uniform", "equal")[k % 3], 21) for k, n in enumerate(sizes)]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n, s = int(off[-1]), len(sizes)
    ref = [oracle.build_leaves(p, ncrit) for p in P]
    cap = sum(r[0].size for r in ref) + 3
    elements, counts, first = (torch.zeros(cap, dtype=dt, device="cuda") for dt in (torch.int64, torch.int32, torch.int32))
    eo = torch.zeros(s + 1, dtype=torch.int64, device="cuda")
    d = torch.from_numpy(np.concatenate(P).astype(np.uint64).view(np.int64)).cuda()
    ne, it = lib.cstone_build_leaves_batched(d, torch.from_numpy(off).cuda(), ncrit, elements, eo, counts, first)
    assert ne == cap - 3 and it == max(r[2] for r in ref)
    want = np.concatenate([[0], np.cumsum([r[0].size for r in ref])])
    assert np.array_equal(eo.cpu().numpy(), want)
    assert np.array_equal(elements[:ne].cpu().numpy().view(np.uint64), np.concatenate([r[0] for r in ref]))
    assert np.array_equal(counts[:ne].cpu().numpy(), np.concatenate([np.append(r[1], 0) for r in ref]))
    assert np.array_equal(first[:ne].cpu().numpy(),
                          np.concatenate([off[k] + np.concatenate([[0], np.cumsum(r[1])]) for k, r in enumerate(ref)]))


@pytest.mark.parametrize("room", [0, 1, 300])
def test_fewer_elements_than_tiles(lib, oracle, room):
    """Capacities below and above the number of tiles, for many particles in one cell."""
    n = 600_000
    tiles = n // 2048 + 1
    P = np.full(n, (1 << 63) // 3, np.uint64)
    K_ref, N_ref, it_ref = oracle.build_leaves(P, 64)
    assert K_ref.size < tiles
    cap = max(K_ref.size - 1, tiles - 2 + room)
    K, N, off, it = _build(lib, P, 64, cap)
    assert np.array_equal(K, K_ref) and np.array_equal(N, N_ref) and it == it_ref
    assert np.array_equal(off, np.concatenate([[0], np.cumsum(N_ref)]))
    eo = torch.zeros(3, dtype=torch.int64, device="cuda")
    d = torch.from_numpy(np.concatenate([P, P[:7]]).view(np.int64)).cuda()
    E, C = (torch.zeros(cap + 3, dtype=t, device="cuda") for t in (torch.int64, torch.int32))
    ne, it = lib.cstone_build_leaves_batched(d, torch.tensor([0, n, n + 7], device="cuda"), 64, E, eo, C)
    assert it == it_ref and eo.tolist() == [0, K_ref.size, K_ref.size + 2]
    assert np.array_equal(E[: K_ref.size].cpu().numpy().view(np.uint64), K_ref) and C[ne - 2].item() == 7


SWEEP, LOOP = 4, 1  # launches of a cold build


@pytest.mark.parametrize("levels,n,ncrit,launches", [
    (21, 1 << 23, 1024, SWEEP), (21, (1 << 23) + 1, 1024, LOOP), (21, (1 << 23) + 1, 32, SWEEP),
    (10, 1 << 22, 1024, SWEEP), (10, (1 << 22) + 1, 1024, LOOP),
    (21, 500, 500, LOOP), (21, 501, 500, SWEEP), (10, 500, 500, LOOP), (10, 501, 500, SWEEP)])
def test_both_sides_of_the_size_rule(lib, oracle, levels, n, ncrit, launches):
    P = _keys(np.random.default_rng(n), n, "clustered", levels)
    K_ref, N_ref, it_ref = oracle.build_leaves(P, ncrit, levels=levels)
    before = lib.cstone_kernel_launches()
    K, N, off, it = _build(lib, P, ncrit, max(K_ref.size, n // 2048 + 1), levels)
    assert lib.cstone_kernel_launches() - before == launches
    assert np.array_equal(K, K_ref) and np.array_equal(N, N_ref) and it == it_ref


@pytest.mark.parametrize("size,launches", [(40, LOOP), (41, SWEEP)])
def test_sets_of_single_leaves(lib, size, launches):
    rng = np.random.default_rng(size)
    s, ncrit = 300, 40
    P = np.concatenate([_keys(rng, size, "uniform", 21) for _ in range(s)])
    off = torch.arange(s + 1, device="cuda") * size
    E, C = (torch.zeros(9 * s, dtype=t, device="cuda") for t in (torch.int64, torch.int32))
    eo = torch.zeros(s + 1, dtype=torch.int64, device="cuda")
    before = lib.cstone_kernel_launches()
    ne, _ = lib.cstone_build_leaves_batched(torch.from_numpy(P.view(np.int64)).cuda(), off, ncrit, E, eo, C)
    assert lib.cstone_kernel_launches() - before == launches
    per = 2 if size <= ncrit else 9
    assert ne == per * s and eo.tolist() == [per * k for k in range(s + 1)]
    counts = C[:ne].view(s, per)
    assert (counts.sum(1) == size).all() and not counts[:, -1].any() and (counts <= ncrit).all()
