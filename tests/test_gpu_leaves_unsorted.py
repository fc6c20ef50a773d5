"""Cold leaf builds of keys that are not sorted: the call reports an error instead of leaves, and neither reads
past the list of leaf starts (which such keys can overfill) nor leaves a half-written array behind."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _kinds(levels):
    end, rng = 1 << (3 * levels), np.random.default_rng(levels)
    octant = end // 8
    # nearly every key opens a leaf of a nine-element array
    yield "alternating octants", np.where(np.arange(5000) % 2, 5 * octant, 2 * octant).astype(np.uint64), 1
    yield "shuffled", rng.integers(0, end, 5000, dtype=np.uint64), 16
    swapped = np.sort(rng.integers(0, end, 5000, dtype=np.uint64))
    swapped[[700, 3000]] = swapped[[3000, 700]]
    yield "two keys exchanged", swapped, 16


def _device(k, levels):
    return torch.from_numpy(k.view(np.int64) if levels == 21 else k.astype(np.uint32).view(np.int32)).cuda()


@pytest.mark.parametrize("levels", [21, 10])
@pytest.mark.parametrize("cap", [15, 20_000])
def test_single_set(lib, levels, cap):
    for name, k, ncrit in _kinds(levels):
        d = _device(k, levels)
        K = torch.zeros(cap + 1, dtype=d.dtype, device="cuda")
        N, off = (torch.zeros(m, dtype=torch.int32, device="cuda") for m in (cap, cap + 1))
        with pytest.raises(lib.CstoneError) as e:
            lib.cstone_build_leaves(d, ncrit, K, N, off, levels=levels)
        assert e.value.status == lib.ERR_INVALID_ARG, name
        assert not K.any() and not N.any() and not off.any(), name


@pytest.mark.parametrize("cap", [40, 20_000])
def test_batched_sets(lib, cap):
    for name, k, ncrit in _kinds(21):
        P = np.concatenate([np.sort(k)[:50], k, np.sort(k)[-50:]])
        so = torch.tensor([0, 50, 50 + k.size, P.size], device="cuda")
        E, N, off = (torch.zeros(cap, dtype=t, device="cuda") for t in (torch.int64, torch.int32, torch.int32))
        eo = torch.zeros(4, dtype=torch.int64, device="cuda")
        with pytest.raises(lib.CstoneError) as e:
            lib.cstone_build_leaves_batched(_device(P, 21), so, ncrit, E, eo, N, off)
        assert e.value.status == lib.ERR_INVALID_ARG, name
        ws = lib.Workspace()
        lib.cstone_build_leaves_batched_async(_device(P, 21), so, ncrit, E, eo, N, off, ws=ws)
        with pytest.raises(lib.CstoneError) as e:
            lib.cstone_leaves_result(ws, cap)
        assert e.value.status == lib.ERR_INVALID_ARG, name
        # without a host to report to, every set gets its root array
        assert eo.tolist() == [0, 2, 4, 6], name
        assert E[:6].tolist() == 3 * [0, -(1 << 63)] and N[:6].tolist() == [50, 0, k.size, 0, 50, 0], name
