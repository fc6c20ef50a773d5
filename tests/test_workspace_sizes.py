"""A workspace sized for more items serves fewer: the size queries never fall as the count grows, across the
sizes where a step changes its tiles or its method. No GPU needed."""
import ctypes

import pytest

EDGES = (1024, 2560, 1536 * 512, 786_432, 1 << 18, 1 << 20, 1 << 22, 1 << 24, (1 << 24) + (1 << 23), 1 << 27)


@pytest.fixture(scope="module")
def clib():
    import paper_2307_06345_gb300 as cs
    cs.build()
    return cs.load()


QUERIES = {
    "sort_workspace_size": lambda f, n, out: f(n, out),
    "link_workspace_size": lambda f, n, out: f(n, out),
    "upsweep_workspace_size": lambda f, n, out: f(n, out),
    "leaves_workspace_size": lambda f, n, out: f(n, 4096, 64, out),
    "build_set_workspace_size": lambda f, n, out: f(n, 4096, 64, out),
    "build_tree_workspace_size": lambda f, n, out: f(n, 1, out),
    "link_batched_workspace_size": lambda f, n, out: f(n, 3, out),
    "sort_segmented_workspace_size": lambda f, n, out: f(n, 3, out),
    "leaves_batched_workspace_size": lambda f, n, out: f(n, 64, out),
}


@pytest.mark.parametrize("name", [p + q for q in QUERIES for p in ("cstone_", "cstone30_")
                                  if p == "cstone_" or "batched" not in q and "segmented" not in q])
def test_size_query_is_monotone(clib, name):
    call, f = QUERIES[name.split("_", 1)[1]], getattr(clib, name)
    sizes = sorted({max(e * k // 4 + d, 8) for e in EDGES for k in (1, 2, 3, 4) for d in (-7, -1, 0, 1, 7)})
    last = 0
    for n in sizes:
        out = ctypes.c_size_t()
        assert call(f, n, ctypes.byref(out)) == 0
        assert out.value >= last, n
        last = out.value


@pytest.mark.parametrize("elements", [64, 4096, 1 << 20])
def test_leaf_workspace_follows_the_capacity(clib, elements):
    """A batch's leaf workspace holds the loop's arrays for its elements (under 64 bytes each, and the passes'
    state), however many particles a batch may have."""
    out = ctypes.c_size_t()
    assert clib.cstone_leaves_batched_workspace_size(elements, 64, ctypes.byref(out)) == 0
    assert out.value <= 64 * elements + (1 << 16)
    assert clib.cstone_leaves_workspace_size(1 << 29, elements, 64, ctypes.byref(out)) == 0
    assert out.value <= 64 * elements + (1 << 16)
