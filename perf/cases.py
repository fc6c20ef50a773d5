"""The work this framework does for its users, as cases that can be timed and compared: whole octree
builds from the smallest to the benchmark's size, batched builds of many independent sets, warm time
steps of several runs, the focused tree, and the multipoles of a tree that is already there. Every
case goes through the package's public entry points on inputs resident on the GPU.

``listed()`` are fixed cases, ``draw(rng)`` gives more of the same ranges; ``prepare`` makes a case's
inputs and the buffers a user's program keeps, ``run`` is one pass, ``work`` its least traffic and
arithmetic, ``exact`` its floating outputs in 64 bits from plain torch.

A case's ``model`` fixes where its matter is, so that the trees of all its inputs have the same size;
the seed draws the order of the particles, the axes' order, the unit of length and the masses.
"""
import math
import random

import torch

import paper_2307_06345_gb300 as cs

CURVES = {"morton": cs.MORTON, "hilbert": cs.HILBERT}


def listed():
    return [
        # a small N-body model rebuilt every step, with its masses: launches and latency
        {"name": "build_20k", "kind": "build", "model": 1, "n": 20_000, "dist": "plummer",
         "curve": "hilbert", "ncrit": 16, "levels": 21, "masses": True, "unit_box": False},
        # a neighbour-search grid of a small simulation box whose frame is known, no masses
        {"name": "build_64k_uniform", "kind": "build", "model": 2, "n": 65_536, "dist": "uniform",
         "curve": "morton", "ncrit": 64, "levels": 21, "masses": False, "unit_box": True},
        # the paper's Table 1 workload at its smallest size
        {"name": "build_1m_gaussian", "kind": "build", "model": 3, "n": 1 << 20, "dist": "gaussian", "curve": "hilbert",
         "ncrit": 64, "levels": 21, "masses": False, "unit_box": False},
        # one galaxy of ordinary size (single-GPU production run of a hydrodynamics code: no masses)
        {"name": "build_32m_plummer", "kind": "build", "model": 4, "n": 1 << 25, "dist": "plummer", "curve": "hilbert",
         "ncrit": 64, "levels": 21, "masses": False, "unit_box": False},
        # the benchmark: clustered matter of a cosmological volume, with the multipoles gravity needs
        {"name": "build_128m_clumps", "kind": "build", "model": 5, "n": 1 << 27, "dist": "clumps", "curve": "hilbert",
         "ncrit": 64, "levels": 21, "masses": True, "unit_box": False},
        # the same matter with small leaves (the gravity solver's choice), a ragged number of particles
        {"name": "build_16m_ncrit16", "kind": "build", "model": 6, "n": 16_789_561, "dist": "clumps",
         "curve": "hilbert", "ncrit": 16, "levels": 21, "masses": True, "unit_box": False},
        # 30-bit keys: a coarse tree of clustered matter whose densest cells stay full
        {"name": "build_16m_30bit", "kind": "build", "model": 7, "n": 16_777_139, "dist": "clumps", "curve": "morton",
         "ncrit": 64, "levels": 10, "masses": True, "unit_box": False},
        # hundreds of independent systems of very different sizes in one call (an ensemble)
        {"name": "batch_512", "kind": "batch", "model": 8, "sets": 512, "lo": 10.0, "hi": 20.0, "sizes_seed": 4,
         "curve": "morton", "ncrit": 32},
        # a few dozen small systems in one call: launches, and many more sets than SMs' worth of work
        {"name": "batch_48_small", "kind": "batch", "model": 9, "sets": 48, "lo": 7.0, "hi": 12.0, "sizes_seed": 9,
         "curve": "hilbert", "ncrit": 16},
        # one time step of several runs: every rebuild starts from the previous step's leaves
        {"name": "steps_4x4m", "kind": "steps", "model": 10, "runs": 4, "n": (1 << 22) + 1027, "curve": "hilbert",
         "ncrit": 64},
        # the locally essential tree of one process: the global tree refined around its key range
        {"name": "focus_4m", "kind": "focus", "model": 11, "n": 1 << 22, "dist": "plummer",
         "curve": "hilbert", "ncrit": 64, "theta": 0.5, "part": 3, "parts": 8},
        # multipoles for new masses on a tree that is already built
        {"name": "moments_8m", "kind": "moments", "model": 12, "n": 8_388_593, "dist": "clumps",
         "curve": "hilbert", "ncrit": 64},
    ]


def draw(rng):
    def log2(lo, hi):
        return int(2.0 ** rng.uniform(lo, hi))

    kind = rng.choice(["build", "build", "build", "build", "batch", "steps", "focus", "moments"])
    curve = rng.choice(["hilbert", "hilbert", "morton"])
    model = rng.randrange(1 << 30)
    if kind == "build":
        dist = rng.choice(["uniform", "plummer", "gaussian", "clumps"])
        return {"kind": "build", "model": model, "n": log2(11.0, 26.0), "dist": dist, "curve": curve,
                "ncrit": rng.choice([16, 16, 24, 32, 64, 64]), "levels": rng.choice([21, 21, 21, 10]),
                "masses": rng.random() < 0.5, "unit_box": dist == "uniform" and rng.random() < 0.5}
    if kind == "batch":
        lo = rng.uniform(6.0, 12.0)
        return {"kind": "batch", "model": model, "sets": log2(3.0, 9.0), "lo": lo, "hi": lo + rng.uniform(1.0, 6.0),
                "sizes_seed": rng.randrange(1 << 30), "curve": curve, "ncrit": rng.choice([16, 32, 64])}
    if kind == "steps":
        return {"kind": "steps", "model": model, "runs": rng.randint(2, 8), "n": log2(12.0, 22.0), "curve": curve,
                "ncrit": 64}
    if kind == "focus":
        parts = rng.randint(4, 16)
        return {"kind": "focus", "model": model, "n": log2(14.0, 23.0),
                "dist": rng.choice(["uniform", "plummer", "gaussian"]),
                "curve": curve, "ncrit": rng.choice([32, 64]), "theta": rng.choice([0.5, 0.8, 1.0]),
                "part": rng.randrange(parts), "parts": parts}
    return {"kind": "moments", "model": model, "n": log2(12.0, 24.0),
            "dist": rng.choice(["uniform", "plummer", "clumps"]), "curve": curve, "ncrit": rng.choice([16, 32, 64])}


# ------------------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _u(g, n):
    return torch.rand(n, dtype=torch.float64, device="cuda", generator=g)


def _randn(g, n):
    return torch.randn(n, dtype=torch.float64, device="cuda", generator=g)


def _plummer(g, n):
    """Plummer sphere of scale radius 1 cut at r = 20, isotropic."""
    u = _u(g, n).clamp_min_(1e-300).mul_((400.0 / 401.0) ** 1.5)
    r = u.pow_(-2.0 / 3.0).sub_(1.0).rsqrt_()
    c = _u(g, n).mul_(2.0).sub_(1.0)
    phi = _u(g, n).mul_(2.0 * math.pi)
    s = (1.0 - c * c).sqrt_().mul_(r)
    return s * torch.cos(phi), s * torch.sin(phi), c.mul_(r)


def _particles(dist, n, g):
    if dist == "uniform":
        return _u(g, n), _u(g, n), _u(g, n)
    if dist == "gaussian":
        return tuple(_randn(g, n).mul_(0.1).add_(0.5) for _ in range(3))
    if dist == "plummer":
        return _plummer(g, n)
    # 1,000 Gaussian clumps of very different widths hold 80 % of the particles, the rest is uniform
    centres = torch.rand((3, 1000), dtype=torch.float64, device="cuda", generator=g)
    sigma = 10.0 ** (2.0 * _u(g, 1000) - 4.0)
    which = torch.randint(0, 1000, (n,), device="cuda", generator=g)
    spread = sigma[which]
    loose = torch.rand(n, device="cuda", generator=g) >= 0.8
    out = []
    for d in range(3):
        c = _randn(g, n).mul_(spread).add_(centres[d][which])
        out.append(torch.where(loose, _u(g, n), c))
    return tuple(out)


def _masses(n, g):
    return torch.empty(n, dtype=torch.float32, device="cuda").log_normal_(0.0, 1.0, generator=g)


def _sizes(case):
    r = random.Random(case["sizes_seed"])
    sizes = [int(2.0 ** r.uniform(case["lo"], case["hi"])) for _ in range(case["sets"])]
    return sizes, [r.random() < 0.5 for _ in sizes]


def _offsets(sizes):
    off = [0]
    for s in sizes:
        off.append(off[-1] + s)
    return off


def _turned(arrays, g, scale=True):
    """Coordinates with their axes in another order and in another unit (a power of two)."""
    r = random.Random(g.initial_seed())
    order = r.sample(range(3), 3)
    unit = 2.0 ** r.randint(-3, 3) if scale else 1.0
    return tuple(arrays[d] * unit for d in order)


def _shuffled(arrays, g):
    p = torch.randperm(arrays[0].numel(), device="cuda", generator=g)
    return tuple(c[p] for c in arrays)


def _inputs(case, seed):
    g = _gen(seed)
    xyz = _particles(case["dist"], case["n"], _gen(case["model"]))
    xyz = _turned(_shuffled(xyz, g), g, scale=not case.get("unit_box"))
    return xyz, (_masses(case["n"], g) if case.get("masses") or case["kind"] == "moments" else None)


def _box(case):
    return torch.tensor([0.0, 0.0, 0.0, 1.0], dtype=torch.float64, device="cuda") if case.get("unit_box") else None


def _batch_inputs(case, seed):
    """Sets back to back, each uniform in the unit cube or a Plummer sphere."""
    sizes, uniform = _sizes(case)
    g, gm = _gen(seed), _gen(case["model"])
    n, size = sum(sizes), torch.tensor(sizes, device="cuda")
    which = torch.repeat_interleave(torch.tensor(uniform, device="cuda"), size)
    xyz = tuple(torch.where(which, _u(gm, n), c) for c in _plummer(gm, n))
    order = torch.argsort(torch.repeat_interleave(torch.arange(len(sizes), device="cuda"), size) + _u(g, n))
    return _turned([c[order] for c in xyz], g), _offsets(sizes)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "build":  # the particles, and the buffers a program keeps from build to build
        xyz, m = _inputs(case, seed)
        bufs = cs.OctreeBuffers.allocate(case["n"], cs.leaf_capacity(case["n"], case["ncrit"]), "cuda", case["levels"])
        return {"kind": kind, "xyz": xyz, "m": m, "box": _box(case), "bufs": bufs, "curve": CURVES[case["curve"]],
                "ncrit": case["ncrit"], "levels": case["levels"]}
    if kind == "batch":
        xyz, off = _batch_inputs(case, seed)
        n, s = off[-1], len(off) - 1
        bufs = cs.BatchBuffers.allocate(n, s, cs.batched_capacity(n, s, case["ncrit"]), "cuda")
        return {"kind": kind, "xyz": xyz, "off": torch.tensor(off, dtype=torch.int64, device="cuda"), "bufs": bufs,
                "ws": cs.Workspace("cuda"), "curve": CURVES[case["curve"]], "ncrit": case["ncrit"]}
    if kind == "steps":  # the positions of two consecutive steps; the first step's trees are built
        g, gm = _gen(seed), _gen(case["model"])
        n, runs = case["n"], case["runs"]
        a = _plummer(gm, n * runs)
        b = tuple(c + 0.04 * _randn(gm, n * runs) for c in a)  # 10^-3 of the cube's side
        both = torch.arange(runs, device="cuda").repeat_interleave(n) + _u(g, n * runs)
        order = torch.argsort(both)
        both = _turned([torch.cat([c[order], d[order]]) for c, d in zip(a, b)], g)
        a, b = (tuple(c[k * n * runs:(k + 1) * n * runs].contiguous() for c in both) for k in (0, 1))
        off = torch.tensor([n * k for k in range(runs + 1)], dtype=torch.int64, device="cuda")
        stepper = cs.TimeStepper(*a, off, curve=CURVES[case["curve"]], ncrit=case["ncrit"])
        stepper.rebuild()
        return {"kind": kind, "stepper": stepper, "at": [a, b], "step": 0}
    if kind == "focus":
        # the process has its sorted keys and the global tree's leaves; it keeps the focused tree in
        # arrays of fixed capacity
        (x, y, z), _ = _inputs(case, seed)
        t = cs.build_octree(x, y, z, curve=CURVES[case["curve"]], ncrit=case["ncrit"])
        nl = t["n_leaves"]
        f0 = int(t["leaves"][nl * case["part"] // case["parts"]])
        f1 = int(t["leaves"][nl * (case["part"] + 1) // case["parts"]]) if case["part"] + 1 < case["parts"] else 1 << 63
        cap = cs.leaf_capacity(case["n"], case["ncrit"])
        return {"kind": kind, "keys": t["sorted_keys"], "leaves": t["leaves"].clone(),
                "ends": (f0, f1 if f1 > f0 else 1 << 63), "ws": cs.Workspace("cuda"),
                "curve": CURVES[case["curve"]], "ncrit": case["ncrit"], "theta": case["theta"],
                "K": torch.zeros(cap + 1, dtype=torch.int64, device="cuda"),
                "N": torch.zeros(cap, dtype=torch.int32, device="cuda")}
    (x, y, z), m = _inputs(case, seed)
    t = cs.build_octree(x, y, z, curve=CURVES[case["curve"]], ncrit=case["ncrit"])
    nn = t["NK"].numel()
    out = [torch.empty(k * nn, dtype=dt, device="cuda")
           for k, dt in ((1, torch.float32), (3, torch.float64), (6, torch.float32))]
    return {"kind": kind, "xyz": (x, y, z), "m": m, "tree": t, "out": out, "ws": cs.Workspace("cuda")}


def run(state):
    kind = state["kind"]
    if kind == "build":
        t = cs.build_octree(*state["xyz"], curve=state["curve"], ncrit=state["ncrit"], box=state["box"],
                            masses=state["m"], buffers=state["bufs"], levels=state["levels"])
        return {k: v for k, v in t.items() if k != "buffers"}
    if kind == "batch":
        t = cs.build_octrees_batched(*state["xyz"], state["off"], curve=state["curve"], ncrit=state["ncrit"],
                                     ws=state["ws"], buffers=state["bufs"])
        return {k: v for k, v in t.items() if isinstance(v, (torch.Tensor, int))}
    if kind == "steps":
        st = state["stepper"]
        state["step"] += 1
        st.x, st.y, st.z = state["at"][state["step"] % 2]
        t = st.rebuild()
        return {k: v for k, v in t.items() if isinstance(v, (torch.Tensor, int)) and k != "boxes"}
    if kind == "focus":
        f0, f1 = state["ends"]
        K, N, passes = cs.build_focus_leaves(state["keys"], state["ncrit"], f0, f1, state["theta"], state["curve"],
                                             warm_leaves=state["leaves"], ws=state["ws"])
        state["K"][:K.numel()].copy_(K)
        state["N"][:N.numel()].copy_(N)
        return {"leaves": state["K"], "counts": state["N"], "n_leaves": N.numel(), "passes": passes}
    t = state["tree"]
    mass, com, quad = state["out"]
    cs.cstone_upsweep_multipoles(*state["xyz"], state["m"], t["perm"], t["leaf_offsets"], t["n_leaves"],
                                 t["leaf_to_node"], t["CO"], t["LO"], t["box"], mass, com, quad, ws=state["ws"])
    return {"mass": mass, "com": com.view(3, -1), "quad": quad.view(6, -1)}


# ------------------------------------------------------------------------------ least work
def _nodes(n, ncrit):
    """Leaves and nodes of the tree of n particles: a leaf holds about 0.28 ncrit of them in these
    distributions (measured 0.27-0.29 at ncrit 64 and 16)."""
    nl = max(8.0, 3.6 * n / ncrit)
    return nl, nl * 8.0 / 7.0


def _tree_bytes(n, nl, nn, key):
    # sorted keys and permutation; leaf keys, counts, offsets, leaf-to-node; node keys, children, counts
    return (key + 4) * n + (key + 12) * nl + (key + 8) * nn


def work(case):
    kind = case["kind"]
    if kind == "build":
        n, key = case["n"], 8 if case["levels"] == 21 else 4
        nl, nn = _nodes(n, case["ncrit"])
        b = 24 * n + key * n + _tree_bytes(n, nl, nn, key)  # coordinates in; keys, sorted keys and tree out
        f = 0.0
        if case["masses"]:
            b += 4 * n + 52 * nn
            f = 30.0 * n + 60.0 * nn
        return {"bytes": b, "flops": f}
    if kind == "batch":
        n = sum(_sizes(case)[0])
        nl, nn = _nodes(n, case["ncrit"])
        return {"bytes": 32 * n + _tree_bytes(n, nl, nn, 8), "flops": 0.0}
    if kind == "steps":
        n = case["n"] * case["runs"]
        nl, nn = _nodes(n, case["ncrit"])
        return {"bytes": 32 * n + 8 * nl + _tree_bytes(n, nl, nn, 8), "flops": 0.0}
    if kind == "focus":  # the particles inside the focus, and the tree in and out
        n = case["n"]
        nl, _ = _nodes(n, case["ncrit"])
        return {"bytes": 8 * n / case["parts"] + 8 * nl + 12 * nl / case["parts"], "flops": 0.0}
    n = case["n"]
    nl, nn = _nodes(n, case["ncrit"])
    return {"bytes": 32 * n + 8 * nl + 56 * nn, "flops": 30.0 * n + 60.0 * nn}


# ------------------------------------------------------------------------------ 64-bit values
def _cube(x, y, z):
    lo = torch.stack([x.min(), y.min(), z.min()])
    side = (torch.stack([x.max(), y.max(), z.max()]) - lo).max()
    return torch.cat([lo, side.reshape(1)])


def _spread(v):
    """Bit b of a 21-bit value to bit 3b."""
    v = v.to(torch.int64)
    for s, m in ((32, 0x001F00000000FFFF), (16, 0x001F0000FF0000FF), (8, 0x100F00F00F00F00F),
                 (4, 0x10C30C30C30C30C3), (2, 0x1249249249249249)):
        v = (v | (v << s)) & m
    return v


def _exact_keys(x, y, z, box, curve):
    """63-bit keys: cells of the 2^21 grid over the cube, Morton (x highest) or Hilbert in Skilling's
    transposed form."""
    scale = 2097152.0 / float(box[3])
    X = [((c - box[d]) * scale).floor_().clamp_(0, 2097151).to(torch.int32) for d, c in enumerate((x, y, z))]
    if curve == "hilbert":
        for b in range(20, 0, -1):
            low = (1 << b) - 1
            for i in range(3):
                on = ((X[i] >> b) & 1).bool()
                if i == 0:
                    X[0] = torch.where(on, X[0] ^ low, X[0])
                    continue
                t = (X[0] ^ X[i]) & low
                X[i] = torch.where(on, X[i], X[i] ^ t)
                X[0] = X[0] ^ torch.where(on, torch.full_like(t, low), t)
        X[1] ^= X[0]
        X[2] ^= X[1]
        flip = torch.zeros_like(X[0])
        for b in range(20, 0, -1):
            flip ^= ((X[2] >> b) & 1) * ((1 << b) - 1)
        X = [v ^ flip for v in X]
    return (_spread(X[0]) << 2) | (_spread(X[1]) << 1) | _spread(X[2])


def _exact_moments(x, y, z, m, box, curve, ncrit, levels):
    """Mass, centre of mass and raw second moments about it of every node of the octree whose leaves
    hold at most ncrit particles, breadth-first, in 64 bits."""
    keys, order = torch.sort(_exact_keys(x, y, z, box, curve), stable=True)
    pos = [c[order] for c in (x, y, z)]
    w = m[order].double()
    del order
    n, dev = keys.numel(), keys.device
    # the levels: start key, particle range and (for split nodes) place of the children
    start = torch.zeros(1, dtype=torch.int64, device=dev)
    a, b = torch.zeros_like(start), torch.full_like(start, n)
    tree = []
    for level in range(levels + 1):
        split = (b - a > ncrit) if level < levels else torch.zeros_like(a, dtype=torch.bool)
        tree.append((a, b, split))
        if not bool(split.any()):
            break
        step = torch.arange(8, device=dev, dtype=torch.int64) << (3 * (20 - level))
        child = start[split][:, None] + step[None, :]
        ca = torch.searchsorted(keys, child.reshape(-1)).view(-1, 8)
        cb = torch.cat([ca[:, 1:], b[split][:, None]], dim=1)
        start, a, b = child.reshape(-1), ca.reshape(-1), cb.reshape(-1)
    del keys
    # leaf sums about each leaf's first particle
    mom = []
    for a, b, split in tree:
        leaf = ~split & (b > a)
        la, lb = a[leaf], b[leaf]
        size = lb - la
        ids = torch.repeat_interleave(torch.arange(la.numel(), device=dev), size)
        first = torch.cumsum(size, 0) - size
        p = torch.arange(ids.numel(), device=dev) - first[ids] + la[ids]
        wm = w[p]
        M = torch.zeros(la.numel(), dtype=torch.float64, device=dev).index_add_(0, ids, wm)
        com = torch.empty((3, la.numel()), dtype=torch.float64, device=dev)
        e = []
        for d in range(3):
            anchor = pos[d][la]
            off = pos[d][p] - anchor[ids]
            mean = torch.zeros_like(M).index_add_(0, ids, wm * off) / M
            com[d] = anchor + mean
            e.append(off - mean[ids])
        Q = torch.stack([torch.zeros_like(M).index_add_(0, ids, wm * e[i] * e[j])
                         for i, j in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))])
        full = [torch.zeros(k + (a.numel(),), dtype=torch.float64, device=dev) for k in ((), (3,), (6,))]
        for f, v in zip(full, (M, com, Q)):
            f[..., leaf] = v
        mom.append(full)
        del ids, p, wm, e
    # internal nodes from their eight children
    for level in range(len(tree) - 2, -1, -1):
        split = tree[level][2]
        M, com, Q = (v.view(v.shape[:-1] + (-1, 8)) for v in mom[level + 1])
        Ms = M.sum(-1)
        c = (M * com).sum(-1) / Ms
        e = com - c[..., None]
        pairs = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))
        Qs = torch.stack([(Q[k] + M * e[i] * e[j]).sum(-1) for k, (i, j) in enumerate(pairs)])
        for f, v in zip(mom[level], (Ms, c, Qs)):
            f[..., split] = v
    return [torch.cat([lv[k] for lv in mom], dim=-1) for k in range(3)]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("build", "moments"):
        (x, y, z), m = _inputs(case, seed)
        box = _box(case)
        box = _cube(x, y, z) if box is None else box
        out = {"box": box} if kind == "build" else {}
        if m is not None:
            levels = case.get("levels", 21)
            moments = _exact_moments(x, y, z, m, box, case["curve"], case["ncrit"], levels)
            out.update(zip(("mass", "com", "quad"), moments))
        return out
    if kind == "batch":
        (x, y, z), off = _batch_inputs(case, seed)
        return {"boxes": torch.stack([_cube(x[a:b], y[a:b], z[a:b]) for a, b in zip(off, off[1:])])}
    return None
