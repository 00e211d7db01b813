"""The measured cases: what a user of this library has it do, through the
package's public entry points.

A case is a dict of plain values. `listed()` names twelve of them, `draw()`
gives more of the same ranges. Every build returns its whole tree
(permutation, split values, split coordinates, leaf offsets, levels), every
query its whole answer. Points, subset ids, workspaces, output buffers,
descriptors, trees to query and the server are made by `prepare()`, as a
program that builds trees again and again keeps them; each `run()` is one
call (the server: one burst of requests).

Tolerances are "exact" throughout: the build selects and moves keys and does
no arithmetic on them, so its outputs are fixed bit for bit; the box query
only compares; the nearest-neighbour distances are defined as sums of
separately rounded float64 products in coordinate order. The Fourier-moment
estimator does sum in float, in an order that the inputs fix, so that two
calls agree bit for bit. Sums in another order move a split by about 1e-7 of
its cell's width, and a point that changes sides shifts whole ranges of the
permutation, so that no element-wise tolerance below "exact" would hold for
another order.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2201_08288_gb300 import kdt
from paper_2201_08288_gb300.workloads import leaf_mode_levels

MODES = {"mod": kdt.KDT_SUBSET_MOD, "contiguous": kdt.KDT_SUBSET_CONTIGUOUS, "explicit": kdt.KDT_SUBSET_EXPLICIT}
RULES = {"cyclic": kdt.KDT_KEY_CYCLIC, "widest": kdt.KDT_KEY_WIDEST_SPREAD}


def _build(n, d, dist, r, mode="mod", rule="cyclic", depth=0, leaf=32, combine="weighted"):
    return {"kind": "build", "n": n, "d": d, "dist": dist, "r": r, "mode": mode, "rule": rule, "depth": depth,
            "leaf": leaf, "combine": combine}


def listed():
    return [
        # one small tree, as a program builds one per object or frame: all latency
        dict(_build(1000, 3, "uniform", 8), name="build_1k"),
        # the benchmark's first configuration: an ordinary point set in three coordinates
        dict(_build(65536, 3, "uniform", 8, depth=10), name="build_64k"),
        # a serving request of ordinary size: many coordinates, a ragged size, leaves of at most 64
        dict(_build(300_007, 16, "mixture8", 32, leaf=64), name="build_300k_d16"),
        # user-given subsets (more than 256, so 16-bit ids), widest spread, ties, d without a compiled kernel
        dict(_build(3_000_017, 5, "student", 1000, "explicit", "widest", leaf=50), name="build_3m_ids16"),
        # the second configuration: subsets that are blocks of the input, as files or partitions come
        dict(_build(1 << 24, 3, "mixture16", 64, "contiguous", depth=16), name="build_16m_blocks"),
        # the simulation study's shape (correlated normals, subsets by index mod 64, depth 10), a ragged size
        dict(_build(50_000_021, 3, "mvn", 64, depth=10), name="build_50m_mvn"),
        # the third configuration, the library's headline: heavy tails, ties, 256 random subsets, widest spread
        dict(_build(1 << 27, 8, "student", 256, "explicit", "widest", depth=20), name="build_128m_widest"),
        # the paper's own estimator on the study's shape
        {"kind": "fourier", "n": 4_000_037, "d": 3, "J": 16, "depth": 10, "name": "fourier_4m"},
        # many independent trees of uneven sizes in one call
        {"kind": "batched", "trees": 512, "lo": 8.0, "hi": 18.0, "leaf": 32, "name": "batched_512"},
        # a burst of requests to the build server
        {"kind": "served", "trees": 48, "lo": 10.0, "hi": 20.0, "leaf": 64, "name": "served_48"},
        # searches in a tree built before: neighbours of points like those in the tree, boxes around them
        {"kind": "knn", "n": 1_000_003, "d": 3, "dist": "mixture16", "leaf": 32, "nq": 100_003, "k": 8,
         "name": "knn_1m_k8"},
        {"kind": "box", "n": 4_000_037, "d": 3, "dist": "uniform", "leaf": 32, "nq": 50_021, "inside": 40.0, "cap": 128,
         "name": "box_4m"},
    ]


def _log_int(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def draw(rng):
    kind = rng.choice(["build"] * 5 + ["fourier", "batched", "served", "knn", "box"])
    if kind == "build":
        n = _log_int(rng, 500, 3e7)
        mode = rng.choice(["mod", "contiguous", "explicit"])
        depth = 0 if rng.random() < 0.5 else max(1, int(math.log2(n)) - rng.randint(4, 9))
        return _build(n, rng.choice([2, 3, 3, 4, 5, 8, 8, 12, 16]), rng.choice(["uniform", "mixture8", "student", "mvn"]),
                      _log_int(rng, 1, 1024), mode, rng.choice(["cyclic", "widest"]), depth, rng.randint(16, 128),
                      "unweighted" if rng.random() < 0.125 else "weighted")
    if kind == "fourier":
        return {"kind": kind, "n": _log_int(rng, 2e4, 1e7), "d": rng.choice([2, 3, 3, 4]), "J": rng.randint(4, 32),
                "depth": rng.randint(5, 11)}
    if kind == "batched":
        lo = rng.uniform(7.0, 11.0)
        return {"kind": kind, "trees": _log_int(rng, 16, 1024), "lo": lo, "hi": lo + rng.uniform(2.0, 7.0),
                "leaf": rng.choice([16, 32, 64])}
    if kind == "served":
        lo = rng.uniform(9.0, 13.0)
        return {"kind": kind, "trees": _log_int(rng, 8, 64), "lo": lo, "hi": lo + rng.uniform(2.0, 7.0),
                "leaf": rng.choice([32, 64])}
    n = _log_int(rng, 1e4, 8e6)
    c = {"kind": kind, "n": n, "d": rng.choice([2, 3, 3, 4, 8]), "dist": rng.choice(["uniform", "mixture16", "mvn"]),
         "leaf": rng.randint(8, 64), "nq": _log_int(rng, 1e3, 2e5)}
    if kind == "knn":
        return dict(c, k=rng.choice([1, 4, 8, 16, 32]))
    return dict(c, inside=_log_int(rng, 4, 400), cap=rng.choice([0, 64, 256]))


# ------------------------------------------------------------------ inputs


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gen(seed):
    return torch.Generator(device=_device()).manual_seed(int(seed))


def _points(n, d, dist, g, out=None):
    """Float32 points [d, n] of the distributions of the benchmark configurations."""
    dev = g.device
    x = torch.empty((d, n), device=dev) if out is None else out
    if dist == "uniform":
        return x.uniform_(generator=g)
    if dist.startswith("mixture"):  # equal isotropic Gaussians, centres uniform in the unit cube
        k = int(dist[len("mixture"):])
        centres = torch.rand((k, d), generator=g, device=dev)
        comp = torch.randint(0, k, (n,), generator=g, device=dev)
        for j in range(d):
            x[j].normal_(0.0, 0.05, generator=g).add_(centres[:, j][comp])
        return x
    if dist == "mvn":  # unit variances, common correlation 1/2
        z0 = torch.randn(n, generator=g, device=dev)
        for j in range(d):
            x[j].normal_(generator=g).add_(z0).mul_(math.sqrt(0.5))
        return x
    if dist == "probit":  # the correlated normals mapped into (0, 1) by the normal distribution function
        _points(n, d, "mvn", g, x)
        return x.copy_(torch.special.ndtr(x).clamp_(2.0 ** -24, 1.0 - 2.0 ** -24))
    if dist == "student":  # three degrees of freedom; a tenth of the values on a grid of 1/256 (ties)
        for j in range(d):
            v = torch.randn(n, generator=g, device=dev).square_()
            for _ in range(2):
                v.addcmul_(*[torch.randn(n, generator=g, device=dev)] * 2)
            x[j].normal_(generator=g).div_(v.div_(3.0).sqrt_().clamp_(min=1e-6))
            snap = torch.rand(n, generator=g, device=dev) < 0.1
            torch.where(snap, torch.round(x[j] * 256.0) / 256.0, x[j], out=x[j])
        return x
    raise ValueError(dist)


def _ids(n, r, g):
    return torch.randint(0, r, (n,), generator=g, device=g.device).to(torch.uint8 if r <= 256 else torch.int16)


def _tree_buffers(n, levels, dev):
    """Output buffers; zeros, since a tree in leaf mode fills what it needs of its capacity."""
    return kdt.Tree(torch.zeros(n, dtype=torch.int32, device=dev),
                    torch.zeros((1 << levels) - 1, device=dev),
                    torch.zeros((1 << levels) - 1, dtype=torch.int8, device=dev),
                    torch.zeros((1 << levels) + 1, dtype=torch.int64, device=dev), 0)


def _workspace(nbytes, dev):
    return torch.empty(nbytes, dtype=torch.uint8, device=dev)


def _tree_args(case):
    """Arguments of kdt_build for a build case (without the ids)."""
    return dict(r=case["r"], subset_mode=MODES[case["mode"]], key_rule=RULES[case["rule"]], depth=case["depth"],
                leaf_size=case["leaf"], max_levels=leaf_mode_levels(case["n"]),
                combine_rule=kdt.KDT_COMBINE_UNWEIGHTED if case["combine"] == "unweighted" else kdt.KDT_COMBINE_WEIGHTED)


def _build_inputs(case, seed):
    g = _gen(seed)
    x = _points(case["n"], case["d"], case["dist"], g)
    return x, _ids(case["n"], case["r"], g) if case["mode"] == "explicit" else None


def _forest(case):
    """Sizes and parameters of a case's independent trees (a function of the case alone)."""
    rng = np.random.default_rng(case["trees"] * 1000 + int(case["lo"] * 10))
    served = case["kind"] == "served"
    out = []
    for _ in range(case["trees"]):
        n = int(2.0 ** rng.uniform(case["lo"], case["hi"]))
        out.append({"n": n, "d": int(rng.choice([3, 16] if served else [2, 3, 8, 16])),
                    "dist": "uniform" if rng.random() < 0.5 else "mixture8",
                    "r": 32 if served else int(rng.choice([4, 16, 64])), "mode": "mod", "rule": "cyclic", "depth": 0,
                    "leaf": case["leaf"], "combine": "weighted"})
    return out


def _forest_points(case, seed):
    """The trees' points, drawn as one stretch of uniform and one of normal values and cut up: each tree's array
    starts on a 256-byte boundary, as one allocation each would."""
    g = _gen(seed)
    trees = _forest(case)
    starts, total = [], 0
    for t in trees:
        starts.append(total)
        total += -(-t["n"] * t["d"] // 64) * 64
    uni = torch.rand(total, generator=g, device=g.device)
    for t, s in zip(trees, starts):
        if t["dist"] != "uniform":
            _points(t["n"], t["d"], t["dist"], g, uni[s:s + t["n"] * t["d"]].view(t["d"], t["n"]))
    return trees, [uni[s:s + t["n"] * t["d"]].view(t["d"], t["n"]) for t, s in zip(trees, starts)]


def _forest_buffers(trees, dev):
    """One buffer per output for all trees, and each tree's part of it."""
    levels = [leaf_mode_levels(t["n"]) for t in trees]
    whole = kdt.Tree(torch.zeros(sum(t["n"] for t in trees), dtype=torch.int32, device=dev),
                     torch.zeros(sum((1 << v) - 1 for v in levels), device=dev),
                     torch.zeros(sum((1 << v) - 1 for v in levels), dtype=torch.int8, device=dev),
                     torch.zeros(sum((1 << v) + 1 for v in levels), dtype=torch.int64, device=dev), 0)
    parts, p, v, o = [], 0, 0, 0
    for t, lv in zip(trees, levels):
        m = 1 << lv
        parts.append(kdt.Tree(whole.perm[p:p + t["n"]], whole.split_vals[v:v + m - 1], whole.split_dims[v:v + m - 1],
                              whole.node_offsets[o:o + m + 1], 0))
        p, v, o = p + t["n"], v + m - 1, o + m + 1
    return whole, parts


class _Serving:
    """A server held by a program, closed with it."""

    def __init__(self, budget, slots):
        self.server = kdt.Server(budget, slots)

    def __del__(self):
        self.server.close()


def prepare(case, seed):
    dev = _device()
    kind = case["kind"]
    if kind == "build":
        x, sid = _build_inputs(case, seed)
        args = _tree_args(case)
        p = kdt.make_params(case["n"], case["d"], sid_ptr=0 if sid is None else sid.data_ptr(),
                            sid_bytes=1 if sid is None else sid.element_size(), **args)
        return {"kind": kind, "x": x, "args": dict(args, sid=sid, workspace=_workspace(kdt.kdt_workspace_size(p), dev),
                                                   outputs=_tree_buffers(case["n"], case["depth"] or args["max_levels"], dev))}
    if kind == "fourier":
        x = _points(case["n"], case["d"], "probit", _gen(seed))
        args = dict(depth=case["depth"], fourier_j=case["J"])
        ws = _workspace(kdt.kdt_workspace_size(kdt.make_params(case["n"], case["d"], **args)), dev)
        return {"kind": kind, "x": x, "args": dict(args, workspace=ws, outputs=_tree_buffers(case["n"], case["depth"], dev))}
    if kind in ("batched", "served"):
        trees, xs = _forest_points(case, seed)
        whole, parts = _forest_buffers(trees, dev)
        items = [dict(points=x, r=t["r"], leaf_size=t["leaf"], max_levels=leaf_mode_levels(t["n"]))
                 for t, x in zip(trees, xs)]
        state = {"kind": kind, "items": items, "whole": whole, "parts": parts}
        if kind == "batched":
            state["descs"] = kdt.make_descs(items, parts)[0]
            state["workspace"] = _workspace(kdt.kdt_workspace_size_batched(state["descs"]), dev)
        else:
            state["serving"] = _Serving(4 << 30, 256)
        return state
    # a search: the tree it searches is there already
    g = _gen(seed)
    n, d = case["n"], case["d"]
    x = _points(n, d, case["dist"], g)
    tree = kdt.kdt_build(x, r=16, leaf_size=case["leaf"], max_levels=leaf_mode_levels(n))
    near = x[:, torch.randint(0, n, (case["nq"],), generator=g, device=g.device)]
    state = {"kind": kind, "x": x, "tree": tree}
    if kind == "knn":
        width = x.std(dim=1, keepdim=True) * n ** (-1.0 / d)
        state.update(q=(near + width * torch.randn(near.shape, generator=g, device=g.device)).contiguous(), k=case["k"])
    else:
        # boxes around points of the set, of sides that hold about `inside` points where it is as dense as on average
        half = (x.amax(dim=1, keepdim=True) - x.amin(dim=1, keepdim=True)) * (0.5 * (case["inside"] / n) ** (1.0 / d))
        half = half * (0.5 + torch.rand(near.shape, generator=g, device=g.device))
        state.update(lo=(near - half).contiguous(), hi=(near + half).contiguous(), cap=case["cap"])
    return state


# -------------------------------------------------------------------- passes


def _of_tree(t):
    return {"perm": t.perm, "split_vals": t.split_vals, "split_dims": t.split_dims, "node_offsets": t.node_offsets,
            "levels": t.levels}


def run(state):
    kind = state["kind"]
    if kind in ("build", "fourier"):
        return _of_tree(kdt.kdt_build(state["x"], **state["args"]))
    if kind == "batched":
        trees, _ = kdt.kdt_build_batched(state["items"], workspace=state["workspace"], outputs=state["parts"],
                                         descs=state["descs"])
        return dict(_of_tree(state["whole"]), levels=np.array([t.levels for t in trees]))
    if kind == "served":
        server = state["serving"].server
        tickets = [server.submit(it, out) for it, out in zip(state["items"], state["parts"])]
        trees = [server.poll(t)[1] for t in tickets]
        return dict(_of_tree(state["whole"]), levels=np.array([t.levels for t in trees]))
    if kind == "knn":
        idx, d2 = kdt.kdt_query_knn(state["x"], state["tree"], state["q"], state["k"])
        return {"idx": idx, "d2": d2}
    counts, lists = kdt.kdt_query_box(state["x"], state["tree"], state["lo"], state["hi"], list_cap=state["cap"])
    return {"counts": counts} if lists is None else {"counts": counts, "lists": lists}


# ---------------------------------------------------------- work and tolerance


def _tree_bytes(n, d, levels, id_bytes=0):
    nodes = (1 << levels) - 1
    return n * (4 * d + id_bytes) + 4 * n + 5 * nodes + 8 * (nodes + 2)


def _build_levels(t):
    return t["depth"] or max(0, math.ceil(math.log2(t["n"] / t["leaf"])))


def work(case):
    kind = case["kind"]
    n, d = case.get("n", 0), case.get("d", 0)
    if kind == "build":
        ids = 0 if case["mode"] != "explicit" else 1 if case["r"] <= 256 else 2
        return {"bytes": _tree_bytes(n, d, _build_levels(case), ids), "flops": 0}
    if kind == "fourier":  # per level and point: the key's sine and cosine, then two sums of a product per harmonic
        return {"bytes": _tree_bytes(n, d, case["depth"]), "flops": case["depth"] * n * (20 + 6 * case["J"])}
    if kind in ("batched", "served"):
        return {"bytes": sum(_tree_bytes(t["n"], t["d"], _build_levels(t)) for t in _forest(case)), "flops": 0}
    # a search reads its query and writes its answer; of the tree, at least the points it returns or counts
    if kind == "knn":
        k = case["k"]
        return {"bytes": case["nq"] * (4 * d + k * (4 * d + 4) + 12 * k), "flops": case["nq"] * k * 3 * d}
    found = case["inside"]
    return {"bytes": int(case["nq"] * (8 * d + found * (4 * d + 4) + 4 + 4 * min(found, case["cap"]))), "flops": 0}


def tolerance(case):
    return "exact"


# ------------------------------------------------------------ 64-bit reference


def _order_key(x):
    """Integers that order like the floats, -0 below +0."""
    b = x.contiguous().view(torch.int32).to(torch.int64)
    return torch.where(b >= 0, b, -1 - (b & 0x7fffffff))


def _from_key(k):
    return torch.where(k >= 0, k, (-1 - k) - (1 << 31)).to(torch.int32).view(torch.float32).to(torch.float64)


def _starts(count):
    """Start of each group, given the groups' sizes in order."""
    return torch.cumsum(count, 0) - count


def _subset_median_splits(keys, cell, sid, r, cells, weighted):
    """Per cell: the median, weighted by size, of the lower medians of its subsets (0 where a cell is empty)."""
    lo = 1 << 31
    order, _ = torch.sort(((cell * r + sid) << 32) + (keys + lo))
    seg, w = torch.unique_consecutive(order >> 32, return_counts=True)
    med = order[_starts(w) + (w - 1) // 2] & 0xffffffff
    of = seg // r
    by, at = torch.sort((of << 32) + med)
    w = w[at] if weighted else torch.ones_like(w)
    total = torch.zeros(cells, dtype=torch.int64, device=w.device).index_add_(0, of, w)
    owner = by >> 32
    before = torch.cumsum(w, 0) - _starts(total)[owner]
    enough = 2 * before >= total[owner] if weighted else before - 1 >= (total[owner] - 1) // 2
    where = torch.where(enough, torch.arange(len(by), device=w.device), len(by))
    first = torch.full((cells,), len(by), dtype=torch.int64, device=w.device).scatter_reduce_(0, owner, where, "amin")
    has = total > 0
    return torch.where(has, (by[first.clamp(max=len(by) - 1)] & 0xffffffff) - lo, 0)


def _fourier_splits(x, cell, cells, a, b, J):
    """Per cell: the root of the estimator's count equation, its sums and the bisection in float64."""
    t = x.to(torch.float64)
    base = torch.zeros(cells, dtype=torch.float64, device=x.device)
    count = torch.bincount(cell, minlength=cells).to(torch.float64)
    ia, ib = (a > 0.0).to(torch.float64), (b < 1.0).to(torch.float64)
    base += 0.5 * count * (ib - ia)
    terms = []
    for k in range(1, J + 1):
        K, q = 2 * k - 1, 2.0 / (math.pi * (2 * k - 1))
        c = torch.zeros_like(base).index_add_(0, cell, torch.cos(K * t))
        s = torch.zeros_like(base).index_add_(0, cell, torch.sin(K * t))
        base += q * (s * (ia * torch.cos(K * a) + ib * torch.cos(K * b)) - c * (ia * torch.sin(K * a) + ib * torch.sin(K * b)))
        terms.append((K, 2.0 * q * c, -2.0 * q * s))
    lo, hi = a.clone(), b.clone()
    for _ in range(60):
        m = 0.5 * (lo + hi)
        f = base.clone()
        for K, c, s in terms:
            f += c * torch.sin(K * m) + s * torch.cos(K * m)
        lo, hi = torch.where(f < 0, m, lo), torch.where(f < 0, hi, m)
    return (0.5 * (lo + hi)).to(torch.float32)


def _tree64(x, sid, t, J=0):
    """The tree of points x [d, n] with subsets sid, level by level, with whole-array sorts."""
    d, n = x.shape
    dev = x.device
    cell = torch.zeros(n, dtype=torch.int64, device=dev)
    stall = torch.zeros(1, dtype=torch.int64, device=dev)
    lo, hi = torch.zeros((1, d), dtype=torch.float64, device=dev), torch.ones((1, d), dtype=torch.float64, device=dev)
    vals, dims = [], []
    widest = t["rule"] == "widest"
    levels = 0
    while levels < t["depth"] or not t["depth"]:
        cells = 1 << levels
        count = torch.bincount(cell, minlength=cells)
        if t["depth"]:
            live = count > 0
        else:
            live = (count > t["leaf"]) & (stall < (1 if widest else d))
            if not bool(live.any()):
                break
        if widest:
            low = torch.full((d, cells), math.inf, dtype=torch.float64, device=dev)
            high = -low
            for j in range(d):
                v = x[j].to(torch.float64)
                low[j].scatter_reduce_(0, cell, v, "amin")
                high[j].scatter_reduce_(0, cell, v, "amax")
            size = torch.where(count > 0, high - low, 0.0)
            j = torch.arange(d, device=dev)[:, None]
            dim = torch.where(size == size.amax(dim=0), j, d).amin(dim=0)
        else:
            dim = torch.full((cells,), levels % d, dtype=torch.int64, device=dev)
        here = x[dim[cell], torch.arange(n, device=dev)] if widest else x[levels % d]
        if J:
            c = levels % d
            split = _fourier_splits(here, cell, cells, lo[:, c], hi[:, c], J)
            right = here > split[cell]
            value = split.to(torch.float64)
            lo, hi = lo.repeat_interleave(2, 0), hi.repeat_interleave(2, 0)
            hi[0::2, c] = torch.minimum(hi[0::2, c], value)
            lo[1::2, c] = torch.maximum(lo[1::2, c], value)
        else:
            keys = _order_key(here)
            split = _subset_median_splits(keys, cell, sid, t["r"], cells, t["combine"] == "weighted")
            right = (keys > split[cell]) & live[cell]
            value = _from_key(split)
        vals.append(torch.where(live, value, math.inf))
        dims.append(torch.where(live, dim, -1))
        cell = 2 * cell + right
        empty = torch.bincount(cell, minlength=2 * cells)[1::2] == 0
        stall = torch.where(live, torch.where(empty, stall + 1, 0), stall).repeat_interleave(2)
        levels += 1
    perm = torch.sort(cell, stable=True).indices
    offs = torch.cat([torch.zeros(1, dtype=torch.int64, device=dev), torch.cumsum(torch.bincount(cell, minlength=1 << levels), 0)])
    none = torch.zeros(0, device=dev)
    return {"perm": perm, "split_vals": torch.cat(vals) if vals else none.to(torch.float64),
            "split_dims": torch.cat(dims) if dims else none.to(torch.int64), "node_offsets": offs, "levels": levels}


def _index_mod(n, r, dev):
    return torch.arange(n, device=dev) % r


def exact(case, seed):
    """The same outputs by torch, in 64 bits and without this repository's kernels."""
    kind = case["kind"]
    if kind == "build":
        if case["n"] * case["d"] * (8 if case["rule"] == "widest" else 1) > 1.4e8:
            return None  # sorts and reductions over all points, every level: too long
        x, sid = _build_inputs(case, seed)
        n, r, dev = case["n"], case["r"], x.device
        if case["mode"] == "mod":
            sid = _index_mod(n, r, dev)
        elif case["mode"] == "contiguous":
            sid = torch.arange(n, device=dev) * r // n
        return _tree64(x, sid.to(torch.int64), case)
    if kind == "fourier":
        x = _points(case["n"], case["d"], "probit", _gen(seed))
        sums = _tree64(x, None, {"depth": case["depth"], "rule": "cyclic", "r": 1}, case["J"])
        # a point that the last bit of a split sends to the other side moves others in the order: splits alone
        return {"perm": None, "split_vals": sums["split_vals"], "split_dims": sums["split_dims"], "node_offsets": None,
                "levels": sums["levels"]}
    if kind in ("batched", "served"):
        trees, xs = _forest_points(case, seed)
        whole, parts = _forest_buffers(trees, xs[0].device)
        vals, at, levels = whole.split_vals.to(torch.float64), 0, []
        for t, x, part in zip(trees, xs, parts):
            tree = _tree64(x, _index_mod(t["n"], t["r"], x.device), t)
            vals[at:at + len(tree["split_vals"])] = tree["split_vals"]
            at += len(part.split_vals)
            part.perm.copy_(tree["perm"])
            part.split_dims[:len(tree["split_dims"])] = tree["split_dims"].to(torch.int8)
            part.node_offsets[:len(tree["node_offsets"])] = tree["node_offsets"]
            levels.append(tree["levels"])
        return {"perm": whole.perm, "split_vals": vals, "split_dims": whole.split_dims,
                "node_offsets": whole.node_offsets, "levels": np.array(levels)}
    if kind == "knn":
        if case["nq"] * case["n"] * case["d"] > 4e11:
            return None  # every query against every point
        s = prepare(case, seed)
        x, q, k = s["x"].to(torch.float64), s["q"].to(torch.float64), case["k"]
        step = max(1, (1 << 28) // case["n"])
        near = []
        for b in range(0, case["nq"], step):
            part = q[:, b:b + step]
            d2 = torch.zeros((part.shape[1], case["n"]), dtype=torch.float64, device=x.device)
            for j in range(case["d"]):
                df = x[j][None, :] - part[j][:, None]
                d2 += df * df
            near.append(torch.topk(d2, min(k, case["n"]), dim=1, largest=False, sorted=True).values)
        return {"idx": None, "d2": torch.cat(near)}
    return None  # counts and indices: whole numbers
