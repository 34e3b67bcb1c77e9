"""Performance cases: list ranking and connected components as a program calls them.

A case is a dict of plain values. ``listed()`` holds the fixed ones, ``draw``
makes more of the same ranges, ``prepare`` puts a case's inputs on the GPU,
``run`` makes one pass through the package's public calls, ``work`` counts the
bytes a pass cannot do without, and ``exact`` gives the results from the
definition alone (positions along the list the inputs were cut from, smallest
ids by plain tensor operations), without this repository's code.

The ranges are those of the package's own workloads: single lists of 2^10 to
2^28 elements, graphs of 2^10 to 2^24 vertices with 1 to 16 edges per vertex
(uniform with up to 6, R-MAT, and collections of paths and of trees), batches of up to 2048
instances of 2^8 to 2^20, and weighted ranks of one list or a forest of lists.
All values are int32, the only type the calls take.
"""
import math

import torch

import paper_1002_4482_gb300 as lrcc

DEVICE = "cuda"
RMAT_A, RMAT_B, RMAT_C = 0.57, 0.19, 0.19   # quadrant probabilities of every R-MAT level
CHUNK = 1 << 26                             # edges handled at a time where a temporary would be large


def listed():
    return [
        # the smallest job a serving loop admits, not a power of two: one call's latency
        {"name": "list_1k", "kind": "list", "n": 1021, "layout": "random"},
        # a serving job from the middle of the size range
        {"name": "list_100k", "kind": "list", "n": 100_003, "layout": "random"},
        # the small list ranking configuration: 2^20 elements
        {"name": "list_1m", "kind": "list", "n": 1 << 20, "layout": "random"},
        # the largest serving jobs, ragged size: the successor array just fits L2
        {"name": "list_15m", "kind": "list", "n": 15_000_001, "layout": "random"},
        # the large list ranking configuration: 2^28 elements, random access in HBM
        {"name": "list_268m", "kind": "list", "n": 1 << 28, "layout": "random"},
        # the smallest graph job, of the batched workload's average degree 4
        {"name": "graph_1k", "kind": "graph", "family": "uniform", "n": 1021, "m": 2042},
        # the small components configuration: uniform graph, 2^20 vertices, 2^22 edges
        {"name": "graph_1m", "kind": "graph", "family": "uniform", "n": 1 << 20, "m": 1 << 22},
        # the large components configuration: R-MAT scale 24, edge factor 16
        {"name": "graph_rmat_16m", "kind": "graph", "family": "rmat", "n": 1 << 24, "m": 1 << 28},
        # the paper's list graphs: 8 paths over 8M vertices, sparse and of large diameter
        {"name": "graph_paths_8m", "kind": "graph", "family": "paths", "n": 8_000_008, "m": 8_000_000},
        # the list half of the batched configuration: 2048 lists, sizes log-uniform in 2^8..2^20
        {"name": "lists_2048", "kind": "lists", "count": 2048, "lo": 8, "hi": 20},
        # the graph half of the batched configuration: 2048 graphs of average degree 4
        {"name": "graphs_2048", "kind": "graphs", "count": 2048, "lo": 8, "hi": 20},
        # weighted ranks of a forest of lists (suffix sums per list, no heads given)
        {"name": "forest_10m", "kind": "forest", "n": 10_000_019, "lists": 4096},
    ]


def _log_uniform(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def draw(rng):
    kind = rng.choice(["list"] * 4 + ["graph"] * 4 + ["lists", "graphs", "scan", "forest"])
    if kind == "list":
        return {"kind": kind, "n": _log_uniform(rng, 1 << 10, 1 << 28), "layout": rng.choice(["random"] * 3 + ["ordered"])}
    if kind == "graph":
        family = rng.choice(["uniform", "uniform", "rmat", "paths", "trees"])
        if family == "uniform":
            n = _log_uniform(rng, 1 << 10, 1 << 24)
            # from one edge per vertex up to where a few vertices are still alone (the labels then depend on the edges)
            return {"kind": kind, "family": family, "n": n, "m": int(n * rng.uniform(1.0, 0.35 * math.log(n)))}
        if family == "rmat":
            n = 1 << rng.randint(10, 24)
            return {"kind": kind, "family": family, "n": n, "m": 16 * n - rng.randint(0, n)}
        count, size = rng.randint(2, 16), _log_uniform(rng, 1 << 10, 1_000_001)
        case = {"kind": kind, "family": family, "n": count * size, "m": count * (size - 1)}
        if family == "trees":
            case["degree"] = rng.choice([2, 3, 5, 10, 20])
        return case
    if kind in ("lists", "graphs"):
        return {"kind": kind, "count": _log_uniform(rng, 4, 2000), "lo": 8, "hi": rng.choice([14, 17, 20])}
    n = _log_uniform(rng, 1 << 10, 1 << 26)
    return {"kind": kind, "n": n, "lists": 1 if kind == "scan" else _log_uniform(rng, 1, min(n, 4096))}


def _generator(seed):
    return torch.Generator(device=DEVICE).manual_seed(seed)


def _permutation(n, gen):
    return torch.randperm(n, generator=gen, device=DEVICE).to(torch.int32)


def _chain(order):
    """Successor array of the list that visits `order`; its tail has -1."""
    succ = torch.empty_like(order)
    succ[order[:-1].long()] = order[1:]
    succ[order[-1:].long()] = -1
    return succ


def _list_order(case, gen):
    if case["layout"] == "ordered":   # stored in list order, the head anywhere in the array
        at = torch.randint(0, case["n"], (1,), generator=gen, device=DEVICE)
        return torch.arange(case["n"], device=DEVICE).add_(at).remainder_(case["n"]).to(torch.int32)
    return _permutation(case["n"], gen)


def _batch_sizes(case):
    """floor(2^(lo + (hi - lo) u)) for every instance, the batched workload's recipe.
    The sizes belong to the case; what fills them comes from the seed."""
    u = torch.rand(case["count"], generator=torch.Generator().manual_seed(5), dtype=torch.float64)
    return [int(x) for x in torch.exp2(case["lo"] + (case["hi"] - case["lo"]) * u).floor().tolist()]


def _offsets(sizes):
    off = torch.zeros(len(sizes) + 1, dtype=torch.int64)
    off[1:] = torch.tensor(sizes, dtype=torch.int64).cumsum(0)
    return off


def _forest_bounds(case, seed):
    """List k of the forest takes positions [bounds[k], bounds[k + 1]) of the order."""
    n, lists = case["n"], case["lists"]
    cuts = torch.randperm(n - 1, generator=_generator(seed + 1), device=DEVICE)[:lists - 1] + 1
    edge = torch.tensor([0, n], dtype=torch.int64, device=DEVICE)
    return torch.cat([edge[:1], cuts.sort().values, edge[1:]])


def _values(case, seed):
    return torch.randint(0, 7, (case["n"],), generator=_generator(seed + 2), device=DEVICE, dtype=torch.int32)


def _rmat(n, m, gen):
    scale = n.bit_length() - 1
    src = torch.zeros(m, dtype=torch.int32, device=DEVICE)
    dst = torch.zeros(m, dtype=torch.int32, device=DEVICE)
    for lo in range(0, m, CHUNK):
        s, d = src[lo:lo + CHUNK], dst[lo:lo + CHUNK]
        for _ in range(scale):
            u = torch.rand(s.numel(), generator=gen, device=DEVICE)
            right = ((u >= RMAT_A) & (u < RMAT_A + RMAT_B)) | (u >= RMAT_A + RMAT_B + RMAT_C)
            s.mul_(2).add_(u >= RMAT_A + RMAT_B)
            d.mul_(2).add_(right)
    ids = _permutation(n, gen)
    for lo in range(0, m, CHUNK):
        src[lo:lo + CHUNK] = ids[src[lo:lo + CHUNK].long()]
        dst[lo:lo + CHUNK] = ids[dst[lo:lo + CHUNK].long()]
    return src, dst


def _edges(case, seed):
    gen = _generator(seed)
    n, m, family = case["n"], case["m"], case["family"]
    if family == "uniform":
        src = torch.randint(0, n, (m,), generator=gen, device=DEVICE, dtype=torch.int32)
        return src, torch.randint(0, n, (m,), generator=gen, device=DEVICE, dtype=torch.int32)
    if family == "rmat":
        return _rmat(n, m, gen)
    # n - m components of equal size at random ids
    ids = _permutation(n, gen).view(n - m, -1)
    if family == "paths":
        src, dst = ids[:, 1:], ids[:, :-1]
    else:   # complete trees, `degree` children to a vertex
        i = torch.arange(1, ids.shape[1], device=DEVICE)
        src, dst = ids[:, 1:], ids[:, (i - 1) // case["degree"]]
    return src.reshape(-1).contiguous(), dst.reshape(-1).contiguous()


def _graph_batch(case, seed):
    sizes = _batch_sizes(case)
    voff, eoff = _offsets(sizes), _offsets([2 * s for s in sizes])
    gen = _generator(seed)
    src = torch.empty(int(eoff[-1]), dtype=torch.int32, device=DEVICE)
    dst = torch.empty_like(src)
    for size, at in zip(sizes, eoff.tolist()):
        torch.randint(0, size, (2 * size,), generator=gen, out=src[at:at + 2 * size], device=DEVICE, dtype=torch.int32)
        torch.randint(0, size, (2 * size,), generator=gen, out=dst[at:at + 2 * size], device=DEVICE, dtype=torch.int32)
    return src, dst, eoff, voff


def prepare(case, seed):
    kind = case["kind"]
    if kind == "list":
        order = _list_order(case, _generator(seed))
        return {"kind": kind, "succ": _chain(order), "head": int(order[0])}
    if kind == "graph":
        src, dst = _edges(case, seed)
        return {"kind": kind, "src": src, "dst": dst, "n": case["n"]}
    if kind == "lists":
        sizes, gen = _batch_sizes(case), _generator(seed)
        off = _offsets(sizes)
        succ = torch.empty(int(off[-1]), dtype=torch.int32, device=DEVICE)
        heads = torch.empty(len(sizes), dtype=torch.int32, device=DEVICE)
        for k, at in enumerate(off[:-1].tolist()):
            order = _permutation(sizes[k], gen)
            succ[at:at + sizes[k]] = _chain(order)
            heads[k] = order[0]
        return {"kind": kind, "succ": succ, "off": off.to(DEVICE), "heads": heads}
    if kind == "graphs":
        src, dst, eoff, voff = _graph_batch(case, seed)
        return {"kind": kind, "src": src, "dst": dst, "eoff": eoff.to(DEVICE), "voff": voff.to(DEVICE), "n": int(voff[-1])}
    order = _permutation(case["n"], _generator(seed))
    succ = _chain(order)
    bounds = _forest_bounds(case, seed)
    succ[order[bounds[1:] - 1].long()] = -1
    return {"kind": kind, "succ": succ, "val": _values(case, seed), "head": int(order[0])}


def run(state):
    kind = state["kind"]
    if kind == "list":
        return lrcc.lr_rank(state["succ"], state["head"])
    if kind == "graph":
        return lrcc.cc_label(state["src"], state["dst"], state["n"])
    if kind == "lists":
        return lrcc.lr_rank_batched(state["succ"], state["off"], state["heads"])
    if kind == "graphs":
        return lrcc.cc_label_batched(state["src"], state["dst"], state["eoff"], state["voff"], n_total=state["n"])
    if kind == "scan":
        return lrcc.lr_scan(state["succ"], state["val"], state["head"])
    return lrcc.lr_scan_forest(state["succ"], state["val"])


def work(case):
    """Each input read once and each output written once, 4 bytes an entry (offsets and heads beside them)."""
    kind = case["kind"]
    if kind == "list":
        nbytes = 8 * case["n"]
    elif kind == "graph":
        nbytes = 8 * case["m"] + 4 * case["n"]
    elif kind in ("lists", "graphs"):
        nbytes = (8 if kind == "lists" else 20) * sum(_batch_sizes(case)) + (12 if kind == "lists" else 16) * case["count"]
    else:
        nbytes = 12 * case["n"]
    return {"bytes": nbytes, "flops": 0}


def _smallest_ids(src, dst, n):
    """Smallest id of every vertex's component: the larger of an edge's two roots
    is linked below the smaller, then every vertex jumps to its root, until no
    edge joins two roots. Every id only ever points to a smaller one."""
    parent = torch.arange(n, dtype=torch.int64, device=DEVICE)
    parts = [(src[lo:lo + CHUNK], dst[lo:lo + CHUNK]) for lo in range(0, src.numel(), CHUNK)]
    while parts:
        left = []
        for s, d in parts:
            a, b = parent[s.long()], parent[d.long()]
            open_ = a != b
            if not bool(open_.any()):
                continue
            a, b = a[open_], b[open_]
            parent.scatter_reduce_(0, torch.maximum(a, b), torch.minimum(a, b), "amin")
            left.append((s[open_], d[open_]))
        parts = left
        while True:
            jumped = parent[parent]
            if torch.equal(jumped, parent):
                break
            parent = jumped
    return parent


def exact(case, seed):
    kind = case["kind"]
    if kind == "list":
        n, order = case["n"], _list_order(case, _generator(seed))
        rank = torch.empty(n, dtype=torch.int64, device=DEVICE)
        rank[order.long()] = torch.arange(n - 1, -1, -1, device=DEVICE)
        return rank
    if kind == "graph":
        src, dst = _edges(case, seed)
        return _smallest_ids(src, dst, case["n"])
    if kind == "lists":
        sizes, gen = _batch_sizes(case), _generator(seed)
        off = _offsets(sizes)
        rank = torch.empty(int(off[-1]), dtype=torch.int64, device=DEVICE)
        for size, at in zip(sizes, off.tolist()):
            order = _permutation(size, gen)
            rank[at:at + size][order.long()] = torch.arange(size - 1, -1, -1, device=DEVICE)
        return rank
    if kind == "graphs":
        # one disjoint union: global ids, then each graph's first id taken off
        src, dst, eoff, voff = _graph_batch(case, seed)
        for k, base in enumerate(voff[:-1].tolist()):
            part = slice(int(eoff[k]), int(eoff[k + 1]))
            src[part] += base
            dst[part] += base
        label = _smallest_ids(src, dst, int(voff[-1]))
        for k, base in enumerate(voff[:-1].tolist()):
            label[base:int(voff[k + 1])] -= base
        return label
    # sum along each list from the element to the list's end
    order = _permutation(case["n"], _generator(seed)).long()
    along = _values(case, seed).long()[order]
    before = torch.cat([along.new_zeros(1), along.cumsum(0)])
    bounds = _forest_bounds(case, seed)
    own = torch.searchsorted(bounds, torch.arange(case["n"], device=DEVICE), right=True)
    out = torch.empty_like(along)
    out[order] = before[bounds[own]] - before[:-1]
    return out
