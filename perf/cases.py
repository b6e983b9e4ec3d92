"""The measured work: pattern counts, batches, listings, directed and labelled
counts and graph builds, each through the public entry points.

A case names what is done (``op``), the graph family and its size, and the
pattern. Graphs are the three families of the workloads: uniform G(n, m),
R-MAT with a/b/c/d = .57/.19/.19/.05, and Chung-Lu with exponent 2.1; they are
drawn here on the GPU from the seed, with self loops and repeated pairs left
in, since removing them is the graph build's work. Counts run the model's
first plan, in its inclusion-exclusion form where the case says so and the
plan has one.
"""

import math

import numpy as np
import torch

from paper_2009_10955_gb300 import native
from synth.patterns import named_pattern, random_pattern_set

RMAT = (0.57, 0.19, 0.19)


# ------------------------------------------------------------------- cases

def listed():
    return [
        # one small query answered at once: launch and call latency
        dict(name="gnm_house", op="count", family="gnm", n=2000, pairs=20000, pattern="house", iep=True),
        # a deep query on the same graph: a 6-cycle's loops are not pruned by triangles
        dict(name="gnm_c6", op="count", family="gnm", n=2000, pairs=20000, pattern="c6", iep=True),
        # the benchmark's graph: triangle, 4-clique and 5-clique of a skewed
        # graph of a million vertices
        dict(name="rmat20_triangle", op="count", family="rmat", n=1 << 20, pairs=16 << 20, pattern="triangle",
             iep=False),
        dict(name="rmat20_k4", op="count", family="rmat", n=1 << 20, pairs=16 << 20, pattern="k4", iep=False),
        dict(name="rmat20_k5", op="count", family="rmat", n=1 << 20, pairs=16 << 20, pattern="k5", iep=False),
        # House under skew, at a size whose count ends in a fraction of a second
        dict(name="rmat14_house", op="count", family="rmat", n=1 << 14, pairs=16 << 14, pattern="house", iep=True),
        # the 6-clique minus an edge on a power-law graph: load balance
        dict(name="cl1m_k6e", op="count", family="cl", n=1_000_000, pairs=8_750_000, pattern="k6e", iep=True),
        # many patterns under their three best plans in one call
        dict(name="batch_rmat10", op="batch", family="rmat", n=1 << 10, pairs=16 << 10, patterns=16, k_lo=3, k_hi=5,
             top=3, iep=True),
        # the triangles themselves, as vertex triples in a device buffer
        dict(name="list_rmat16", op="list", family="rmat", n=1 << 16, pairs=16 << 16, pattern="triangle",
             capacity=16 << 20),
        # the House with a label on every vertex
        dict(name="labeled_rmat13", op="labeled", family="rmat", n=1 << 13, pairs=16 << 13, pattern="house",
             labels=8),
        # feed-forward loops of a digraph
        dict(name="ffl_rmat14", op="directed", family="rmat", n=1 << 14, pairs=16 << 14, pattern="ffl"),
        # from raw pairs to the resident graph, once per data set
        dict(name="build_rmat20", op="build", family="rmat", n=1 << 20, pairs=16 << 20),
    ]


# Undirected pattern -> (graph family, smallest n, largest n): the sizes at
# which one count stays below the largest listed case.
COUNT_RANGES = [
    ("triangle", "rmat", 1 << 8, 1 << 20), ("triangle", "cl", 10_000, 1_000_000), ("triangle", "gnm", 200, 200_000),
    ("k4", "rmat", 1 << 8, 1 << 20), ("k4", "cl", 10_000, 1_000_000), ("k4", "gnm", 200, 200_000),
    ("k5", "rmat", 1 << 8, 1 << 20), ("k5", "cl", 10_000, 1_000_000),
    ("k6", "rmat", 1 << 8, 1 << 16), ("k6e", "cl", 10_000, 1_000_000), ("k6e", "rmat", 1 << 8, 1 << 13),
    ("diamond", "rmat", 1 << 8, 1 << 18), ("diamond", "cl", 10_000, 1_000_000),
    ("tailed_triangle", "rmat", 1 << 8, 1 << 16), ("c4", "rmat", 1 << 8, 1 << 15), ("c4", "gnm", 200, 200_000),
    ("house", "gnm", 200, 200_000), ("house", "rmat", 1 << 8, 1 << 14), ("house", "cl", 10_000, 40_000),
    ("three_ears", "rmat", 1 << 8, 1 << 15), ("star5", "rmat", 1 << 8, 1 << 16),
    ("c5", "gnm", 200, 20_000), ("c6", "gnm", 200, 2000), ("grid3x2", "gnm", 200, 4000),
]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["count"] * 6 + ["batch", "list", "labeled", "directed", "build"])
    if op == "count":
        pattern, family, lo, hi = rng.choice(COUNT_RANGES)
        n = _between(rng, lo, hi)
        case = dict(op=op, family=family, n=n, pattern=pattern, iep=rng.random() < 0.7)
        if family == "gnm":
            case["ordered"] = rng.random() < 0.8
        if pattern in ("house", "three_ears", "star5", "k6e", "diamond", "tailed_triangle"):
            case["iep"] = True
    elif op == "batch":
        n = _between(rng, 1 << 7, 1 << 10)
        case = dict(op=op, family="rmat", n=n, patterns=rng.randint(2, 16), k_lo=3, k_hi=rng.randint(3, 5),
                    top=rng.randint(1, 3), iep=True)
    elif op == "list":
        # a buffer that may be too small for all of them: a call then ends at
        # the last task that fits
        pattern, hi, per_pair = rng.choice([("triangle", 1 << 16, 16), ("k4", 1 << 12, 64), ("c4", 1 << 10, 256)])
        n = _between(rng, 1 << 7, hi)
        case = dict(op=op, family="rmat", n=n, pattern=pattern, capacity=per_pair * 16 * n)
    elif op == "labeled":
        pattern, hi = rng.choice([("triangle", 1 << 16), ("house", 1 << 12), ("k4", 1 << 13)])
        n = _between(rng, 1 << 8, hi)
        case = dict(op=op, family="rmat", n=n, pattern=pattern, labels=rng.randint(4, 16))
    elif op == "directed":
        pattern, hi = rng.choice([("ffl", 1 << 14), ("cycle3", 1 << 14), ("bifan", 1 << 11)])
        n = _between(rng, 1 << 8, hi)
        case = dict(op=op, family="rmat", n=n, pattern=pattern)
    else:
        case = dict(op=op, family=rng.choice(["rmat", "gnm", "cl"]), n=_between(rng, 1 << 10, 1 << 20))
    per_vertex = {"gnm": (4.0, 12.0), "rmat": (6.0, 16.0), "cl": (6.0, 8.75)}[case["family"]]
    case["pairs"] = int(case["n"] * rng.uniform(*per_vertex))
    return case


# ------------------------------------------------------------------- inputs

def _pairs(case, seed):
    """(src, dst): int32 device tensors of the case's raw pairs."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(0x5EED0000 + int(seed))
    n, m, family = case["n"], case["pairs"], case["family"]
    if family == "gnm":
        uv = torch.randint(0, n, (2, m), generator=gen, device="cuda", dtype=torch.int32)
        return uv[0].contiguous(), uv[1].contiguous()
    if family == "rmat":
        # quadrant by quadrant; a size that is no power of two folds the top
        # ids back, which keeps the skew
        a, b, c = RMAT
        src = torch.zeros(m, dtype=torch.int32, device="cuda")
        dst = torch.zeros(m, dtype=torch.int32, device="cuda")
        for _ in range(max(1, (n - 1).bit_length())):
            u = torch.rand(m, generator=gen, device="cuda")
            src = 2 * src + (u >= a + b).int()
            dst = 2 * dst + (((u >= a) & (u < a + b)) | (u >= a + b + c)).int()
        return src % n, dst % n
    # Chung-Lu: weights (i + i0)^(-1/1.1), the largest 20000 sqrt(n / 4e6)
    # times over a mean of 17.5, endpoints by inverse CDF
    i = torch.arange(n, dtype=torch.float64, device="cuda")
    target = 20000.0 * math.sqrt(n / 4_000_000) / 17.5
    lo, hi = 1e-6, float(n)
    for _ in range(60):
        mid = math.sqrt(lo * hi)
        w = (i + mid).pow(-1.0 / 1.1)
        if float(w[0] / w.mean()) > target:
            lo = mid
        else:
            hi = mid
    cdf = torch.cumsum((i + math.sqrt(lo * hi)).pow(-1.0 / 1.1), 0)
    u = torch.rand(2, m, generator=gen, device="cuda", dtype=torch.float64) * cdf[-1]
    v = torch.searchsorted(cdf, u, right=True).clamp_(max=n - 1).int()
    return v[0].contiguous(), v[1].contiguous()


def _directed_pattern(name):
    arcs = {"ffl": (3, [(0, 1), (1, 2), (0, 2)]), "cycle3": (3, [(0, 1), (1, 2), (2, 0)]),
            "bifan": (4, [(0, 2), (0, 3), (1, 2), (1, 3)])}
    k, lst = arcs[name]
    adj = np.zeros((k, k), np.uint8)
    for a, b in lst:
        adj[a, b] = 1
    return adj


def prepare(case, seed):
    N = native()
    stream = torch.cuda.current_stream()
    src, dst = _pairs(case, seed)
    op, n = case["op"], case["n"]
    state = {"op": op, "N": N, "stream": stream}
    if op == "build":
        state.update(src=src, dst=dst, n=n)
        state["cols"] = torch.zeros(2 * case["pairs"], dtype=torch.int32, device="cuda")
        return state
    if op == "directed":
        state["graph"] = N.gp_dgraph_create(src, dst, n, N.GP_DEVICE_PTRS, stream)
        state["pattern"] = N.gp_dpattern_create(_directed_pattern(case["pattern"]))
        return state
    order = N.GP_DEGREE_ORDER if case.get("ordered", True) else 0
    graph = N.gp_graph_create_edges(src, dst, n, N.GP_DEVICE_PTRS | order, stream)
    state["graph"] = graph
    if op == "batch":
        # the same patterns for every seed: a service's queries over new graphs
        adjs = random_pattern_set(case["patterns"], case["k_lo"], case["k_hi"], 0.5, 7)
        scheds, idx = [], []
        for adj in adjs:
            s = N.gp_schedule(N.gp_pattern_create(adj), graph, case["top"], stream)
            s.set_iep(case["iep"])
            scheds += [s] * len(s)
            idx += list(range(len(s)))
        state.update(graphs=[graph] * len(idx), scheds=scheds, idx=idx)
        return state
    adj = named_pattern(case["pattern"])
    if op == "labeled":
        rs = np.random.RandomState(int(seed) % (1 << 31))
        N.gp_graph_set_labels(graph, rs.randint(0, case["labels"], n).astype(np.int32), stream)
        labels = [a % 3 for a in range(adj.shape[0])]
        state["sched"] = N.gp_schedule(N.gp_pattern_create_labeled(adj, labels), graph, 1, stream)
        return state
    state["sched"] = N.gp_schedule(N.gp_pattern_create(adj), graph, 1, stream)
    if op == "list":
        state["capacity"] = case["capacity"]
        state["out"] = torch.zeros((case["capacity"], adj.shape[0]), dtype=torch.int32, device="cuda")
        return state
    state["sched"].set_iep(case["iep"])
    return state


class _DeviceArray:
    """A device array of the graph as torch can take it; it keeps the graph."""

    def __init__(self, graph, address, length, kind):
        self.graph = graph
        self.__cuda_array_interface__ = {"shape": (length,), "typestr": kind, "data": (address, False), "version": 3,
                                         "strides": None}


def run(state):
    N, stream, op = state["N"], state["stream"], state["op"]
    if op == "count" or op == "labeled":
        return N.gp_count(state["graph"], state["sched"], 0, None, stream)[1]
    if op == "batch":
        return N.gp_count_batch(state["graphs"], state["scheds"], state["idx"], None, stream).astype(np.int64)
    if op == "list":
        _, written, after = N.gp_list(state["graph"], state["sched"], 0, 0, 0, state["out"], state["capacity"], stream)
        return written, after, state["out"]
    if op == "directed":
        return N.gp_dcount(state["graph"], state["pattern"], stream=stream)
    graph = N.gp_graph_create_edges(state["src"], state["dst"], state["n"], N.GP_DEVICE_PTRS | N.GP_DEGREE_ORDER,
                                    stream)
    rows, cols, entries = graph.device_csr()
    # the neighbour lists go into the caller's buffer, whose size the pairs bound
    state["cols"][:entries].copy_(torch.as_tensor(_DeviceArray(graph, cols, entries, "<i4"), device="cuda"))
    return torch.as_tensor(_DeviceArray(graph, rows, state["n"] + 1, "<i8"), device="cuda"), state["cols"]


# --------------------------------------------------------------------- work

def work(case):
    """Bytes: the graph's rows (8-byte offsets, 4-byte ids, both directions of
    an undirected edge, every pair taken as one edge) read once and the
    results written once; a build reads the pairs and writes the rows. No
    floating-point operations are in the definition of a count."""
    n, m = case["n"], case["pairs"]
    rows = 8 * (n + 1) + 8 * m
    if case["op"] == "build":
        return {"bytes": 8 * m + rows, "flops": 0}
    if case["op"] == "directed":
        return {"bytes": 8 * (n + 1) + 4 * m + 8, "flops": 0}
    if case["op"] == "labeled":
        return {"bytes": rows + 4 * n + 8, "flops": 0}
    if case["op"] == "list":
        # every written tuple: between a third and all of the buffer
        return {"bytes": rows + 4 * case["capacity"], "flops": 0}
    return {"bytes": rows + 8 * case.get("patterns", 1), "flops": 0}


# -------------------------------------------------------------------- exact

def _simple(case, seed):
    """Sorted unique directed keys u * n + v of the simple undirected graph,
    relabelled by non-increasing degree (ties by id)."""
    n = case["n"]
    src, dst = (x.long() for x in _pairs(case, seed))
    keep = src != dst
    src, dst = src[keep], dst[keep]
    keys = torch.unique(torch.cat([src * n + dst, dst * n + src]))
    deg = torch.bincount(keys // n, minlength=n)
    order = torch.argsort(-deg, stable=True)
    rank = torch.empty_like(order)
    rank[order] = torch.arange(n, device="cuda")
    return torch.sort(rank[keys // n] * n + rank[keys % n]).values


def _has(keys, wanted):
    if keys.numel() == 0:
        return torch.zeros_like(wanted, dtype=torch.bool)
    at = torch.searchsorted(keys, wanted).clamp_(max=keys.numel() - 1)
    return keys[at] == wanted


def _closed_wedges(keys, n, chunk=1 << 25):
    """Pairs of arcs a -> b, b -> c of the sorted keys with the arc a -> c."""
    a, b = keys // n, keys % n
    start = torch.searchsorted(keys, torch.arange(n + 1, device="cuda") * n)
    size = start[b + 1] - start[b]
    upto = torch.cumsum(size, 0)
    total, found = int(upto[-1]) if keys.numel() else 0, 0
    for lo in range(0, total, chunk):
        w = torch.arange(lo, min(total, lo + chunk), device="cuda")
        e = torch.searchsorted(upto, w, right=True)
        c = b[start[b[e]] + (w - (upto[e] - size[e]))]
        found += int(_has(keys, a[e] * n + c).sum())
    return found


def exact(case, seed):
    op, n = case["op"], case["n"]
    if op == "build":
        keys = _simple(case, seed)
        cols = torch.zeros(2 * case["pairs"], dtype=torch.int32, device="cuda")
        cols[:keys.numel()] = (keys % n).int()
        return torch.searchsorted(keys, torch.arange(n + 1, device="cuda") * n), cols
    if op == "directed" and case["pattern"] == "ffl":
        src, dst = (x.long() for x in _pairs(case, seed))
        return _closed_wedges(torch.unique((src * n + dst)[src != dst]), n)
    if op != "count" or case["pattern"] not in ("triangle", "house", "c4"):
        return None
    keys = _simple(case, seed)
    u, v = keys // n, keys % n
    if case["pattern"] == "triangle":
        return _closed_wedges(keys[u > v], n)
    if n > 4096:
        return None
    u, v = u.cpu(), v.cpu()
    A = torch.zeros(n, n, dtype=torch.float64)
    A[u, v] = 1.0
    A2 = A @ A
    deg = A.sum(1)
    if case["pattern"] == "c4":       # every 4-cycle has two diagonals
        pairs = A2.triu(1)
        return int((pairs * (pairs - 1) / 2).sum()) // 2
    # House: an edge (u, v), an apex among the t common neighbours, and a path
    # u-a-b-v that avoids u, v and the apex
    paths = (A2 @ A)[u, v] - deg[u] - deg[v] + 1
    t = A2[u, v]
    return int((t * paths - 2 * t * t + 2 * t).sum()) // 2
