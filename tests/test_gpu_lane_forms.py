"""Plans whose last outer loop runs one candidate per lane, and cycles counted
with root counters: against the oracle on small graphs and against the general
kernel (forced by its options) where lists pass a lane's share, where the core
matrix covers part of the graph only, and at the limits of the counters."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

from paper_2009_10955_gb300 import native  # noqa: E402
from synth import named_pattern  # noqa: E402
from synth.graphs import er_edges, rmat_edges  # noqa: E402

TREE = np.zeros((5, 5), np.uint8)            # two centres: one with two leaves, one with one
for _a, _b in ((0, 1), (0, 2), (0, 3), (3, 4)):
    TREE[_a, _b] = TREE[_b, _a] = 1

PATTERNS = ["c4", "c5", "c6", "c7", "grid3x2", "path5", "tree", "house", "c6chord"]


def adjacency(name):
    return TREE if name == "tree" else named_pattern(name)


def both(N, g, name, iep, top=4):
    """Counts of the top plans by the default path and by the general kernel."""
    s = N.gp_schedule(N.gp_pattern_create(adjacency(name)), g, top)
    s.set_iep(iep)
    general = N.make_opts(flags=N.GP_COUNT_NO_CORE, blocks_per_sm=4)
    return ([N.gp_count(g, s, i)[1] for i in range(len(s))],
            [N.gp_count(g, s, i, general)[1] for i in range(len(s))])


@pytest.mark.parametrize("ordered", [True, False])
@pytest.mark.parametrize("name", PATTERNS)
def test_against_oracle(oracle_lib, name, ordered):
    N = native()
    n, (src, dst) = 70, er_edges(70, 260, seed=5)
    g = N.gp_graph_create_edges(src, dst, n, N.GP_DEGREE_ORDER if ordered else 0)
    expect = oracle_lib.count(adjacency(name), oracle_lib.build_csr(n, src, dst))
    for iep in (True, False):
        mine, general = both(N, g, name, iep)
        assert mine == general == [expect] * len(mine)


def hub_graph(n, m, seed, spokes):
    """Uniform pairs and one vertex joined to `spokes` others."""
    src, dst = er_edges(n, m, seed)
    return (np.concatenate([src, np.full(spokes, 7, np.int32)]),
            np.concatenate([dst, 11 + np.arange(spokes, dtype=np.int32)]))


@pytest.mark.parametrize("ordered", [True, False])
@pytest.mark.parametrize("name", ["c4", "c5", "grid3x2", "tree"])
@pytest.mark.parametrize("n,m,spokes", [(300, 1500, 63), (300, 1500, 65), (300, 3000, 95), (300, 3000, 97),
                                        (9000, 30_000, 40), (9001, 30_000, 200)])
def test_lists_beyond_a_lane(name, n, m, spokes, ordered):
    N = native()
    g = N.gp_graph_create_edges(*hub_graph(n, m, n + m, spokes), n, N.GP_DEGREE_ORDER if ordered else 0)
    for iep in (True, False):
        mine, general = both(N, g, name, iep, 2)
        assert mine == general


@pytest.mark.parametrize("n", [28 * 1024 - 1, 28 * 1024, 28 * 1024 + 1])
def test_counter_limits(n):
    N = native()
    g = N.gp_graph_create_edges(*er_edges(n, 3 * n, seed=2), n, N.GP_DEGREE_ORDER)
    mine, general = both(N, g, "c5", True, 2)
    assert mine == general


@pytest.mark.parametrize("name", ["c5", "c6"])
def test_task_ranges(name):
    N = native()
    n = 1 << 7
    for src, dst in (er_edges(n, 500, seed=8), rmat_edges(7, 6, 0.57, 0.19, 0.19, seed=8)):
        g = N.gp_graph_create_edges(src, dst, n, N.GP_DEGREE_ORDER)
        s = N.gp_schedule(N.gp_pattern_create(named_pattern(name)), g, 2)
        nnz = g.device_csr()[2]
        for a, b in ((0, nnz // 5), (nnz // 5, nnz // 5 + 3), (nnz // 2 + 1, nnz)):
            got = [N.gp_count_raw(g, s, i, task_begin=a, task_end=b) for i in range(len(s))]
            ref = [N.gp_count_raw(g, s, i, task_begin=a, task_end=b, flags=N.GP_COUNT_NO_CORE, blocks_per_sm=4)
                   for i in range(len(s))]
            assert got == ref


def test_batch_mixes_kernels(oracle_lib):
    """Cliques, joins, the House, cycles and general plans in one call."""
    N = native()
    n, (src, dst) = 90, er_edges(90, 420, seed=12)
    g = N.gp_graph_create_edges(src, dst, n, N.GP_DEGREE_ORDER)
    ref = oracle_lib.build_csr(n, src, dst)
    names = ["triangle", "house", "c6", "diamond", "k4", "tailed_triangle", "c5", "tree", "star4", "k5"]
    scheds = []
    for name in names:
        s = N.gp_schedule(N.gp_pattern_create(adjacency(name)), g, 1)
        s.set_iep(True)
        scheds.append(s)
    got = N.gp_count_batch([g] * len(names), scheds)
    assert [int(x) for x in got] == [oracle_lib.count(adjacency(name), ref) for name in names]


def falling_total(degrees, leaves):
    return sum(int(np.prod([int(d) - t for t in range(leaves)], dtype=object)) for d in degrees)


@pytest.mark.parametrize("leaves", [3, 4, 5, 6])
def test_stars_share_one_inner_set(leaves):
    """Three to five inner leaves drawing from one list: a falling factorial."""
    from math import factorial
    N = native()
    src, dst = rmat_edges(7, 8, 0.57, 0.19, 0.19, seed=6)
    g = N.gp_graph_create_edges(src, dst, 1 << 7, N.GP_DEGREE_ORDER)
    rows = g.csr()[0]
    expect = falling_total(np.diff(rows), leaves) // factorial(leaves)
    s = N.gp_schedule(N.gp_pattern_create(named_pattern(f"star{leaves + 1}")), g, 3)
    s.set_iep(True)
    assert [N.gp_count(g, s, i)[1] for i in range(len(s))] == [expect] * len(s)


@pytest.mark.parametrize("ordered", [True, False])
@pytest.mark.parametrize("n,m", [(31, 60), (300, 2500), (5000, 40_000), (70_000, 200_000)])
def test_four_cycles_by_counters(n, m, ordered):
    N = native()
    src, dst = er_edges(n, m, seed=n)
    g = N.gp_graph_create_edges(src, dst, n, N.GP_DEGREE_ORDER if ordered else 0)
    mine, general = both(N, g, "c4", False, 6)
    assert mine == general


@pytest.mark.parametrize("name", ["tailed_triangle", "path4", "diamond", "path3", "star4"])
@pytest.mark.parametrize("n,m,spokes", [(40, 7, 9), (300, 1500, 63), (300, 1500, 70), (9000, 30_000, 400)])
def test_one_task_per_lane(name, n, m, spokes):
    N = native()
    for flags in (N.GP_DEGREE_ORDER, 0):
        g = N.gp_graph_create_edges(*hub_graph(n, m, n + m, spokes), n + spokes + 11, flags)
        for iep in (True, False):
            mine, general = both(N, g, name, iep, 3)
            assert mine == general
