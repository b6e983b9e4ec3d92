"""House counts with the sums exchanged, against closed forms, the oracle and
the general kernel: counters in shared memory (two block sizes) and in global
memory, lists longer than a warp walks, every House plan, ordered or not."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

from math import comb  # noqa: E402

from paper_2009_10955_gb300 import native  # noqa: E402
from synth import named_pattern  # noqa: E402
from synth.graphs import er_edges, rmat_edges  # noqa: E402


def plans(N, graph, top=12):
    s = N.gp_schedule(N.gp_pattern_create(named_pattern("house")), graph, top)
    s.set_iep(True)
    return s


@pytest.mark.parametrize("n", [4, 5, 6, 33, 130])
def test_complete_graph(n):
    N = native()
    a, b = np.triu_indices(n, 1)
    g = N.gp_graph_create_edges(a.astype(np.int32), b.astype(np.int32), n, N.GP_DEGREE_ORDER)
    assert N.gp_count(g, plans(N, g), 0)[1] == 60 * comb(n, 5)      # 5! / |Aut|, |Aut| = 2


@pytest.mark.parametrize("ordered", [True, False])
def test_every_plan_against_oracle(oracle_lib, ordered):
    N = native()
    src, dst = rmat_edges(8, 8, 0.57, 0.19, 0.19, seed=3)
    g = N.gp_graph_create_edges(src, dst, 1 << 8, N.GP_DEGREE_ORDER if ordered else 0)
    expect = oracle_lib.count(named_pattern("house"), oracle_lib.build_csr(1 << 8, src, dst))
    s = plans(N, g, 40)
    assert [N.gp_count(g, s, i)[1] for i in range(len(s))] == [expect] * len(s)
    # ranges of tasks go to the general kernel; they add up to the same
    nnz = g.device_csr()[2]
    div = s.iep(0)[1]
    cuts = [0, 5, nnz // 2, nnz]
    assert sum(N.gp_count_raw(g, s, 0, task_begin=a, task_end=b)[1] for a, b in zip(cuts, cuts[1:])) == expect * div


@pytest.mark.parametrize("n,m", [(28_159, 120_000), (28_161, 120_000), (57_344, 200_000), (57_345, 200_000)])
@pytest.mark.parametrize("hub", [False, True])
def test_against_general_kernel(n, m, hub):
    N = native()
    src, dst = er_edges(n, m, seed=n)
    if hub:                                   # one vertex joined to 3000 others: a list the block walks
        src = np.concatenate([src, np.full(3000, n // 2, np.int32)])
        dst = np.concatenate([dst, np.arange(3000, dtype=np.int32) * 9])
    for flags in (N.GP_DEGREE_ORDER, 0):
        g = N.gp_graph_create_edges(src, dst, n, flags)
        s = plans(N, g, 1)
        assert N.gp_count(g, s, 0) == N.gp_count(g, s, 0, N.make_opts(flags=N.GP_COUNT_NO_CORE))


# (0 > 1 > 2, 0 > 3) passes the validation on the complete graph (3 of 24
# orders) but not on every 4-cycle: it counts some twice and some never
@pytest.mark.parametrize("res", [[(0, 1), (1, 2), (0, 3)], [(1, 0), (2, 1), (3, 0)], [(0, 1), (0, 2), (0, 3), (1, 3)]])
def test_four_cycle_under_an_explicit_restriction_set(oracle_lib, res):
    N = native()
    src, dst = rmat_edges(8, 8, 0.57, 0.19, 0.19, seed=3)
    g = N.gp_graph_create_edges(src, dst, 1 << 8)
    s = N.gp_schedule_explicit(N.gp_pattern_create(named_pattern("c4")), [0, 1, 2, 3], res)
    expect = oracle_lib.count_restricted(named_pattern("c4"), [0, 1, 2, 3], res,
                                         oracle_lib.build_csr(1 << 8, src, dst))
    assert N.gp_count(g, s, 0)[1] == expect
    nnz = g.device_csr()[2]
    assert sum(N.gp_count(g, s, 0, N.make_opts(task_begin=a, task_end=b))[1]
               for a, b in ((0, nnz // 3), (nnz // 3, nnz))) == expect


# lists that the block walks: two of them, more than it can set aside at once,
# counters in shared and in global memory, with and without the degree order
@pytest.mark.parametrize("ordered", [True, False])
@pytest.mark.parametrize("leaves", [511, 513, 3000])
def test_four_cycles_of_two_hubs(leaves, ordered):
    N = native()
    leaf = np.arange(2, 2 + leaves, dtype=np.int32)
    g = N.gp_graph_create_edges(np.concatenate([0 * leaf, 0 * leaf + 1]), np.concatenate([leaf, leaf]), 2 + leaves,
                                N.GP_DEGREE_ORDER if ordered else 0)
    s = N.gp_schedule(N.gp_pattern_create(named_pattern("c4")), g, 1)
    assert N.gp_count(g, s, 0)[1] == comb(leaves, 2)


@pytest.mark.parametrize("ordered", [True, False])
@pytest.mark.parametrize("core,n,m", [(250, 900, 3000), (800, 2000, 3000), (800, 57_400, 500_000)])
def test_four_cycles_with_many_long_lists(core, n, m, ordered):
    N = native()
    rs = np.random.RandomState(core)
    a, b = np.triu_indices(core, 1)
    keep = rs.rand(len(a)) < 0.9
    src, dst = er_edges(n, m, seed=n)
    hubs = np.repeat(np.arange(core), 400)     # the core's lists exceed 512 entries
    src = np.concatenate([src, a[keep], hubs]).astype(np.int32)
    dst = np.concatenate([dst, b[keep], rs.randint(0, n, 400 * core)]).astype(np.int32)
    order = rs.permutation(n).astype(np.int32)
    g = N.gp_graph_create_edges(order[src], order[dst], n, N.GP_DEGREE_ORDER if ordered else 0)
    s = N.gp_schedule(N.gp_pattern_create(named_pattern("c4")), g, 1)
    assert N.gp_count(g, s, 0) == N.gp_count(g, s, 0, N.make_opts(flags=N.GP_COUNT_NO_CORE))
