"""Clique counts on local bit matrices against the oracle, at the sizes where
the kernel changes its form: matrices of one 32-bit word and of four, roots
counted by a warp and by a block, rows with more neighbours than a warp's
matrix holds, roots whose matrix does not fit shared memory, every clique
size, graphs with and without the degree order, task ranges."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

from math import comb  # noqa: E402

from paper_2009_10955_gb300 import native  # noqa: E402
from synth import named_pattern  # noqa: E402
from synth.graphs import rmat_edges  # noqa: E402


def dense_edges(n, p, seed):
    rs = np.random.RandomState(seed)
    a, b = np.triu_indices(n, 1)
    keep = rs.rand(len(a)) < p
    return a[keep].astype(np.int32), b[keep].astype(np.int32)


def count(graph, pattern, **opts):
    N = native()
    s = N.gp_schedule(N.gp_pattern_create(named_pattern(pattern)), graph, 1)
    return N.gp_count(graph, s, 0, N.make_opts(**opts) if opts else None)[1]


# n vertices all joined: root v has |U| = v, so n crosses the widths of the
# matrices (32 rows, 128 rows, the shared-memory limit 640)
@pytest.mark.parametrize("n", [2, 3, 31, 32, 33, 34, 64, 65, 127, 128, 129, 130, 160, 257])
@pytest.mark.parametrize("k", [3, 4, 5, 6, 7])
def test_complete_graph(n, k):
    N = native()
    g = N.gp_graph_create_edges(*dense_edges(n, 2.0, 0), n, N.GP_DEGREE_ORDER)
    assert count(g, "triangle" if k == 3 else f"k{k}") == comb(n, k)


@pytest.mark.parametrize("n,k", [(640, 5), (641, 4), (641, 5)])
def test_complete_graph_beyond_shared_memory(n, k):
    N = native()
    g = N.gp_graph_create_edges(*dense_edges(n, 2.0, 0), n, N.GP_DEGREE_ORDER)
    assert count(g, f"k{k}") == comb(n, k)


@pytest.mark.parametrize("ordered", [True, False])
@pytest.mark.parametrize("pattern", ["triangle", "k4", "k5", "k6"])
@pytest.mark.parametrize("name,n,edges", [("dense", 150, lambda: dense_edges(150, 0.5, 3)),
                                          ("rmat", 1 << 9, lambda: rmat_edges(9, 8, 0.57, 0.19, 0.19, seed=9))])
def test_against_oracle(oracle_lib, pattern, name, n, edges, ordered):
    N = native()
    src, dst = edges()
    g = N.gp_graph_create_edges(src, dst, n, N.GP_DEGREE_ORDER if ordered else 0)
    ref = oracle_lib.build_csr(n, src, dst)
    k = len(named_pattern(pattern))
    chain = [(a, a + 1) for a in range(k - 1)]
    expect = oracle_lib.count_restricted(named_pattern(pattern), list(range(k)), chain, ref)
    assert count(g, pattern) == expect
    # ranges of tasks add up to the whole count, whatever they cut
    nnz = g.device_csr()[2]
    cuts = [0, 1, nnz // 3, nnz // 3 + 5, 2 * nnz // 3, nnz]
    assert sum(count(g, pattern, task_begin=a, task_end=b) for a, b in zip(cuts, cuts[1:])) == expect


def test_general_kernel_agrees_on_ranges():
    """A range's count is the plan's own: the general kernel (core matrix off)
    gives the same number for the same tasks."""
    N = native()
    src, dst = rmat_edges(12, 16, 0.57, 0.19, 0.19, seed=4)
    g = N.gp_graph_create_edges(src, dst, 1 << 12, N.GP_DEGREE_ORDER)
    nnz = g.device_csr()[2]
    for pattern in ("triangle", "k4", "k5"):
        for a, b in ((0, nnz // 7), (nnz // 7, nnz // 2), (nnz // 2, nnz // 2 + 33)):
            assert count(g, pattern, task_begin=a, task_end=b) == \
                count(g, pattern, task_begin=a, task_end=b, flags=N.GP_COUNT_NO_CORE)


# without the degree order: hubs of the largest ids whose smaller neighbours
# have lists much shorter than their rows (looked up in the row's vertices), as
# long as them (pairs probed) and in between; roots beyond shared memory
@pytest.mark.parametrize("hubs,rows,low", [(3, 65, 300), (40, 300, 600), (30, 700, 900), (20, 1400, 2000)])
@pytest.mark.parametrize("k", [5, 6, 7])
def test_hubs_of_the_largest_ids(k, hubs, rows, low):
    N = native()
    rs = np.random.RandomState(rows)
    core = np.arange(60)                       # a dense part, so that there are cliques
    a, b = dense_edges(60, 0.7, rows)
    src = np.concatenate([a, rs.randint(0, low, 3 * low), np.repeat(low + np.arange(hubs), rows + 60)])
    dst = np.concatenate([b, rs.randint(0, low, 3 * low)] +
                         [np.concatenate([core, rs.choice(low, rows, replace=False)]) for _ in range(hubs)])
    g = N.gp_graph_create_edges(src.astype(np.int32), dst.astype(np.int32), low + hubs)
    assert count(g, f"k{k}") == count(g, f"k{k}", flags=N.GP_COUNT_NO_CORE) > 0


# roots of more smaller neighbours than a matrix in shared memory has rows,
# random ones: over ranges of tasks and whole, against the general kernel
@pytest.mark.parametrize("n,p", [(700, 0.25), (1300, 0.1)])
@pytest.mark.parametrize("k", [4, 5, 6, 7])
def test_random_matrices_beyond_shared_memory(k, n, p):
    N = native()
    rs = np.random.RandomState(n)
    a, b = dense_edges(n, p, n)
    hub = np.repeat(n + np.arange(4), n)       # joined to every vertex, the last ids in id order
    src = np.concatenate([a, hub]).astype(np.int32)
    dst = np.concatenate([b, np.tile(rs.permutation(n), 4)]).astype(np.int32)
    g = N.gp_graph_create_edges(src, dst, n + 4)
    assert count(g, f"k{k}") == count(g, f"k{k}", flags=N.GP_COUNT_NO_CORE)
