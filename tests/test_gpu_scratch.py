"""Scratch of the plans that a kernel of their own counts: what the admission
query answers, and counts on a device with little memory left."""

from contextlib import contextmanager

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

from paper_2009_10955_gb300 import native  # noqa: E402
from synth import named_pattern  # noqa: E402
from synth.graphs import er_edges  # noqa: E402


def plan(N, graph, pattern):
    s = N.gp_schedule(N.gp_pattern_create(named_pattern(pattern)), graph, 1)
    s.set_iep(True)
    return s


def bipartite(n, planted):
    """Every vertex of one half joined to every one of the other, and
    `planted` vertices of the first half to one another."""
    a, b = np.meshgrid(np.arange(n), n + np.arange(n), indexing="ij")
    x, y = np.triu_indices(planted, 1)
    return 2 * n, (np.concatenate([a.ravel(), x]).astype(np.int32), np.concatenate([b.ravel(), y]).astype(np.int32))


def uniform(n, degree):
    return n, er_edges(n, n * degree // 2, seed=n)


# counters in global memory (0.4 MB a block), root matrices (0.3 and 0.8 MB):
# the answer is that of the kernel that time slices run
@pytest.mark.parametrize("pattern,graph", [
    ("house", lambda: uniform(100_003, 20)), ("c4", lambda: uniform(100_003, 20)),
    ("k5", lambda: bipartite(1000, 8)), ("k6e", lambda: bipartite(1000, 8)),
])
def test_query_answers_for_time_slices(pattern, graph):
    N = native()
    n, (src, dst) = graph()
    g = N.gp_graph_create_edges(src, dst, n, N.GP_DEGREE_ORDER)
    s = plan(N, g, pattern)
    assert N.gp_count_scratch_bytes(g, s, 0) == N.gp_count_scratch_bytes(g, s, 0, N.make_opts(budget_cycles=1 << 30))


@contextmanager
def free_megabytes(left):
    """All device memory but `left` megabytes taken (and never touched)."""
    torch.cuda.empty_cache()
    held = []
    try:
        while True:
            free = torch.cuda.mem_get_info()[0] - (left << 20)
            if free < 4 << 20:
                break
            held.append(torch.empty(min(free, 16 << 30) >> 21 << 21, dtype=torch.uint8, device="cuda"))
        yield
    finally:
        held.clear()
        torch.cuda.empty_cache()


# root matrices of 2500 rows take 1.7 MB a block (1.6 MB of K4 plans with two
# inner vertices), 0.26 GB with one block an SM: with 300 MB left that is more
# than half of it and the general kernel counts, with 700 MB the grid shrinks.
# Counters of a million vertices take 4 MB a block
@pytest.mark.parametrize("pattern,graph,left", [
    ("k4", lambda: bipartite(2500, 8), 300), ("k5", lambda: bipartite(2500, 8), 300),
    ("k5", lambda: bipartite(2500, 8), 700), ("k6", lambda: bipartite(2500, 8), 300),
    ("k6e", lambda: bipartite(2500, 8), 300), ("k6e", lambda: bipartite(2500, 8), 700),
    ("house", lambda: uniform(1_000_003, 16), 60), ("house", lambda: uniform(1_000_003, 16), 800),
    ("c4", lambda: uniform(1_000_003, 24), 300), ("c4", lambda: uniform(1_000_003, 24), 3000),
])
def test_counts_with_little_memory_left(pattern, graph, left):
    N = native()
    n, (src, dst) = graph()
    g = N.gp_graph_create_edges(src, dst, n, N.GP_DEGREE_ORDER)
    s = plan(N, g, pattern)
    t = plan(N, g, "triangle")
    expect = N.gp_count(g, s, 0)
    triangles = N.gp_count(g, t, 0)[1]
    with free_megabytes(left):
        assert N.gp_count(g, s, 0) == expect
        assert N.gp_count_batch([g, g, g], [s, t, s], [0] * 3).tolist() == [expect[1], triangles, expect[1]]


def test_a_failed_call_leaves_no_error_for_the_next():
    N = native()
    n, (src, dst) = uniform(2000, 20)
    g = N.gp_graph_create_edges(src, dst, n, N.GP_DEGREE_ORDER)
    s = plan(N, g, "triangle")
    expect = N.gp_count(g, s, 0)
    many = torch.zeros(1 << 25, dtype=torch.int32, device="cuda")
    with free_megabytes(300):
        with pytest.raises(N.GraphPiError):
            N.gp_graph_create_edges(many, many, 1000, N.GP_DEVICE_PTRS)
        assert N.gp_count(g, s, 0) == expect


# seven labels: fourteen sets of up to 40,006 vertices a warp and a spare one,
# 2.9 GB with one block an SM; the four sets of the prefixes alone take 1 GB
def test_labelled_count_and_list_with_little_memory_left():
    N = native()
    leaves = 40_000
    a, b = np.triu_indices(7, 1)
    src = np.concatenate([a, np.zeros(leaves)]).astype(np.int32)
    dst = np.concatenate([b, 7 + np.arange(leaves)]).astype(np.int32)
    g = N.gp_graph_create_edges(src, dst, 7 + leaves, N.GP_DEGREE_ORDER)
    N.gp_graph_set_labels(g, (np.arange(7 + leaves) % 7).astype(np.int32))
    s = N.gp_schedule(N.gp_pattern_create_labeled(named_pattern("k7"), list(range(7))), g, 1)
    out = torch.zeros((16, 7), dtype=torch.int32, device="cuda")
    with free_megabytes(2600):
        assert N.gp_count(g, s, 0) == (N.GP_OK, 1)
        assert N.gp_list(g, s, 0, 0, 0, out, 16)[:2] == (N.GP_OK, 1)
