"""Scratch of the plans that a kernel of their own counts: what the admission
query answers."""

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
