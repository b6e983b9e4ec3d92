"""Graphs on which a plan's own kernel costs more than the general one: the
default count must not take much longer than the general kernel's (forced by
GP_COUNT_NO_CORE, which these graphs' counts hardly feel), and both agree."""

import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

from paper_2009_10955_gb300 import native  # noqa: E402
from synth import named_pattern  # noqa: E402
from synth.graphs import er_edges  # noqa: E402


def joined(*parts):
    return tuple(np.concatenate([p[i] for p in parts]).astype(np.int32) for i in (0, 1))


def late_hubs(hubs, neighbours):
    """A sparse uniform graph and hubs of the largest ids over it."""
    n = 20_000
    rs = np.random.RandomState(hubs)
    return n + hubs, joined(er_edges(n, 80_000, 3), (np.repeat(n + np.arange(hubs), neighbours),
                                                     rs.randint(0, n, hubs * neighbours)))


def best(call):
    call()
    times = []
    for _ in range(5):
        t = time.perf_counter()
        got = call()
        times.append(time.perf_counter() - t)
    return min(times), got


def uniform(n, degree):
    return n, er_edges(n, n * degree // 2, seed=n)


def two_hubs(leaves):
    """A ring of vertices joined to two hubs."""
    leaf = 2 + np.arange(leaves)
    return 2 + leaves, joined((leaf, 2 + (leaf - 1) % leaves), (0 * leaf, leaf), (0 * leaf + 1, leaf))


# these took 18, 110, 36, 5, 4, 4 and 7 times as long as the general kernel
@pytest.mark.parametrize("pattern,ordered,graph", [
    ("k5", False, lambda: late_hubs(500, 3000)),
    ("k6", False, lambda: late_hubs(500, 3000)),
    ("k6", False, lambda: late_hubs(10, 4000)),
    ("house", True, lambda: uniform(1_000_000, 4)),
    ("house", False, lambda: uniform(500_000, 4)),
    ("c4", True, lambda: two_hubs(30_000)),
    ("c4", False, lambda: two_hubs(30_000)),
])
def test_not_much_slower_than_the_general_kernel(pattern, ordered, graph):
    N = native()
    n, (src, dst) = graph()
    g = N.gp_graph_create_edges(src, dst, n, N.GP_DEGREE_ORDER if ordered else 0)
    s = N.gp_schedule(N.gp_pattern_create(named_pattern(pattern)), g, 1)
    s.set_iep(True)
    t, got = best(lambda: N.gp_count(g, s, 0))
    t_general, expect = best(lambda: N.gp_count(g, s, 0, N.make_opts(flags=N.GP_COUNT_NO_CORE)))
    assert got == expect
    assert t < 3 * t_general
