"""Counts from several threads at once, on graphs of two sizes: kernels
whose shared memory depends on the graph are launched from both, so a limit
set for one launch must hold for the other."""

import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

from paper_2009_10955_gb300 import native  # noqa: E402
from synth import named_pattern  # noqa: E402
from synth.graphs import er_edges  # noqa: E402


def uniform(n):
    return n, er_edges(n, 4 * n, seed=n)


def stacked(core, n):
    """A clique of `core` vertices and a sparse rest: the largest root matrix has core - 1 rows."""
    a, b = np.triu_indices(core, 1)
    src, dst = er_edges(n, n, seed=core)
    return n, (np.concatenate([a, src]).astype(np.int32), np.concatenate([b, dst]).astype(np.int32))


# pattern, the two graphs: launches whose shared memory goes beyond the default
# 48 KB by different amounts
@pytest.mark.parametrize("pattern,first,second", [
    ("house", uniform(20_000), uniform(12_500)),
    ("c4", uniform(50_000), uniform(12_500)),
    ("c4", uniform(20_000), uniform(12_500)),
    ("c5", uniform(27_000), uniform(25_000)),
    ("k4", stacked(640, 1000), stacked(128, 1000)),
    ("k5", stacked(240, 1000), stacked(129, 1000)),
    ("k7", uniform(8192), uniform(7600)),
])
def test_two_sizes_from_four_threads(pattern, first, second):
    N = native()
    jobs = []
    for n, (src, dst) in (first, second):
        g = N.gp_graph_create_edges(src, dst, n, N.GP_DEGREE_ORDER)
        s = N.gp_schedule(N.gp_pattern_create(named_pattern(pattern)), g, 1)
        s.set_iep(True)
        # 7-cliques through the general kernel's bit matrices as well
        opts = N.make_opts(flags=N.GP_COUNT_LANE_BITMAP) if pattern == "k7" else None
        jobs.append((g, s, opts, N.gp_count(g, s, 0, opts)[1]))
    failures = []

    def work(g, s, opts, expect):
        stream = torch.cuda.Stream()
        try:
            for _ in range(2000):
                got = N.gp_count(g, s, 0, opts, stream)[1]
                if got != expect:
                    failures.append((got, expect))
        except N.GraphPiError as e:
            failures.append(e)

    threads = [threading.Thread(target=work, args=j) for j in jobs + jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failures
