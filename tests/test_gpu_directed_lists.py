"""Directed counts where the kernel changes its form: last-depth lists at and
beyond the length that goes to a whole warp, tasks at the edges of a warp's
32, arcs both ways, restrictions from above and below."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

from paper_2009_10955_gb300 import native  # noqa: E402


def pat(k, arcs):
    a = np.zeros((k, k), np.uint8)
    for x, y in arcs:
        a[x, y] = 1
    return a


def fan(leaves):
    """Vertices 0 and 1 joined both ways, both pointing at every leaf."""
    x = np.arange(leaves, dtype=np.int32) + 2
    src = np.concatenate([[0, 1], np.zeros(leaves), np.ones(leaves)]).astype(np.int32)
    dst = np.concatenate([[1, 0], x, x]).astype(np.int32)
    return src, dst, leaves + 2


@pytest.mark.parametrize("leaves", [1, 7, 8, 9, 31, 32, 33, 255, 256, 257, 600])
def test_fan_closed_forms(leaves):
    N = native()
    src, dst, n = fan(leaves)
    g = N.gp_dgraph_create(src, dst, n)

    def count(k, arcs):
        return N.gp_dcount(g, N.gp_dpattern_create(pat(k, arcs)))

    assert count(3, [(0, 1), (0, 2), (1, 2)]) == 2 * leaves             # feed-forward: either hub first
    assert count(3, [(0, 1), (1, 0), (0, 2), (1, 2)]) == leaves         # the hubs as a mutual pair
    assert count(3, [(0, 1), (0, 2)]) == 2 * (leaves * (leaves - 1) // 2 + leaves)
    assert count(4, [(0, 2), (0, 3), (1, 2), (1, 3)]) == leaves * (leaves - 1) // 2


@pytest.mark.parametrize("n,m", [(40, 31), (40, 33), (90, 2000), (500, 9000)])
@pytest.mark.parametrize("k,arcs", [(3, [(0, 1), (1, 0), (1, 2)]), (3, [(0, 1), (1, 2), (2, 0)]),
                                    (4, [(0, 1), (0, 2), (0, 3), (1, 2), (2, 1)]), (4, [(1, 0), (2, 0), (3, 0)]),
                                    (5, [(0, 1), (1, 2), (2, 3), (3, 4), (4, 0), (0, 2)])])
def test_against_oracle(oracle_lib, n, m, k, arcs):
    N = native()
    rs = np.random.RandomState(n + m)
    src = np.minimum((rs.rand(m) ** 2 * n).astype(np.int32), n - 1)
    dst = rs.randint(0, n, m).astype(np.int32)
    a = pat(k, arcs)
    expect = oracle_lib.count_directed(a, oracle_lib.build_dcsr(n, src, dst))
    g = N.gp_dgraph_create(src, dst, n)
    p = N.gp_dpattern_create(a)
    assert N.gp_dcount(g, p) == expect
    assert N.gp_dcount(g, p, order=list(range(k)), restrictions=[]) == expect
