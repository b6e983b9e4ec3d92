"""Labelled counts and listings over the surviving tasks: label choices that
leave no task, few tasks (cut into parts) or all of them, sets shared by
depths of one label and kept apart for different ones, lists beyond one
lane's share, listings at the edges of a warp's 32 tasks."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

from math import comb  # noqa: E402

from paper_2009_10955_gb300 import native  # noqa: E402
from synth import named_pattern  # noqa: E402
from synth.graphs import rmat_edges  # noqa: E402


@pytest.mark.parametrize("pattern,plab", [("triangle", [0, 1, 2]), ("triangle", [1, 1, 1]), ("path3", [0, 2, 0]),
                                          ("k4", [0, 1, 0, 1]), ("c4", [0, 1, 0, 2]), ("house", [0, 1, 2, 0, 1]),
                                          ("house", [1, 1, 1, 1, 1]), ("k5", [0, 1, 2, 3, 4]), ("house", [0, 9, 0, 0, 0])])
@pytest.mark.parametrize("nlab", [2, 5])
def test_against_oracle(oracle_lib, pattern, plab, nlab):
    N = native()
    n = 1 << 8
    src, dst = rmat_edges(8, 8, 0.57, 0.19, 0.19, seed=11)
    glab = np.random.RandomState(nlab).randint(0, nlab, n).astype(np.int32)
    adj = named_pattern(pattern)
    expect = oracle_lib.count_labeled(adj, np.array(plab, np.int32), oracle_lib.build_csr(n, src, dst), glab)
    for flags in (N.GP_DEGREE_ORDER, 0):
        g = N.gp_graph_create_edges(src, dst, n, flags)
        N.gp_graph_set_labels(g, glab)
        s = N.gp_schedule(N.gp_pattern_create_labeled(adj, plab), g, 3)
        for i in range(len(s)):
            assert N.gp_count(g, s, i)[1] == expect
        if 0 < expect < 200_000:
            out = torch.zeros(expect + 1, len(plab), dtype=torch.int32, device="cuda")
            _, written, _ = N.gp_list(g, s, 0, 0, 0, out, expect + 1)
            assert written == expect


@pytest.mark.parametrize("leaves", [31, 32, 33, 192, 193, 500])
def test_star_leaves_by_label(leaves):
    """A hub with `leaves` of label 1 and as many of label 2."""
    N = native()
    n = 2 * leaves + 1
    g = N.gp_graph_create_edges(np.zeros(n - 1, np.int32), np.arange(1, n, dtype=np.int32), n, N.GP_DEGREE_ORDER)
    N.gp_graph_set_labels(g, np.array([0] + [1] * leaves + [2] * leaves, np.int32))

    def count(pattern, labels):
        s = N.gp_schedule(N.gp_pattern_create_labeled(named_pattern(pattern), labels), g, 1)
        return N.gp_count(g, s, 0)[1]

    assert count("path3", [1, 0, 2]) == leaves * leaves
    assert count("path3", [1, 0, 1]) == comb(leaves, 2)
    assert count("star4", [0, 1, 1, 2]) == comb(leaves, 2) * leaves


@pytest.mark.parametrize("n", [3, 8, 9, 12, 33])
def test_listing_complete_graph(n):
    N = native()
    a, b = np.triu_indices(n, 1)
    g = N.gp_graph_create_edges(a.astype(np.int32), b.astype(np.int32), n, N.GP_DEGREE_ORDER)
    for pattern, k in (("triangle", 3), ("k4", 4)):
        s = N.gp_schedule(N.gp_pattern_create(named_pattern(pattern)), g, 1)
        total = comb(n, k)
        out = torch.zeros(total + 5, k, dtype=torch.int32, device="cuda")
        status, written, after = N.gp_list(g, s, 0, 0, 0, out, total + 5)
        assert (status, written, after) == (N.GP_OK, total, n * (n - 1))
        got = np.sort(out[:written].cpu().numpy(), axis=1)
        assert len(np.unique(got, axis=0)) == total
