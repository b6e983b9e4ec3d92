"""Inclusion-exclusion counts of a clique joined to independent vertices: the
root bit matrices against closed forms and against the general kernel, at the
sizes where the form changes (one 32-bit word of columns, 31/32 rows, 512/513
columns, compacted matrices beyond a warp's area, task ranges)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA device")]

from math import comb, perm  # noqa: E402

from paper_2009_10955_gb300 import native  # noqa: E402
from synth import named_pattern  # noqa: E402
from synth.graphs import chung_lu_edges, rmat_edges  # noqa: E402


def clique_join(m, t):
    """K_m joined to t independent vertices."""
    adj = np.ones((m + t, m + t), np.uint8) - np.eye(m + t, dtype=np.uint8)
    adj[m:, m:] = 0
    return adj


# pattern -> adjacency; the copies of it in K_n are perm(n, k) / (m! t!)
PATTERNS = {"diamond": (2, 2), "k5e": (3, 2), "k6e": (4, 2), "book3": (2, 3), "k3_3": (3, 3), "book4": (2, 4),
            "k4_3": (4, 3)}


def plan(N, graph, name):
    """The clique first, then the independent vertices, restricted to one order."""
    m, t = PATTERNS[name]
    order = list(range(m + t))
    res = [(a, b) for a in range(m) for b in range(a + 1, m)] + \
          [(a, b) for a in range(m, m + t) for b in range(a + 1, m + t)]
    s = N.gp_schedule_explicit(N.gp_pattern_create(clique_join(m, t)), order, res)
    s.set_iep(True)
    assert s.iep(0)[0] == t
    return s


def core_and_leaves(core, leaves):
    """A clique of `core` vertices, all joined to `leaves` further ones."""
    a, b = np.triu_indices(core, 1)
    x, y = np.meshgrid(np.arange(core), core + np.arange(leaves), indexing="ij")
    return np.concatenate([a, x.ravel()]).astype(np.int32), np.concatenate([b, y.ravel()]).astype(np.int32)


@pytest.mark.parametrize("n", [2, 4, 6, 31, 32, 33, 34, 64, 65, 129, 200])
@pytest.mark.parametrize("name", sorted(PATTERNS))
def test_complete_graph(n, name):
    N = native()
    a, b = np.triu_indices(n, 1)
    g = N.gp_graph_create_edges(a.astype(np.int32), b.astype(np.int32), n, N.GP_DEGREE_ORDER)
    m, t = PATTERNS[name]
    expect = comb(n, m) * comb(max(n - m, 0), t)
    assert perm(n, m + t) == expect * perm(m, m) * perm(t, t)
    assert N.gp_count(g, plan(N, g, name), 0)[1] == expect


@pytest.mark.parametrize("name", ["diamond", "k5e", "k6e", "k4_3"])
@pytest.mark.parametrize("n,edges", [
    (40 + 472, lambda: core_and_leaves(40, 472)),         # 511 neighbours of a core vertex
    (40 + 474, lambda: core_and_leaves(40, 474)),         # 513: hubs
    (30 + 3000, lambda: core_and_leaves(30, 3000)),
    (120 + 700, lambda: core_and_leaves(120, 700)),       # compacted matrices beyond a warp's area
    (1 << 11, lambda: rmat_edges(11, 12, 0.57, 0.19, 0.19, seed=9)),
    (12_001, lambda: chung_lu_edges(12_001, 100_003, 2.1, 900.0, 17.5, seed=6)),
])
def test_against_general_kernel(name, n, edges):
    N = native()
    src, dst = edges()
    g = N.gp_graph_create_edges(src, dst, n, N.GP_DEGREE_ORDER)
    s = plan(N, g, name)
    nnz = g.device_csr()[2]
    for a, b in ((0, 0), (0, nnz // 3), (nnz // 3, nnz // 3 + 7), (nnz // 2, nnz)):
        got = N.gp_count_raw(g, s, 0, task_begin=a, task_end=b)
        assert got == N.gp_count_raw(g, s, 0, task_begin=a, task_end=b, flags=N.GP_COUNT_NO_CORE)


def hub_and_ring(ring, common):
    """Four mutually adjacent hubs and `common` vertices adjacent to all of
    them; the last hub is also joined to a ring of vertices of degree five, so
    that the common vertices are its last neighbours, behind 3 + ring others;
    leaves keep the other hubs ahead of it in the degree order."""
    src, dst = [0, 0, 0, 1, 1, 2], [1, 2, 3, 2, 3, 3]
    for c in range(4, 4 + common):
        src += [0, 1, 2, 3]
        dst += [c] * 4
    at = 4 + common
    parts = [(np.array(src), np.array(dst))]
    r = np.arange(ring)
    parts += [(np.full(ring, 3), at + r), (at + r, at + (r + 1) % ring), (at + r, at + (r + 2) % ring)]
    at += ring
    for hub, leaves in ((2, ring + 1000), (1, ring + 2000), (0, ring + 3000)):
        parts.append((np.full(leaves, hub), at + np.arange(leaves)))
        at += leaves
    return at, np.concatenate([a for a, _ in parts]).astype(np.int32), \
        np.concatenate([b for _, b in parts]).astype(np.int32)


# the common vertices' positions among the last hub's neighbours end at
# 65535, straddle 65536 and lie beyond it; with 700 of them the row of the
# other hubs has more members than a warp compacts
@pytest.mark.parametrize("ring,common", [(65_531, 2), (65_532, 2), (65_533, 3), (70_000, 4), (70_000, 700)])
def test_positions_beyond_16_bits(ring, common):
    N = native()
    n, src, dst = hub_and_ring(ring, common)
    g = N.gp_graph_create_edges(src, dst, n, N.GP_DEGREE_ORDER)
    for name in ("k6e", "k4_3"):
        assert N.gp_count(g, plan(N, g, name), 0)[1] == comb(common, PATTERNS[name][1])
