"""The sampling sweep of the GPU hierarchy builder where its point lists and
rounds take other paths than on the meshes: lists longer than a point's own
row (a second search into CSR rows), frontiers longer than one block takes
(a point cloud in random order) and the longest chains of short rounds (points
on a line).  Every level is the host builder's, bit for bit."""
import numpy as np
import pytest

from gmg_inputs import meshes, operators
from gmg_inputs.hierarchy import build_level

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gmg(cuda):
    import paper_2307_04886_gb300 as g

    g.load_library()
    return g


def _cloud(n, k):
    V = meshes.noisy_sphere_cloud(n, np.random.default_rng(2))
    return (V, *operators.edges_to_adjacency(n, operators.knn_graph(V, k)[0]))


def _line(n):
    rng = np.random.default_rng(0)
    V = np.stack([np.cumsum(rng.uniform(0.1, 1.0, n)), rng.uniform(0.0, 0.3, n), np.zeros(n)], axis=1)
    return (V, *operators.edges_to_adjacency(n, np.stack([np.arange(n - 1), np.arange(1, n)], axis=1)))


@pytest.mark.parametrize("graph,phi", [(lambda: _cloud(20000, 8), 1.0 / 64.0), (lambda: _cloud(90000, 5), 1.0 / 8.0),
                                       (lambda: _cloud(4097, 3), 1.0 / 2.0), (lambda: _line(5000), 1.0 / 8.0),
                                       (lambda: _line(2), 1.0 / 8.0)],
                         ids=["long_lists", "long_frontiers", "one_past_a_tile", "line", "two_points"])
def test_levels_are_the_host_builders(gmg, graph, phi):
    V, rp, ci = graph()
    levels, _ = gmg.build_hierarchy(V, rp, ci, phi=phi, stop=50 if V.shape[0] > 50 else 1, max_levels=3)
    X, r, c = V, rp, ci
    for G in levels:
        P, Xc, crp, cci = build_level(X, r, c, phi)
        assert G.n_coarse == P.n_coarse and np.array_equal(G.samples, P.samples) and np.array_equal(G.cell, P.seed)
        assert np.array_equal(G.Xc, Xc) and np.array_equal(G.graph_rowptr, crp) and np.array_equal(G.graph_col, cci)
        assert np.array_equal(G.idx, P.idx) and np.array_equal(G.w, P.w) and G.stats == P.stats
        X, r, c = Xc, crp, cci
    assert levels
