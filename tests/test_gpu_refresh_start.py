"""Where one cluster launch is the whole cycle, a CG solve after a refresh joins
the pending coarsest inverse first and runs in the graph of every other solve
(there is no down-leg to overlap); elsewhere its start overlaps the inverse on
the stream and has a graph of its own.  The solutions are those of a handle made
with the new values."""
import numpy as np
import pytest

import gmg_inputs as gi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gmg(cuda):
    import paper_2307_04886_gb300 as g

    g.load_library()
    return g


@pytest.mark.parametrize("make,graphs", [(lambda: gi.icosphere_system(4), 1),
                                         (lambda: gi.torus_system(420, 240, 1e-4, 3), 2)],
                         ids=["one_launch", "down_leg"])
@pytest.mark.parametrize("precision", [2, 3])
def test_graphs_of_a_solve_after_a_refresh(gmg, make, graphs, precision, monkeypatch, capfd):
    import torch

    s = make()
    b = torch.tensor(s.b, device="cuda")
    g = gmg.Solver(s.A, s.Ps, precision=precision)
    assert (g.paths[0] in (1, 2)) == (graphs == 1)
    monkeypatch.setenv("GMG_VERBOSE", "1")  # a line for every graph that is built
    capfd.readouterr()
    g.solve(b, tol=1e-10)
    for f in (1.5, 0.75):
        g.set_values(f * s.A.data)
        x, it, _, _, _ = g.solve(b, tol=1e-10)
        h = gmg.Solver((f * s.A).tocsr(), s.Ps, precision=precision, use_graphs=False)
        y, it2, _, _, _ = h.solve(b, tol=1e-10)
        assert it == it2 and np.array_equal(x.cpu().numpy(), y.cpu().numpy())
        h.close()
    assert capfd.readouterr().err.count("device-side loop for mode") == graphs
    g.close()
