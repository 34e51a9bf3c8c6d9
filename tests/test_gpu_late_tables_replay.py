"""FP32 cycles that a caller captured on a handle whose solves run FP64 cycles,
replayed after refreshes: they have the refreshed values, as a cycle called
afresh and one of a handle with FP32 cycles have."""
import numpy as np
import pytest

import gmg_inputs as gi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gmg(cuda):
    import paper_2307_04886_gb300 as g

    g.load_library()
    return g


@pytest.mark.parametrize("precision", [0, 3])
@pytest.mark.parametrize("stale", [False, True])
def test_a_captured_cycle_follows_refreshes(gmg, precision, stale):
    import torch

    s = gi.icosphere_system(4)
    b = torch.tensor(s.b, device="cuda")
    x0 = torch.tensor(np.random.default_rng(5).standard_normal(s.n), device="cuda")
    g, h = gmg.Solver(s.A, s.Ps, precision=precision), gmg.Solver(s.A, s.Ps, precision=2)
    g.vcycle(x0.clone(), b, fp32=True)  # the tables are there and filled
    if stale:  # captured with a fill of its own
        g.set_values(2.0 * s.A.data)
        g.vcycle(x0.clone(), b, fp32=False)
    x, graph = x0.clone(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        g.vcycle(x, b, fp32=True)
    for f in (1.5, 0.75):
        for q in (g, h):
            q.set_values(f * s.A.data)
            q.vcycle(x0.clone(), b, fp32=False)  # joins the coarsest inverse
        x.copy_(x0)
        graph.replay()
        want = h.vcycle(x0.clone(), b, fp32=True)
        assert torch.equal(x, want), f
        assert torch.equal(g.vcycle(x0.clone(), b, fp32=True), want), f
    g.close()
    h.close()
