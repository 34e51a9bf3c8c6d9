"""FP32 cycles on handles whose solves run FP64 cycles: their cluster tables are
built by the first FP32 cycle (or the first question for the level paths) and
filled again for the first one after a refresh.  They give the bits of a handle
that has them from the start, refreshes do no work for them, and inside a stream
capture the cycle runs with what there is."""
import numpy as np
import pytest

import gmg_inputs as gi
import oracle
from parity_util import assert_close as close
from parity_util import stencil_factor

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gmg(cuda):
    import paper_2307_04886_gb300 as g

    g.load_library()
    return g


SYSTEMS = {
    "one_launch": lambda: gi.icosphere_system(4),
    "streamed": lambda: gi.torus_system(250, 122, 1e-4, 5),
    "below_a_colour_launch": lambda: gi.torus_system(420, 240, 1e-4, 3),
}


@pytest.fixture(scope="module", params=sorted(SYSTEMS))
def system(request):
    return SYSTEMS[request.param]()


@pytest.mark.parametrize("ask_first", [False, True])
@pytest.mark.parametrize("precision", [0, 3])
def test_fp32_cycles_of_fp64_handles(gmg, system, precision, ask_first):
    import torch

    s = system
    b = torch.tensor(s.b, device="cuda")
    x0 = torch.tensor(np.random.default_rng(5).standard_normal(s.n), device="cuda")
    g, h = gmg.Solver(s.A, s.Ps, precision=precision), gmg.Solver(s.A, s.Ps, precision=2)
    if ask_first:
        assert g.paths == h.paths
    counts = []
    for f in (1.0, 1.5, 0.75, 0.5):
        if f != 1.0:
            for q in (g, h):
                before = gmg.kernel_launches()
                q.set_values(f * s.A.data)
                counts.append(gmg.kernel_launches() - before)
        if f != 0.75:  # two refreshes between cycles, too
            for _ in range(2):
                assert torch.equal(g.vcycle(x0.clone(), b, fp32=True), h.vcycle(x0.clone(), b, fp32=True))
        assert torch.isfinite(g.vcycle(x0.clone(), b, fp32=False)).all()
    assert g.paths == h.paths
    assert len(set(counts)) == 1, counts  # the tables of one precision are filled, on either handle
    g.close()
    h.close()


@pytest.mark.parametrize("built", [False, True])
def test_cycles_in_a_capture(gmg, built):
    import torch

    s = gi.icosphere_system(4)
    o = oracle.Oracle(s.A, s.Ps)
    g = gmg.Solver(s.A, s.Ps, precision=0)
    b = torch.tensor(s.b, device="cuda")
    x0 = torch.tensor(np.random.default_rng(5).standard_normal(s.n), device="cuda")
    if built:
        g.vcycle(x0.clone(), b, fp32=True)
    g.set_values(1.5 * s.A.data)  # the FP32 tables are not there, or not filled
    g.vcycle(x0.clone(), b, fp32=False)  # joins the inverse outside the capture
    x, graph = x0.clone(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        g.vcycle(x, b, fp32=True)
    xo = oracle.Oracle((1.5 * s.A).tocsr(), s.Ps).vcycle(x0.cpu().numpy(), s.b)
    x.copy_(x0)
    graph.replay()
    close(x.cpu().numpy(), xo, 1e-6, "captured cycle", stencil_factor(s.A))
    close(g.vcycle(x0.clone(), b, fp32=True).cpu().numpy(), xo, 1e-6, "cycle after the capture", stencil_factor(s.A))
    assert o.nlev == g.nlev and g.paths[0] in (1, 2)
    g.close()
