"""Set-up and the late tables on a stream that the legacy stream does not order:
what they upload is there when their kernels read it."""
import numpy as np
import pytest

import gmg_inputs as gi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gmg(cuda):
    import paper_2307_04886_gb300 as g

    g.load_library()
    return g


@pytest.mark.parametrize("precision", [0, 2])
def test_first_calls_on_a_stream_of_their_own(gmg, precision):
    import torch

    s = gi.torus_system(250, 122, 1e-4, 5)
    b = torch.tensor(s.b, device="cuda")
    x0 = torch.tensor(np.random.default_rng(5).standard_normal(s.n), device="cuda")
    h = gmg.Solver(s.A, s.Ps, precision=precision)
    want = [h.vcycle(x0.clone(), b, fp32=f) for f in (True, False)]
    sol, it, _, _, _ = h.solve(b, tol=1e-9)
    torch.cuda.synchronize()
    for _ in range(5):
        with torch.cuda.stream(torch.cuda.Stream()):  # non-blocking
            g = gmg.Solver(s.A, s.Ps, precision=precision)
            got = [g.vcycle(x0.clone(), b, fp32=f) for f in (True, False)]
            y, it2, _, _, _ = g.solve(b, tol=1e-9)
            torch.cuda.current_stream().synchronize()
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
        assert it2 == it and torch.equal(y, sol)
        g.close()
    h.close()
