"""A cycle without a cluster launch after one of the same handle whose wait gave
up: the error word that the failed cycle left behind is not its own."""
import numpy as np
import pytest

import gmg_inputs as gi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gmg(cuda):
    import paper_2307_04886_gb300 as g

    g.load_library()
    return g


@pytest.mark.parametrize("precision", [1, 2])
def test_fp64_cycle_after_a_failed_fp32_cycle(gmg, precision):
    import torch

    s = gi.icosphere_system(4)
    b = torch.tensor(s.b, device="cuda")
    x0 = torch.tensor(np.random.default_rng(5).standard_normal(s.n), device="cuda")
    g = gmg.Solver(s.A, s.Ps, precision=precision)  # FP64 cycles: colour launches
    lib = gmg.load_library()
    ref = g.vcycle(x0.clone(), b, fp32=False).cpu().numpy()
    assert np.all(np.isfinite(ref))
    assert lib.gmg_wait_limit(g.handle, 0) == gmg.GMG_OK
    assert torch.isnan(g.vcycle(x0.clone(), b, fp32=True)).all()
    assert lib.gmg_wait_limit(g.handle, -1) == gmg.GMG_OK
    assert np.array_equal(g.vcycle(x0.clone(), b, fp32=False).cpu().numpy(), ref)
    g.close()
