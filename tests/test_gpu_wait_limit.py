"""Solves whose cluster launches' waits give up (a limit of no polls: the path
of a copy that does not come, without losing one): GMG_ERR_TIMEOUT, nothing
read or written that should not be, and the bits of an undisturbed handle once
the limit is back."""
import numpy as np
import pytest

import gmg_inputs as gi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gmg(cuda):
    import paper_2307_04886_gb300 as g

    g.load_library()
    return g


SYSTEMS = {
    "one_launch": lambda: gi.icosphere_system(4),
    "streamed": lambda: gi.workloads.bilaplacian_system(256, 120),
    "below_a_colour_launch": lambda: gi.torus_system(420, 240, 1e-4, 3),
}


@pytest.mark.parametrize("name", sorted(SYSTEMS))
@pytest.mark.parametrize("host_loop", [False, True])
@pytest.mark.parametrize("precision", [0, 1, 2, 3])
def test_a_wait_that_gives_up_is_reported(gmg, name, precision, host_loop):
    import torch

    s = SYSTEMS[name]()
    b = torch.tensor(s.b, device="cuda")
    g = gmg.Solver(s.A, s.Ps, precision=precision, max_iter=60)
    assert any(p in (1, 2) for p in g.paths) and (g.paths[0] == 0) == (name == "below_a_colour_launch")
    g.profile(host_loop)
    x, it, rr, _, st = g.solve(b, tol=1e-9)
    lib = gmg.load_library()
    for _ in range(2):
        assert lib.gmg_wait_limit(g.handle, 0) == gmg.GMG_OK
        assert g.solve(b, tol=1e-9, raise_on_fail=False)[4] == gmg.GMG_ERR_TIMEOUT
        assert lib.gmg_wait_limit(g.handle, -1) == gmg.GMG_OK
        y, it2, rr2, _, st2 = g.solve(b, tol=1e-9)
        assert st2 == gmg.GMG_OK and it2 == it and rr2 == rr
        assert np.array_equal(y.cpu().numpy(), x.cpu().numpy())
    g.close()


@pytest.mark.parametrize("name", sorted(SYSTEMS))
@pytest.mark.parametrize("fp32", [False, True])
@pytest.mark.parametrize("precision", [0, 2])
def test_a_cycle_whose_wait_gives_up_leaves_nan(gmg, name, precision, fp32):
    """A single cycle does not synchronise: its x is NaN, and neither the next
    cycle nor the next solve takes the blame."""
    import torch

    s = SYSTEMS[name]()
    b = torch.tensor(s.b, device="cuda")
    x0 = torch.tensor(np.random.default_rng(5).standard_normal(s.n), device="cuda")
    g = gmg.Solver(s.A, s.Ps, precision=precision, max_iter=60)
    lib = gmg.load_library()
    ref = g.vcycle(x0.clone(), b, fp32=fp32).cpu().numpy()
    sol, it, _, _, _ = g.solve(b, tol=1e-9)
    assert np.all(np.isfinite(ref))
    clustered = fp32 or precision == 0  # FP32 handles run FP64 cycles as colour launches
    for follow in ("cycle", "solve"):
        lib.gmg_wait_limit(g.handle, 0)
        bad = g.vcycle(x0.clone(), b, fp32=fp32).cpu().numpy()
        assert np.all(np.isnan(bad)) if clustered else np.array_equal(bad, ref)
        lib.gmg_wait_limit(g.handle, -1)
        if follow == "cycle":
            assert np.array_equal(g.vcycle(x0.clone(), b, fp32=fp32).cpu().numpy(), ref)
        else:
            y, it2, _, _, st = g.solve(b, tol=1e-9, raise_on_fail=False)
            assert st == gmg.GMG_OK and it2 == it and np.array_equal(y.cpu().numpy(), sol.cpu().numpy())
    g.close()
