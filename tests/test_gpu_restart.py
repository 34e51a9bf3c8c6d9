"""A CG solve whose restart finds no graph for the iterations after it (the
driver refused it: GMG_NO_RESTART_LOOP=1 stands for that): the host loop goes
on from the restart, with the bits of a solve that the host drives throughout,
and later solves still start in the whole-solve graph."""
import numpy as np
import pytest

import gmg_inputs as gi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gmg(cuda):
    import paper_2307_04886_gb300 as g

    g.load_library()
    return g


@pytest.mark.parametrize("precision", [2, 3])
@pytest.mark.parametrize("tol,max_iter,refresh", [(1e-17, 40, False), (2e-16, 40, False), (1e-10, 40, True)])
def test_the_host_loop_goes_on_after_a_restart(gmg, precision, tol, max_iter, refresh, monkeypatch):
    import torch

    s = gi.icosphere_system(4)
    b = torch.tensor(s.b, device="cuda")
    monkeypatch.setenv("GMG_NO_RESTART_LOOP", "1")
    out = []
    for host in (False, True):
        g = gmg.Solver(s.A, s.Ps, precision=precision, max_iter=max_iter)
        g.profile(host)
        if refresh:
            g.set_values(1.5 * s.A.data)
        x, it, rr, hist, st = g.solve(b, tol=tol, history=max_iter + 1, raise_on_fail=False)
        y, it2, _, _, st2 = g.solve(b, tol=1e-10)
        out.append((x.cpu().numpy(), it, rr, hist, st, y.cpu().numpy(), it2, st2))
        g.close()
    d, h = out
    assert d[4] == h[4] and d[1] == h[1] and d[2] == h[2]
    # a solve that does not converge has used every iteration that it may
    assert d[4] == gmg.GMG_OK or d[1] == max_iter
    for k in (0, 3, 5):
        assert np.array_equal(d[k], h[k])
    assert d[6] == h[6] and d[7] == h[7] == gmg.GMG_OK
