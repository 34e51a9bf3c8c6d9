"""The coarsest solve of FP32 cycles on hierarchies with one smoothed level, or
with a last smoothed level of many rows: the FP64 inverse with FP64 sums, in the
cluster launch as in the launch-per-phase form (GMG_NO_TAIL=1).  On a nearly singular system (condition number of
the coarsest operator far above 2^24) an FP32 inverse carries no accuracy in
the modes beside the near-constant one, and iterations that converge stall."""
import numpy as np
import pytest

import gmg_inputs as gi
from gmg_inputs import operators

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gmg(cuda):
    import paper_2307_04886_gb300 as g

    g.load_library()
    return g


def _t(x):
    import torch

    return torch.tensor(np.asarray(x, dtype=np.float64), device="cuda")


def _solvers(gmg, A, Ps, monkeypatch, **kw):
    g = gmg.Solver(A, Ps, **kw)
    monkeypatch.setenv("GMG_NO_TAIL", "1")
    h = gmg.Solver(A, Ps, **kw)
    monkeypatch.delenv("GMG_NO_TAIL")
    assert g.paths[-2] in (1, 2) and all(p in (0, 3) for p in h.paths)
    return g, h


SYSTEMS = {
    "two_levels_402": (lambda: gi.icosphere_system(4, stop=450), 1),
    "two_levels_102": (lambda: gi.icosphere_system(3, stop=200), 1),
    "two_levels_more_columns_than_registers": (lambda: gi.torus_system(80, 50, 1e-4, 3, stop=1000), 1),
    "many_rows_on_the_last_smoothed_level": (lambda: gi.torus_system(320, 150, 1e-4, 3, stop=1500), 2),
}


@pytest.mark.parametrize("name,eta", [("two_levels_402", 1e-6), ("two_levels_402", 1e-8), ("two_levels_102", 1e-7),
                                      ("two_levels_more_columns_than_registers", 1e-8),
                                      ("many_rows_on_the_last_smoothed_level", 1e-8)])
@pytest.mark.parametrize("precision", [1, 2])
def test_converges_as_with_a_launch_per_phase(gmg, name, eta, precision, monkeypatch):
    make, smoothed = SYSTEMS[name]
    s = make()
    assert len(s.Ps) == smoothed
    A = operators.poisson_matrix(s.Mdiag, s.L, eta)
    b = s.b - s.Mdiag * (s.b.sum() / s.Mdiag.sum())  # no constant part: the solution is of order one
    g, h = _solvers(gmg, A, s.Ps, monkeypatch, precision=precision)
    xg, ig, rg, _, sg = g.solve(_t(b), tol=1e-7, raise_on_fail=False)
    xh, ih, rh, _, sh = h.solve(_t(b), tol=1e-7, raise_on_fail=False)
    assert sh == gmg.GMG_OK, (ih, rh)
    assert sg == gmg.GMG_OK and abs(ig - ih) <= 1, (ig, rg, ih, rh)
    g.close()
    h.close()
