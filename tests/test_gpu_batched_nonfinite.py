"""NaN and infinite entries in one column of a batched or many-mesh call are
reported as in gmg_solve (GMG_ERR_NONFINITE), whatever the other columns hold,
and leave X as it was."""
import numpy as np
import pytest

import gmg_inputs as gi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gmg(cuda):
    import paper_2307_04886_gb300 as g

    g.load_library()
    return g


def _t(x):
    import torch

    return torch.tensor(np.ascontiguousarray(x, dtype=np.float64), device="cuda")


@pytest.mark.parametrize("where", ["b", "x"])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("nrhs,column,others", [(1, 0, "plain"), (3, 1, "plain"), (8, 7, "plain"), (5, 2, "zero"),
                                                (4, 0, "solved")])
def test_a_non_finite_column_is_reported(gmg, nrhs, column, others, value, where):
    systems = gi.spheres_batch(count=2, lo=600, hi=1500, nrhs=nrhs, seed=8, stop=200)
    s = systems[1]
    one, many = gmg.Solver(s.A, s.Ps), gmg.SolverMany([(q.A, q.Ps) for q in systems])
    B = [q.b.copy() for q in systems]
    X = [np.random.default_rng(3).standard_normal(q.b.shape) for q in systems]
    if others == "zero":  # the columns beside it need no solve
        for q in range(nrhs):
            if q != column:
                for a in B + X:
                    a[:, q] = 0.0
    elif others == "solved":
        X = [x.cpu().numpy() for x in many.solve([_t(b) for b in B], tol=1e-12)[0]]
    (B if where == "b" else X)[1][17, column] = value

    xb, it, _, _, st = one.solve_batched(_t(B[1]), _t(X[1]), tol=1e-10, raise_on_fail=False)
    assert st == gmg.GMG_ERR_NONFINITE and it == 0
    assert np.array_equal(xb.cpu().numpy(), X[1], equal_nan=True)
    Xs, its, rels, st = many.solve([_t(b) for b in B], [_t(x) for x in X], tol=1e-10, raise_on_fail=False)
    assert st == gmg.GMG_ERR_NONFINITE and not np.isfinite(rels[1])
    for a, b in zip(Xs, X):
        assert np.array_equal(a.cpu().numpy(), b, equal_nan=True)
    one.close()
    many.close()
