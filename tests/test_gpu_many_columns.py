"""The many-mesh solve called with several column counts on one handle: the
loop of a block width is captured once, and serves every count that the width
holds, so the columns that it tests must be those of the call."""
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


@pytest.mark.parametrize("counts", [(3, 4), (5, 8, 6), (9, 16), (8, 5)])
def test_every_column_of_every_call_is_solved(gmg, counts):
    systems = gi.spheres_batch(count=3, lo=600, hi=2500, nrhs=max(counts), seed=8, stop=200)
    many = gmg.SolverMany([(s.A, s.Ps) for s in systems])
    first, _, _, _ = many.solve([_t(s.b[:, : counts[0]]) for s in systems], tol=1e-10)
    for k in counts[1:]:
        # the columns of the first call start 1e-9 from their solution, the others from zero
        X0 = [np.zeros((s.n, k)) for s in systems]
        for x0, x in zip(X0, first):
            m = min(k, counts[0])
            x0[:, :m] = x.cpu().numpy()[:, :m] * (1.0 + 1e-9)
        Xs, its, rels, st = many.solve([_t(s.b[:, :k]) for s in systems], [_t(x) for x in X0], tol=1e-10)
        assert st == gmg.GMG_OK and max(rels) <= 1e-10
        for s, X in zip(systems, Xs):
            X = X.cpu().numpy()
            for c in range(k):
                r = np.linalg.norm(s.b[:, c] - s.A @ X[:, c]) / np.linalg.norm(s.b[:, c])
                assert r <= 1.1e-10, f"column {c} of {k}: {r:.1e}"  # the device's residual, summed in another order
    many.close()
