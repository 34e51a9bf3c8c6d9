"""The V-cycle with its coarse levels on one thread-block cluster, against the
oracle, at the sizes and options where its tables can go wrong: fewer rows
than CTAs on a level, colours missing from a CTA's range, levels whose entries
stream from L2, every sweep count and order, a first colour that the caller
has or has not smoothed, and both precisions.

Tolerances are those of the cycle tests: max(1e-12, 10 kappa 2^-53) in FP64
(summation order; the coarsest solves differ in rounding, which the coarsest
operator amplifies by its condition number kappa), max(1e-6, 10 kappa 2^-24)
in FP32, element-wise times the stencil factor."""
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


def _t(x):
    import torch

    return torch.tensor(np.asarray(x, dtype=np.float64), device="cuda")


SYSTEMS = {
    "tiny": lambda: gi.icosphere_system(2, stop=20),            # 162 rows -> 28 -> 10
    "few_rows_per_cta": lambda: gi.icosphere_system(3, stop=8),  # 642 -> ... -> fewer rows than CTAs
    "ragged": lambda: gi.torus_system(61, 37, 1e-4, 3, stop=12),
    "wide": lambda: gi.torus_system(250, 122, 1e-4, 5),          # one thread per row on the finest level
    "streamed": lambda: gi.workloads.bilaplacian_system(256, 120),  # entries streamed from the finest level
    "book": lambda: gi.nonmanifold_system(3, 60, 80, stop=200),
}


@pytest.fixture(scope="module", params=sorted(SYSTEMS))
def system(request):
    return SYSTEMS[request.param]()


@pytest.mark.parametrize("nu", [(2, 2, False), (1, 0, False), (0, 1, True), (3, 1, True)])
def test_cycle_matches_oracle(gmg, system, nu):
    s = system
    pre, post, fwd = nu
    o = oracle.Oracle(s.A, s.Ps, nu_pre=pre, nu_post=post, post_forward=fwd)
    g = gmg.Solver(s.A, s.Ps, precision=gmg.GMG_FP64, nu_pre=pre, nu_post=post, post_forward=fwd)
    assert g.paths[0] in (1, 2), g.paths  # the whole FP32 cycle is one launch
    ev = np.linalg.eigvalsh(o.level(o.nlev - 1)[0].toarray())
    kappa = ev[-1] / ev[0]
    x0 = np.random.default_rng(17).standard_normal(s.n)

    def check(o, what):
        xo = o.vcycle(x0, s.b)
        close(g.vcycle(_t(x0), _t(s.b), fp32=False).cpu().numpy(), xo, max(1e-12, 10 * kappa * 2.0**-53),
              "FP64 cycle" + what)
        close(g.vcycle(_t(x0), _t(s.b), fp32=True).cpu().numpy(), xo, max(1e-6, 10 * kappa * 2.0**-24),
              "FP32 cycle" + what, stencil_factor(s.A))

    check(o, "")
    # after a numeric refresh the tables hold the new values
    g.set_values(1.5 * s.A.data)
    check(oracle.Oracle((1.5 * s.A).tocsr(), s.Ps, nu_pre=pre, nu_post=post, post_forward=fwd), " after a refresh")
    g.close()


@pytest.mark.parametrize("precision", [0, 1, 2, 3])
def test_solves_match_the_launch_per_phase_form(gmg, system, precision, monkeypatch):
    """A solve with the cluster and with GMG_NO_TAIL=1 (one launch per phase)
    reach the tolerance in the same number of iterations (one more or less:
    rounding may move a residual across it) and agree."""
    s = system
    g = gmg.Solver(s.A, s.Ps, precision=precision)
    monkeypatch.setenv("GMG_NO_TAIL", "1")
    h = gmg.Solver(s.A, s.Ps, precision=precision)
    monkeypatch.delenv("GMG_NO_TAIL")
    assert all(p in (0, 3) for p in h.paths)
    xg, ig, rg, _, _ = g.solve(_t(s.b), tol=1e-10)
    xh, ih, rh, _, _ = h.solve(_t(s.b), tol=1e-10)
    assert abs(ig - ih) <= 1 and max(rg, rh) <= 1e-10
    close(xg.cpu().numpy(), xh.cpu().numpy(), 1e-8, "solution")
    g.close()
    h.close()
