"""Plans of the cluster launch that few sizes take: eight CTAs (where sixteen
cannot be scheduled; forced) and two entry stages (where no more fit), against the oracle's cycle and the launch-per-phase form's solves.  Tolerances
are those of the cycle tests."""
import re

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


# system, precision of the handle, CTAs forced (0: the library's choice), stages expected (None: any)
PLANS = {
    "8_ctas_tiny_fp32": (lambda: gi.icosphere_system(2, stop=20), 2, 8, 0),
    "8_ctas_tiny_fp64": (lambda: gi.icosphere_system(2, stop=20), 0, 8, 0),
    "8_ctas_ragged_fp32": (lambda: gi.torus_system(61, 37, 1e-4, 3, stop=12), 2, 8, None),
    "8_ctas_ragged_fp64": (lambda: gi.torus_system(61, 37, 1e-4, 3, stop=12), 3, 8, None),
    "8_ctas_streamed_fp32": (lambda: gi.torus_system(160, 125, 1e-4, 5), 1, 8, None),
    "8_ctas_streamed_fp64": (lambda: gi.torus_system(120, 90, 1e-4, 5), 0, 8, None),
    "5_ctas_fp32": (lambda: gi.torus_system(61, 37, 1e-4, 3, stop=12), 2, 5, None),
    "2_stages_fp32": (lambda: gi.torus_system(300, 170, 1e-4, 5), 2, 0, 2),
    "2_stages_fp64": (lambda: gi.torus_system(210, 120, 1e-4, 5), 0, 0, 2),
}


@pytest.mark.parametrize("name", sorted(PLANS))
def test_cycle_and_solve(gmg, name, monkeypatch, capfd):
    import torch

    make, precision, ctas, stages = PLANS[name]
    s = make()
    fp32 = precision in (1, 2)
    monkeypatch.setenv("GMG_VERBOSE", "1")
    if ctas:
        monkeypatch.setenv("GMG_TAIL_CTAS", str(ctas))
    capfd.readouterr()
    g = gmg.Solver(s.A, s.Ps, precision=precision)
    m = re.search(r"FP(\d+) cluster: from level (\d+), (\d+) CTAs, (\d+) stages", capfd.readouterr().err)
    assert m and int(m[1]) == (32 if fp32 else 64) and int(m[2]) == 0, m
    assert int(m[3]) == (ctas or 16) and (stages is None or int(m[4]) == stages), m
    monkeypatch.delenv("GMG_TAIL_CTAS", raising=False)
    monkeypatch.delenv("GMG_VERBOSE")
    o = oracle.Oracle(s.A, s.Ps)
    x0 = np.random.default_rng(17).standard_normal(s.n)
    xo = o.vcycle(x0, s.b)
    ev = np.linalg.eigvalsh(o.level(o.nlev - 1)[0].toarray())
    kappa = ev[-1] / ev[0]
    b, t0 = torch.tensor(s.b, device="cuda"), torch.tensor(x0, device="cuda")
    for _ in range(2):
        x = g.vcycle(t0.clone(), b, fp32=fp32).cpu().numpy()
        if fp32:
            close(x, xo, max(1e-6, 10 * kappa * 2.0**-24), "FP32 cycle", stencil_factor(s.A))
        else:
            close(x, xo, max(1e-12, 10 * kappa * 2.0**-53), "FP64 cycle")
    monkeypatch.setenv("GMG_NO_TAIL", "1")
    h = gmg.Solver(s.A, s.Ps, precision=precision)
    monkeypatch.delenv("GMG_NO_TAIL")
    xg, ig, rg, _, _ = g.solve(b, tol=1e-10)
    xh, ih, rh, _, _ = h.solve(b, tol=1e-10)
    assert abs(ig - ih) <= 1 and max(rg, rh) <= 1e-10
    close(xg.cpu().numpy(), xh.cpu().numpy(), 1e-8, "solution")
    g.close()
    h.close()
