"""Starts, restarts and ends of the device-driven solve (one graph holding the
start, the loop and the final residual) against the host-driven loop, which
profiling selects: the same kernels in the same order, so iterates, counts,
histories, statuses and what is left in x agree bit for bit."""
import numpy as np
import pytest

import gmg_inputs as gi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gmg(cuda):
    import paper_2307_04886_gb300 as g

    g.load_library()
    return g


def _both(gmg, s, precision, b, x0, tol, max_iter, history, device, refresh=False):
    import torch

    out = []
    for host_loop in (False, True):
        g = gmg.Solver(s.A, s.Ps, precision=precision, max_iter=max_iter)
        g.profile(host_loop)
        if refresh:
            g.set_values(1.5 * s.A.data)
        bb, xx = (torch.tensor(v, device="cuda") if device else v.copy() for v in (b, x0))
        x, it, rr, hist, st = g.solve(bb, x=xx, tol=tol, history=history, raise_on_fail=False)
        out.append((np.asarray(x.cpu() if device else x), it, np.float64(rr), np.array(hist), st))
        g.close()
    return out


@pytest.mark.parametrize("device", [False, True])
@pytest.mark.parametrize("precision", [0, 1, 2, 3])
@pytest.mark.parametrize("case", ["plain", "zero_b", "nan_b", "inf_b", "nan_x", "one_step", "tight", "long", "refresh"])
def test_device_driven_matches_host_driven(gmg, case, precision, device):
    s = gi.icosphere_system(4)
    rng = np.random.default_rng(31)
    b, x0 = s.b.copy(), rng.standard_normal(s.n)
    tol, max_iter, history, refresh = 1e-10, 100, 101, False
    if case == "zero_b":
        b[:] = 0.0
    elif case in ("nan_b", "inf_b"):
        b[7] = np.nan if case == "nan_b" else np.inf
    elif case == "nan_x":
        x0[11] = np.nan
    elif case == "one_step":
        max_iter, tol, history = 1, 0.0, 2
    elif case == "tight":  # the recursive residual passes, the true one does not: CG restarts
        tol, max_iter, history = 1e-17, 40, 41
    elif case == "long":  # more history than the report of one solve holds
        tol, max_iter, history = 0.0, 90, 91
    elif case == "refresh":  # CG's start joins a pending coarsest inverse
        refresh = True
    d, h = _both(gmg, s, precision, b, x0, tol, max_iter, history, device, refresh)
    assert d[4] == h[4] and d[1] == h[1]
    assert np.array_equal(d[0], h[0], equal_nan=True)
    assert np.array_equal(d[2], h[2], equal_nan=True)
    m = d[1] if d[4] == gmg.GMG_ERR_NONFINITE else None  # the non-finite step itself need not be in the history
    assert np.array_equal(d[3][:m], h[3][:m], equal_nan=True)
