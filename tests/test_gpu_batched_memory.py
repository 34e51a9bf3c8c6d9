"""Batched calls that find too little device memory for their blocks: an error
status, and the next call, with the memory there, solves as on a fresh handle."""
import numpy as np
import pytest

import gmg_inputs as gi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gmg(cuda):
    import paper_2307_04886_gb300 as g

    g.load_library()
    return g


@pytest.mark.parametrize("left_mb", [12, 60, 76])
def test_a_batched_solve_after_one_without_memory(gmg, left_mb):
    import torch

    s = gi.torus_system(512, 256, 1e-4, 5)  # blocks: 34 MB of FP32, 50 of FP64
    g, h = gmg.Solver(s.A, s.Ps), gmg.Solver(s.A, s.Ps)
    B = torch.tensor(np.random.default_rng(1).standard_normal((s.n, 8)), device="cuda")
    X = torch.zeros_like(B)
    want, it, _, _, _ = h.solve_batched(B, X.clone(), tol=1e-9)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hog, size = [], 1 << 35
    while size >= 1 << 21:
        if torch.cuda.mem_get_info()[0] - size < left_mb << 20:
            size //= 2
            continue
        try:
            hog.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
        except torch.OutOfMemoryError:
            size //= 2
    st = g.solve_batched(B, X, tol=1e-9, raise_on_fail=False)[4]
    hog.clear()
    torch.cuda.empty_cache()
    assert st == 7  # GMG_ERR_OOM
    assert not X.any()
    got, it2, _, _, _ = g.solve_batched(B, X, tol=1e-9)
    assert it2 == it and torch.equal(got, want)
    g.close()
    h.close()
