"""Coarse levels that block 0 runs alone for longer than the other blocks' wait limit (a few seconds):
their iteration cap is large and their tolerance out of reach."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2512_08728_gb300 as pkg
from workloads import make_problem

pytestmark = pytest.mark.gpu


def test_the_others_wait():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()
    pr = make_problem(2, 1, (16, 16), 3, nu_kind="jump", seed=1)
    iters = 200_000                                  # of some 50 us
    s = pkg.KCycleSolver(pr, lmax=30, lvl_rtol=[0.0] * 3, lvl_maxit=[1, iters, 1])
    x, info = s.solve(pr.b, rtol=1e-10, maxiter=1)
    s.close()
    assert info["status"] == 1 and info["level_iters"][1] == iters and info["kernel_launches"] < 10
    assert np.isfinite(x).all() and info["rel_res"] < 1.0
