"""Corrections that depend on the basis up to the rounding of FP32 vectors: the second Gram-Schmidt
pass takes most of what the first has left, and the column is still one to keep.  Discarding it
ended the FP32 inner solves of iterative refinement with a breakdown."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2512_08728_gb300 as pkg
from workloads import make_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["ir32", "ir32_bf16"])
@pytest.mark.parametrize("d,p,n,lv", [(3, 2, (32, 32, 32), 4), (2, 3, (32, 32), 3)])
def test_refinement_does_not_break_down(precision, d, p, n, lv):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()
    pr = make_problem(d, p, n, lv, nu_kind="jump", seed=0)
    s = pkg.KCycleSolver(pr, precision=precision, async_smooth=12, lmax=400, coarse_persistent=False)
    x, info = s.solve(pr.b, rtol=1e-10, maxiter=100)      # raises on a breakdown
    s.close()
    assert info["status"] in (0, 1) and info["rel_res"] < 0.1 and np.isfinite(x).all()
