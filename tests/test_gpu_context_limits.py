"""Contexts of one basis and different sizes share the persistent kernel and its attributes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2512_08728_gb300 as pkg
from workloads import make_problem

pytestmark = pytest.mark.gpu


def test_a_smaller_context_leaves_a_larger_one_usable():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()
    big = make_problem(2, 3, (64, 48), 4)       # three levels of coefficients: 60 KB of shared memory a block
    small = make_problem(2, 3, (8, 8), 3)
    a = pkg.KCycleSolver(big)
    x0, info0 = a.solve(big.b, maxiter=2)
    b = pkg.KCycleSolver(small)
    b.solve(small.b, maxiter=2)
    x1, info1 = a.solve(big.b, maxiter=2)
    assert info0["status"] in (0, 1) and info1["status"] == info0["status"]
    assert np.array_equal(x0, x1)
    a.close()
    b.close()
