"""x of Alg. 1 from the corrections as they came and R y = alpha, at basis lengths around a block's
threads, against numpy's least squares.

The corrections are random: A Z (768 x 600) has a condition number of 3e4, so that R y = alpha loses
up to that factor on the sums' rounding, 1e-15 x 3e4 x a few = 1e-10 of ||r0||; 1e-9 is asked for.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2512_08728_gb300 as pkg
from workloads import dense_matrix, make_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ncorr", [0, 1, 2, 33, 512, 513, 600])
def test_iterate_of_a_long_basis(ncorr):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()
    pr = make_problem(2, 1, (16, 16), 3, nu_kind="jump", seed=1)
    A = dense_matrix(pr.blocks, pr.nbr)
    rng = np.random.default_rng(8)
    zs, x0 = rng.standard_normal((ncorr, pr.ndof)), rng.standard_normal(pr.ndof)
    s = pkg.KCycleSolver(pr, lmax=700)
    x, r, l = s.rm_sequence(0, pr.b, x0, zs)
    s.close()
    r0 = pr.b - A @ x0
    scale = np.linalg.norm(r0)
    assert l == ncorr and np.linalg.norm(pr.b - A @ x - r) <= 1e-9 * scale
    if ncorr:
        best = r0 - (A @ zs.T) @ np.linalg.lstsq(A @ zs.T, r0, rcond=None)[0]
        assert np.linalg.norm(r - best) <= 1e-9 * scale
