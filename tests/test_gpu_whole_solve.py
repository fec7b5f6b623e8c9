"""Small problems, whose whole solve is one persistent kernel, against the per-step kernels
(``coarse_persistent=False`` runs every level on those).

Tolerances: with two levels no level-local criterion takes part, so both run the same steps and
differ by the order of sums.  In FP64 a step rounds to about 100 units in the last place of ||b||
(up to 140 products a row, Gram coefficients over all rows), and the reorthogonalisation test
allows a factor 2 for each of the 3 x 3 columns: 100 x 2^9 x 2e-16 = 1e-11 of ||b||.  FP32 sweeps
round a correction to sqrt(140) x 6e-8 a sweep, 4e-6 after five, and the 9 corrections together
to 4e-5: 1e-4 of ||b||.
"""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2512_08728_gb300 as pkg
from workloads import dense_matrix, make_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()


def _solve(pr, maxiter, rtol, **kw):
    s = pkg.KCycleSolver(pr, **kw)
    x, info = s.solve(pr.b, rtol=rtol, maxiter=maxiter)
    s.close()
    return x, info


# one block for all levels, block 0 alone from the second level on, fewer cells than SMs, more
# cells than SMs with a ragged share, every degree
GRIDS = [(2, 1, (4, 2)), (2, 1, (16, 10)), (2, 2, (30, 14)), (2, 3, (20, 18)), (3, 1, (2, 2, 2)), (3, 1, (10, 6, 6)),
         (3, 2, (6, 4, 8)), (3, 3, (4, 4, 6))]


@pytest.mark.parametrize("d,p,n", GRIDS)
@pytest.mark.parametrize("kw", [{}, {"async_smooth": 2}, {"smoother": "as", "omega": 0.5, "sweeps": 2}, {"sweeps": 1},
                                {"lmax": 4}], ids=["mg", "async", "as", "sweep", "restart"])
@pytest.mark.parametrize("precision", ["fp64", "mixed", "mixed_bf16"])
def test_steps_equal_the_per_step_kernels(d, p, n, kw, precision):
    pr = make_problem(d, p, n, 2, nu_kind="lognormal", seed=3)
    x0, i0 = _solve(pr, 3, 1e-30, precision=precision, coarse_persistent=False, **kw)
    x1, i1 = _solve(pr, 3, 1e-30, precision=precision, **kw)
    assert i1["kernel_launches"] < i0["kernel_launches"]
    tol = (1e-11 if precision == "fp64" else 1e-4) * i0["hist"][0]
    assert np.array_equal(i0["hist_type"], i1["hist_type"]) and i0["iters"] == i1["iters"]
    assert np.abs(i0["hist"] - i1["hist"]).max() <= tol
    A = dense_matrix(pr.blocks, pr.nbr)
    assert np.linalg.norm(A @ (x1 - x0)) <= tol


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_long_basis_and_its_restart(precision):
    """More columns than a block keeps coefficients of in shared memory, then a restart."""
    pr = make_problem(2, 2, (16, 16), 2, nu_kind="jump", seed=4)
    kw = dict(precision=precision, sweeps=1, omega=0.3, lmax=90)
    x, info = _solve(pr, 400, 1e-10, **kw)
    assert info["status"] == 0 and info["kernel_launches"] < 40 and info["iters"] > 20
    A = dense_matrix(pr.blocks, pr.nbr)
    assert np.linalg.norm(pr.b - A @ x) <= 1.01e-10 * np.linalg.norm(pr.b)


@pytest.mark.parametrize("d,p,n,lv", [(2, 1, (16, 8), 3), (3, 1, (4, 4, 8), 3)])
def test_blocks_towards_missing_neighbours_are_not_read(d, p, n, lv):
    pr = make_problem(d, p, n, lv, nu_kind="jump", seed=2)
    blocks = pr.blocks.copy()
    for s in range(1, blocks.shape[0]):
        blocks[s, np.asarray(pr.nbr).reshape(blocks.shape[1], -1)[:, s - 1] < 0] = 7.0
    x0, _ = _solve(pr, 4, 1e-30)
    x1, _ = _solve(dataclasses.replace(pr, blocks=blocks), 4, 1e-30)
    assert np.isfinite(x0).all() and np.array_equal(x0, x1)
