"""Batched solves of small problems, every column on its own group of blocks of one kernel, against
the batched kernels (``coarse_persistent=False``).

Tolerances as for the single column's whole solve (test_gpu_whole_solve.py): two levels run the
same steps and differ by the order of sums, 1e-11 of ||b|| in FP64; 1e-4 where sweeps are FP32.
"""
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


def _solve(pr, b, x0, maxiter, rtol=1e-30, atol=0.0, **kw):
    s = pkg.KCycleSolver(pr, **kw)
    x, info = s.solve(b, x0=x0, rtol=rtol, atol=atol, maxiter=maxiter)
    s.close()
    return x, info


# one block a column, fewer and more cells than a group has blocks, more columns than groups fit
# (the shares of 26 x 26 x 10 cells at 32 columns need more than an equal part of the SMs)
@pytest.mark.parametrize("d,p,n,nrhs", [(2, 1, (4, 2), 2), (2, 1, (16, 10), 32), (2, 2, (30, 14), 5), (2, 3, (20, 18), 3),
                                        (3, 1, (26, 26, 10), 32), (3, 2, (6, 4, 8), 17), (3, 3, (4, 4, 6), 24)])
@pytest.mark.parametrize("kw", [{}, {"async_smooth": 2}, {"lmax": 4}, {"lmax": 70, "sweeps": 1}],
                         ids=["mg", "async", "restart", "long"])
@pytest.mark.parametrize("precision", ["fp64", "mixed", "mixed_bf16"])
def test_steps_equal_the_batched_kernels(d, p, n, nrhs, kw, precision):
    pr = make_problem(d, p, n, 2, nu_kind="lognormal", seed=3)
    rng = np.random.default_rng(7)
    b, x0 = rng.uniform(-1, 1, (pr.ndof, nrhs)), 1e-3 * rng.uniform(-1, 1, (pr.ndof, nrhs))
    xa, ia = _solve(pr, b, x0, 3, precision=precision, coarse_persistent=False, **kw)
    xb, ib = _solve(pr, b, x0, 3, precision=precision, **kw)
    assert ib["kernel_launches"] == 1 < ia["kernel_launches"]
    assert ia["iters"] == ib["iters"] and ia["status"] == ib["status"]
    assert np.isclose(ia["res0"], ib["res0"], rtol=1e-12)
    assert np.array_equal(ib["hist"], [nrhs] * 4)
    tol = 1e-11 if precision == "fp64" else 1e-4
    s = pkg.KCycleSolver(pr)
    for j in range(nrhs):
        r0 = np.linalg.norm(b[:, j] - s.apply(0, x0[:, j]))
        assert np.linalg.norm(s.apply(0, xa[:, j] - xb[:, j])) <= tol * r0
    s.close()


@pytest.mark.parametrize("kw", [{}, {"async_smooth": 3}], ids=["mg", "async"])
@pytest.mark.parametrize("precision", ["fp64", "mixed", "mixed_bf16"])
def test_where_the_single_solve_keeps_its_finest_level_kernels(kw, precision):
    """A finest level too large (or a cycle too parallel) for one column's whole solve in the
    kernel; one iteration on the level between, which doubles the steps and the tolerance."""
    pr = make_problem(3, 2, (16, 16, 8), 3, nu_kind="lognormal", seed=3)
    b = np.random.default_rng(7).uniform(-1, 1, (pr.ndof, 3))
    kw = dict(kw, precision=precision, lvl_rtol=[0.0] * 3, lvl_maxit=[1] * 3)
    xa, ia = _solve(pr, b, None, 3, coarse_persistent=False, **kw)
    xb, ib = _solve(pr, b, None, 3, **kw)
    assert ib["kernel_launches"] == 1 < ia["kernel_launches"] and ia["level_iters"][:2] == ib["level_iters"][:2]
    s = pkg.KCycleSolver(pr)
    for j in range(3):
        assert (np.linalg.norm(s.apply(0, xa[:, j] - xb[:, j]))
                <= 2 * (1e-11 if precision == "fp64" else 1e-4) * np.linalg.norm(b[:, j]))
    s.close()


def test_columns_stop_and_fail_by_themselves():
    """A zero column, one that starts at its solution and one that is not finite leave the others
    what they are alone, in either form."""
    pr = make_problem(2, 1, (16, 8), 3, nu_kind="jump", seed=4)
    A = dense_matrix(pr.blocks, pr.nbr)
    rng = np.random.default_rng(5)
    b = rng.uniform(-1, 1, (pr.ndof, 4))
    b[:, 1] = 0.0
    x0 = np.zeros_like(b)
    x0[:, 2] = np.linalg.solve(A, b[:, 2])
    for precision in ("fp64", "mixed"):
        x, info = _solve(pr, b, x0, 200, rtol=1e-9, atol=1e-10, precision=precision)
        assert info["status"] == 0 and np.array_equal(x[:, 2], x0[:, 2])
        assert np.all(x[:, 1] == 0.0)
        for j in (0, 3):
            assert np.linalg.norm(b[:, j] - A @ x[:, j]) <= 1.01e-9 * np.linalg.norm(b[:, j])
        bad = b.copy()
        bad[3, 3] = np.nan
        xn = x0.copy()
        s = pkg.KCycleSolver(pr, precision=precision)
        with pytest.raises(pkg.KcmgError) as e:
            pkg.kcmg_solve(s.ctx, bad, xn, rtol=1e-9, atol=1e-10, maxiter=200)
        s.close()
        assert e.value.status == 3 and np.array_equal(xn[:, :3], x[:, :3])


def test_tuning_and_other_batched_calls_after_a_small_solve():
    pr = make_problem(3, 1, (6, 4, 4), 2, nu_kind="jump", seed=4)
    b = np.random.default_rng(5).uniform(-1, 1, (pr.ndof, 6))
    s = pkg.KCycleSolver(pr)
    with pytest.raises(pkg.KcmgError):
        s.mrhs_tuning()
    x1, i1 = s.solve(b, rtol=1e-10, maxiter=100)
    assert i1["kernel_launches"] == 1 and s.mrhs_tuning()["nrhs"] == 6
    s.solve(b[:, :3], rtol=1e-10, maxiter=100)
    assert s.mrhs_tuning()["nrhs"] == 3
    x2, _ = s.solve(torch.from_numpy(b).cuda(), rtol=1e-10, maxiter=100)
    assert np.array_equal(x1, x2.cpu().numpy())
    s.close()
