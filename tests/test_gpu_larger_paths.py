"""Paths that small problems no longer take by default (their whole solve is one kernel): the graph of
the cycle above the persistent kernel, and the batched solve's loop over the batched kernels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2512_08728_gb300 as pkg
from oracle import OracleSolver
from workloads import make_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()


@pytest.mark.parametrize("kw", [{}, {"async_smooth": 4}], ids=["mg", "async"])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_graph_and_eager_are_bitwise_identical_above_the_persistent_kernel(kw, precision):
    pr = make_problem(3, 2, (16, 16, 8), 3, seed=5)
    out = []
    for g in (False, True, True):
        s = pkg.KCycleSolver(pr, precision=precision, use_graph=g, **kw)
        x, info = s.solve(pr.b, rtol=1e-10)
        x2, _ = s.solve(pr.b, rtol=1e-10)
        assert s.kernel_report()["coarse_launches"] == 2 * info["iters"]   # one a cycle, not one a solve
        s.close()
        assert info["status"] == 0 and np.array_equal(x, x2)
        out.append(x)
    assert np.array_equal(out[0], out[1]) and np.array_equal(out[1], out[2])


@pytest.mark.parametrize("d,p,n,lv,nrhs", [(2, 1, (16, 16), 3, 32), (3, 2, (8, 8, 8), 3, 8), (3, 2, (6, 6, 2), 2, 5),
                                           (2, 2, (16, 16), 3, 12)])
@pytest.mark.parametrize("precision", ["fp64", "mixed", "mixed_bf16"])
@pytest.mark.parametrize("kw", [{}, {"async_smooth": 3}], ids=["mg", "async"])
def test_batched_loop_matches_oracle_per_column(d, p, n, lv, nrhs, precision, kw):
    pr = make_problem(d, p, n, lv, nu_kind="jump", seed=0, nrhs=nrhs)
    s = pkg.KCycleSolver(pr, precision=precision, coarse_persistent=False, **kw)
    X, info = s.solve(pr.b, rtol=9e-11, maxiter=2000)   # the oracle's plain residual rounds differently
    s.close()
    assert info["status"] == 0 and info["kernel_launches"] > 100 and info["rel_res"] <= 1e-10
    orc = OracleSolver.from_problem(pr)
    for j in range(0, nrhs, 3):
        x, io = orc.solve(pr.b[:, j], rtol=1e-10, maxiter=600)
        assert io["status"] == 0 and np.linalg.norm(X[:, j] - x) <= 1e-8 * np.linalg.norm(x)
        assert np.linalg.norm(pr.b[:, j] - orc.apply(0, X[:, j])) <= 1.1e-10 * np.linalg.norm(pr.b[:, j])
