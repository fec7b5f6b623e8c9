"""A batched adjoint solve refuses the Schwarz smoother as the batched forward solve does (the
batched engine has block Jacobi only, which it would use in its place)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2512_08728_gb300 as pkg
from workloads import make_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("adjoint", [False, True])
def test_batched_schwarz_is_refused(adjoint):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()
    pr = make_problem(2, 1, (16, 8), 3, seed=1)
    s = pkg.KCycleSolver(pr, smoother="as", omega=0.5, sweeps=2)
    with pytest.raises(pkg.KcmgError) as e:
        s.solve(np.ones((pr.ndof, 2)), adjoint=adjoint)
    assert e.value.status == 5
    x, info = s.solve(pr.b, rtol=1e-10, adjoint=adjoint)
    s.close()
    assert info["status"] == 0
