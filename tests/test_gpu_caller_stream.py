"""Calls start after the work that their caller has queued on the stream given at setup: here an
input that a kernel still waiting behind 0.2 s of other work is going to write."""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2512_08728_gb300 as pkg
from workloads import make_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()


def _late(values):
    """A tensor that becomes values once the pending work of the current stream is through."""
    t = torch.zeros_like(values)
    torch.cuda.synchronize()
    torch.cuda._sleep(400_000_000)
    t.copy_(values)
    return t


@pytest.mark.parametrize("nrhs,kw", [(1, {}), (3, {}), (3, {"coarse_persistent": False})],
                         ids=["one", "groups", "batched"])
def test_adjoint_of_a_nonsymmetric_operator(nrhs, kw):
    pr = make_problem(3, 1, (8, 4, 4), 3, seed=1)
    rng = np.random.default_rng(4)
    blocks = pr.blocks.copy()
    for sl in range(1, blocks.shape[0]):
        blocks[sl] *= 1.0 + 0.2 * rng.uniform(-1, 1, blocks.shape[1])[:, None, None]
    stream = torch.cuda.Stream()
    s = pkg.KCycleSolver(dataclasses.replace(pr, blocks=blocks), stream=stream.cuda_stream, **kw)
    with torch.cuda.stream(stream):
        g = torch.from_numpy(rng.uniform(-1, 1, (pr.ndof, nrhs) if nrhs > 1 else pr.ndof)).cuda()
        first, _ = s.solve(g, rtol=1e-10, adjoint=True)     # builds the transposed hierarchy
        late = _late(g)
        second, _ = s.solve(late, x0=torch.zeros_like(g), rtol=1e-10, adjoint=True)
    torch.cuda.synchronize()
    s.close()
    assert torch.equal(first, second)


@pytest.mark.parametrize("own", [False, True], ids=["default", "own"])
@pytest.mark.parametrize("call", ["solve", "solve_multi", "adjoint", "apply", "smooth", "restrict", "apply_multi",
                                  "residual"])
def test_every_call_waits(call, own):
    pr = make_problem(3, 1, (8, 4, 4), 3, seed=1)
    stream = torch.cuda.Stream() if own else torch.cuda.default_stream()
    s = pkg.KCycleSolver(pr, stream=stream.cuda_stream or None)
    multi = call in ("solve_multi", "apply_multi")
    v = torch.from_numpy(np.random.default_rng(4).uniform(-1, 1, (pr.ndof, 3) if multi else pr.ndof)).cuda()
    f = {"solve": lambda a: s.solve(a, maxiter=2)[0], "solve_multi": lambda a: s.solve(a, maxiter=2)[0],
         "adjoint": lambda a: s.solve(a, maxiter=2, adjoint=True)[0], "apply": lambda a: s.apply(0, a),
         "smooth": lambda a: s.smooth(0, a), "restrict": lambda a: s.restrict(0, a),
         "apply_multi": lambda a: s.apply_multi(0, a),
         "residual": lambda a: torch.tensor(pkg.kcmg_residual_noalloc(s.ctx, a, torch.zeros_like(a),
                                                                      torch.empty_like(a)))}[call]
    with torch.cuda.stream(stream):
        torch.cuda.synchronize()
        want = f(v)
        got = f(_late(v))
    torch.cuda.synchronize()
    s.close()
    assert want.abs().max() > 0 and torch.equal(want, got)
