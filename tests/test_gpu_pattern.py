"""Finest-level kernels that store and multiply only the nonzero entries of a tensor basis's
blocks (pattern_ops.cuh) against the dense kernels.

A row sees its nonzero entries in the dense kernels' order and the products left out are exact
zeros, so every result is the dense kernels' bit for bit.  The dense kernels run when a block has
an entry outside the pattern; the smallest denormal as that entry changes no sum.
"""
import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2512_08728_gb300 as pkg
from workloads import make_problem

pytestmark = pytest.mark.gpu

# every (dimension, degree); cells that leave a ragged last group of 32, and fewer than 32
GRIDS = [(2, 1, (16, 10)), (2, 2, (6, 4)), (2, 3, (10, 14)), (3, 1, (6, 4, 2)), (3, 2, (6, 6, 2)), (3, 2, (2, 2, 4)),
         (3, 3, (4, 6, 2))]


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    pkg.build()


def _pair(d, p, n, precision, **kw):
    """Contexts of the same operator on the pattern kernels and on the dense kernels.  The blocks
    are random within the pattern, so that a transposed or misplaced entry shows."""
    pr = make_problem(d, p, n, 2, nu_kind="lognormal", seed=5)
    rng = np.random.default_rng(6)
    blocks = pr.blocks * rng.uniform(0.5, 1.5, pr.blocks.shape)
    dense = blocks.copy()
    s, K = 2, 0                       # the +x neighbour of cell 0 exists on every grid
    i, j = np.argwhere(pr.blocks[s, K] == 0.0)[0]
    dense[s, K, i, j] = 5e-324
    make = lambda b: pkg.KCycleSolver(dataclasses.replace(pr, blocks=b), precision=precision, **kw)
    return pr, make(blocks), make(dense), rng


@pytest.mark.parametrize("d,p,n", GRIDS)
@pytest.mark.parametrize("precision", ["fp64", "mixed", "mixed_bf16", "ir32"])
def test_pattern_operator_and_sweeps_equal_the_dense_kernels(d, p, n, precision):
    pr, a, b, rng = _pair(d, p, n, precision)
    x = rng.standard_normal(pr.ndof)
    xd = torch.from_numpy(x).cuda()
    for op in ([0] if precision == "fp64" else [0, 1]):
        ya, yb = a.apply(0, x, op=op), b.apply(0, x, op=op)
        assert np.array_equal(ya, yb)
        assert np.array_equal(a.apply(0, xd, op=op).cpu().numpy(), ya)   # on the caller's vectors
    za = a.smooth(0, x)
    assert np.array_equal(za, b.smooth(0, x))
    assert np.array_equal(a.smooth(0, xd).cpu().numpy(), za)
    a.close()
    b.close()


@pytest.mark.parametrize("sweeps", [1, 2])
def test_pattern_sweeps_with_fp32_conversions_in_one_and_two_sweeps(sweeps):
    pr, a, b, rng = _pair(3, 2, (6, 6, 2), "mixed", sweeps=sweeps)
    r = rng.standard_normal(pr.ndof)
    assert np.array_equal(a.smooth(0, r), b.smooth(0, r))
    a.close()
    b.close()


@pytest.mark.parametrize("d,p,n", GRIDS)
def test_pattern_residuals_equal_the_dense_kernels(d, p, n):
    pr, a, b, rng = _pair(d, p, n, "fp64")
    store = torch.from_numpy(rng.standard_normal(pr.ndof + 1)).cuda()
    rhs = torch.from_numpy(pr.b).cuda()
    ra, rb = torch.empty_like(rhs), torch.empty_like(rhs)
    for x in (store[:-1], store[1:]):              # on and off the 16-byte boundary
        na = pkg.kcmg_residual_noalloc(a.ctx, rhs, x, ra)
        nb = pkg.kcmg_residual_noalloc(b.ctx, rhs, x, rb)
        assert torch.equal(ra, rb)
        assert abs(na - nb) <= 1e-14 * nb          # other partial sums
    # the compensated residual and its norm: a solve of no cycles reports them
    x0 = store[:-1].clone()
    ia, ib = (pkg.kcmg_solve(s.ctx, rhs, x0.clone(), 1e-10, 0.0, 0) for s in (a, b))
    assert abs(ia["res0"] - ib["res0"]) <= 1e-14 * ib["res0"]
    a.close()
    b.close()


@pytest.mark.parametrize("d,p,n", [(2, 3, (10, 14)), (3, 2, (6, 6, 2)), (3, 3, (4, 6, 2))])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_pattern_kernels_keep_infinities_and_nans_of_the_dense_products(d, p, n, precision):
    pr, a, b, rng = _pair(d, p, n, precision)
    for bad in (np.inf, -np.inf, np.nan):
        x = rng.standard_normal(pr.ndof)
        x[[3, pr.ndof // 2 + 1]] = bad
        ya, yb = a.apply(0, x), b.apply(0, x)
        assert np.array_equal(ya, yb, equal_nan=True) and not np.isfinite(ya).all() and np.isfinite(ya).any()
        assert np.array_equal(a.smooth(0, x), b.smooth(0, x), equal_nan=True)
    a.close()
    b.close()


def test_calls_on_overlapping_and_misaligned_vectors_are_staged():
    pr, a, b, rng = _pair(3, 2, (6, 6, 2), "fp64")
    x = torch.from_numpy(rng.standard_normal(pr.ndof + 1)).cuda()
    lib = pkg.load_library()
    for call in (lambda s, u, v: lib.kcmg_apply(s.ctx, 0, 0, u, v), lambda s, u, v: lib.kcmg_smooth(s.ctx, 0, u, v)):
        want = torch.empty(pr.ndof, dtype=torch.float64, device="cuda")
        assert call(b, x[:-1].clone().data_ptr(), want.data_ptr()) == 0
        buf = x.clone()
        assert call(a, buf.data_ptr(), buf.data_ptr()) == 0            # in place
        assert torch.equal(buf[:-1], want)
        src = torch.cat([x[:1], x[:-1]])                                # 8 bytes off the boundary
        out = torch.empty(pr.ndof + 1, dtype=torch.float64, device="cuda")
        assert call(a, src[1:].data_ptr(), out[1:].data_ptr()) == 0
        assert torch.equal(out[1:], want)
    a.close()
    b.close()


@pytest.mark.parametrize("d,p,n", GRIDS)
@pytest.mark.parametrize("nrhs", [2, 8, 9, 32])
def test_batched_pattern_kernels_equal_the_dense_kernels(d, p, n, nrhs, monkeypatch):
    """FP64 against the batched dense kernels; FP32 against the CUDA-core sweep (the forced sweep
    kernel runs on every level).  Columns that fill a lane group, one more, and a full warp."""
    pr, a, b, rng = _pair(d, p, n, "fp64")
    X = rng.standard_normal((pr.ndof, nrhs))
    X[[3, pr.ndof // 2], 1] = np.inf, np.nan            # in one column only
    assert np.array_equal(a.apply_multi(0, X), b.apply_multi(0, X), equal_nan=True)
    assert np.array_equal(a.smooth_multi(0, X), b.smooth_multi(0, X), equal_nan=True)
    Xd = torch.from_numpy(X).cuda()                     # on the caller's vectors
    assert np.array_equal(a.apply_multi(0, Xd).cpu().numpy(), a.apply_multi(0, X), equal_nan=True)
    a.close()
    b.close()
    for precision in ("mixed", "mixed_bf16"):
        pr, a, b, rng = _pair(d, p, n, precision)
        za = a.smooth_multi(0, X)
        monkeypatch.setenv("KCMG_SWEEP", "simt")
        zb = b.smooth_multi(0, X)
        monkeypatch.delenv("KCMG_SWEEP")
        assert np.array_equal(za, zb, equal_nan=True)
        assert np.array_equal(a.smooth_multi(0, Xd).cpu().numpy(), za, equal_nan=True)
        a.close()
        b.close()


@pytest.mark.parametrize("sweeps", [1, 2])
def test_batched_pattern_sweeps_with_fp32_conversions(sweeps, monkeypatch):
    pr, a, b, rng = _pair(3, 2, (6, 6, 2), "mixed", sweeps=sweeps)
    R = rng.standard_normal((pr.ndof, 8))
    if sweeps == 1:
        monkeypatch.setenv("KCMG_SWEEP", "simt")        # both on the kernel that a single sweep takes
    za = a.smooth_multi(0, R)
    monkeypatch.setenv("KCMG_SWEEP", "simt")
    assert np.array_equal(za, b.smooth_multi(0, R))
    a.close()
    b.close()
