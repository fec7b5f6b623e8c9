"""Single kernels of the residual minimisation (Alg. 1), called with vectors and states of the test's
own (minimisation_kernels.cu, compiled here against the library)."""
import ctypes as C
import importlib
import math
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2512_08728_gb300 as pkg

B = importlib.import_module("paper_2512_08728_gb300.build")   # pkg.build is the function
pytestmark = pytest.mark.gpu
TYPES = {"f32": np.float32, "f64": np.float64}


def _compile(source, folder, *flags):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    path = pkg.build()
    so = str(folder.mktemp("kernels") / (source + ".so"))
    here = os.path.dirname(os.path.abspath(__file__))
    subprocess.run([B._nvcc(), *B.ARCH, *B.FLAGS, *flags, "-I", B.CSRC, "-shared", "-o", so,
                    os.path.join(here, source + ".cu")], check=True)
    C.CDLL(path, mode=C.RTLD_GLOBAL)
    return C.CDLL(so)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return _compile("minimisation_kernels", tmp_path_factory)


@pytest.fixture(scope="module")
def batched(tmp_path_factory):
    return _compile("batched_minimisation_kernels", tmp_path_factory, "-Xptxas", "-O1")


def _p(a):
    return a.ctypes.data_as(C.c_void_p)


# FP32 vectors whose squares vanish beside 1 in an FP32 sum: 2^-26 against half a unit of 2^-24.  The
# FP64 sum's error is at most a unit of 2^-53 an addition, 150 of them a thread and 300 in the trees.
@pytest.mark.parametrize("t", ["f32", "f64"])
@pytest.mark.parametrize("N", [2 * 256 * 64, 256 * 64 + 1, 700])
def test_residual_norm_of_an_update_sums_in_fp64(lib, t, N):
    T = TYPES[t]
    r = np.full(N, 2.0**-13, dtype=T)
    r[:min(N, 512)] = 1.0
    want = math.sqrt(math.fsum(float(v) ** 2 for v in r))
    W, w, z, h = np.zeros((1, N), T), np.ones(N, T), np.ones(N, T), np.zeros(1)
    rn = C.c_double()
    assert getattr(lib, "update_" + t)(N, 0, _p(W), _p(w), _p(z), _p(h), C.c_double(1.0), C.c_double(0.0), _p(r), 1,
                                       C.byref(rn)) == 0
    assert abs(rn.value - want) <= 450 * 2.0**-53 * want


# the same for the persistent kernel's sums: eight lanes a sum, so the first 16 entries of every
# vector are the ones that the others vanish beside; FP64 sums of N / 8 terms a lane
@pytest.mark.parametrize("t", ["f32", "f64"])
@pytest.mark.parametrize("N,l", [(2400, 0), (2400, 5), (2400, 20), (27, 2)])
def test_norms_of_the_persistent_kernel_sum_in_fp64(lib, t, N, l):
    T = TYPES[t]
    w, r = np.full(N, 2.0**-13, dtype=T), np.full(N, -(2.0**-13), dtype=T)
    w[:16], r[:16] = 1.0, 1.0
    W = np.random.default_rng(1).standard_normal((l + 1, N)).astype(T)
    out = np.zeros(l + 4)
    assert getattr(lib, "dots_" + t)(N, l, _p(W), _p(w), _p(r), _p(out)) == 0
    tol = (N / 8 + 5) * 2.0**-53
    for got, a, b in ((out[l], w, w), (out[l + 1], w, r), (out[l + 2], r, r)) + (((out[l + 3], W[l - 1], r),) if l else ()):
        terms = a.astype(np.float64) * b.astype(np.float64)
        assert abs(got - math.fsum(terms)) <= tol * np.abs(terms).sum()
    # the columns' sums are in the vectors' type: N / 16 terms an accumulator
    eps = 2.0**-24 if t == "f32" else 2.0**-53
    for c in range(l):
        terms = W[c].astype(np.float64) * w.astype(np.float64)
        assert abs(out[c] - math.fsum(terms)) <= (N / 16 + 8) * eps * np.abs(terms).sum()


def _basis(T, N, l, left, seed=3):
    """l orthonormal columns, a vector with the share ``left`` of its square outside them, and a residual
    orthogonal to them, all rounded to T."""
    rng = np.random.default_rng(seed)
    Q = np.linalg.qr(rng.standard_normal((N, l + 2)))[0].T
    c = rng.standard_normal(l)
    w = math.sqrt(1 - left) * (c / np.linalg.norm(c)) @ Q[:l] + math.sqrt(left) * Q[l]
    W = np.zeros((l + 1, N), T)
    W[:l] = Q[:l]
    return W, w.astype(T), (0.6 * Q[l] + 0.8 * Q[l + 1]).astype(T)


# After the second pass the new column has unit length and r is orthogonal to it, to the rounding of the
# sums in the vectors' type: 13 units for a thread's products and sums (12 terms at most), 16 with the
# normalisation and the storing, times 4 where the norm is ||w'||^2 - ||h2||^2 with a quarter left.
@pytest.mark.parametrize("t", ["f32", "f64"])
@pytest.mark.parametrize("N,nblk", [(3000, 1), (3000, 7), (5001, 4)])
@pytest.mark.parametrize("left", [0.9, 0.3, 0.2, 1e-2, 2e-4])
def test_column_after_the_second_pass(lib, t, N, nblk, left):
    T, l = TYPES[t], 9
    eps = np.finfo(T).eps / 2
    W, w, r = _basis(T, N, l, left)
    rn0 = np.linalg.norm(r.astype(np.float64))
    g, a, rn = C.c_double(), C.c_double(), C.c_double()
    assert getattr(lib, "second_pass_" + t)(N, l, _p(W), _p(w), _p(w), C.c_double(4.0), _p(r), nblk, C.byref(g),
                                            C.byref(a), C.byref(rn)) == 0
    wl, rl = W[l].astype(np.float64), r.astype(np.float64)
    tol = 4 * 16 * eps
    assert abs(np.linalg.norm(wl) - 1) <= tol
    assert abs(rl @ wl) <= tol * rn0
    assert abs(rn.value - np.linalg.norm(rl)) <= 64 * 2.0**-53
    assert abs(g.value * math.sqrt(left) - 1) <= 32 * eps / left and abs(a.value - 0.6) <= 32 * eps / left


# what is left is below brk = 1e-14 of ||A z||: discarded, the residual as it was
@pytest.mark.parametrize("t", ["f32", "f64"])
def test_dependent_after_the_second_pass(lib, t):
    T, N, l = TYPES[t], 3000, 9
    W, w, r = _basis(T, N, l, 1e-2)
    before = r.copy()
    g, a, rn = C.c_double(), C.c_double(), C.c_double()
    assert getattr(lib, "second_pass_" + t)(N, l, _p(W), _p(w), _p(w), C.c_double(1e28), _p(r), 3, C.byref(g),
                                            C.byref(a), C.byref(rn)) == 2
    assert np.array_equal(r, before) and abs(rn.value - np.linalg.norm(r.astype(np.float64))) <= 64 * 2.0**-53


# the batched kernels: every right-hand side has its own basis and its own share left; one takes no part
# (its correction is discarded already).  A thread sums N / (8 blocks) rows.
@pytest.mark.parametrize("blocks,in_kernel", [(1, 1), (5, 1), (5, 0)])
def test_columns_after_the_second_pass(batched, blocks, in_kernel):
    N, l, left = 3000, 9, [0.9, 0.3, 0.2, 1e-3, 1e-6, 0.5]
    R, part = len(left), np.array([1, 1, 1, 1, 1, 0], dtype=np.int32)
    cols = [_basis(np.float64, N, l, s, seed=k) for k, s in enumerate(left)]
    W, w, r = (np.ascontiguousarray(np.stack([c[k] for c in cols], axis=-1)) for k in range(3))
    rng = np.random.default_rng(11)
    Z, z, x = rng.standard_normal((l + 1, N, R)), rng.standard_normal((N, R)), rng.standard_normal((N, R))
    W0, r0, x0 = W.copy(), r.copy(), x.copy()
    ln, rn = np.zeros(R, dtype=np.int32), np.zeros(R)
    assert batched.batched_second_pass(N, R, l, _p(W), _p(Z), _p(w), _p(z), C.c_double(4.0), _p(x), _p(r), _p(part),
                                       in_kernel, blocks, _p(ln), _p(rn)) == 0
    tol = 4 * (N / (8 * blocks) + 16) * 2.0**-53
    for k in range(R):
        if not part[k]:
            assert ln[k] == l and np.array_equal(r[:, k], r0[:, k]) and np.array_equal(x[:, k], x0[:, k])
            continue
        wl = W[l, :, k]
        assert ln[k] == l + 1 and abs(np.linalg.norm(wl) - 1) <= tol and abs(r[:, k] @ wl) <= tol
        assert abs(rn[k] - np.linalg.norm(r[:, k])) <= 2 * tol
        h = W0[:l, :, k] @ w[:, k]
        g, al = 1.0 / np.linalg.norm(w[:, k] - h @ W0[:l, :, k]), (r0[:, k] - r[:, k]) @ wl
        zl = g * (z[:, k] - h @ Z[:l, :, k])
        assert np.abs(Z[l, :, k] - zl).max() <= tol / left[k] * np.abs(zl).max()
        assert np.abs(x[:, k] - x0[:, k] - al * Z[l, :, k]).max() <= tol * np.abs(zl).max()


# The persistent kernel makes further passes until at least a quarter of the square is left, and discards
# what the passes have brought down to brk = 1e-14 of ||A z||; no norm is a difference of less.
TAKE, AGAIN, DISCARD = 0, 1, 2


@pytest.mark.parametrize("l,passes,n2,left,want", [
    (0, 0, 1.0, 1.0, TAKE), (5, 0, 1.0, 0.26, TAKE), (5, 0, 1.0, 0.24, AGAIN), (5, 0, 0.0, 0.0, DISCARD),
    (5, 0, math.nan, 1.0, DISCARD), (5, 0, 1.0, -1e-15, AGAIN), (5, 1, 1e-20, 0.9, TAKE), (5, 1, 1e-20, 0.1, AGAIN),
    (5, 1, 1e-20, -1e-7, AGAIN), (5, 1, 1e-29, 1.0, DISCARD), (5, 2, 1e-10, 0.1, AGAIN), (5, 3, 1e-10, 0.1, AGAIN),
    (5, 3, 1e-10, 0.3, TAKE), (5, 3, 1e-29, 0.1, DISCARD), (5, 48, 1e-10, 0.1, DISCARD), (5, 48, 1e-10, 0.3, TAKE)])
def test_what_follows_a_pass(lib, l, passes, n2, left, want):
    h = math.sqrt(n2 * (1.0 - left)) if n2 == n2 else 0.0
    f = lib.decide
    assert f(l, passes, C.c_double(1.0), C.c_double(n2), C.c_double(h if l else 0.0)) == want
