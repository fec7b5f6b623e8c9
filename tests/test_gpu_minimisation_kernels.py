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


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    path = pkg.build()
    so = str(tmp_path_factory.mktemp("kernels") / "minimisation_kernels.so")
    here = os.path.dirname(os.path.abspath(__file__))
    subprocess.run([B._nvcc(), *B.ARCH, *B.FLAGS, "-I", B.CSRC, "-shared", "-o", so,
                    os.path.join(here, "minimisation_kernels.cu")], check=True)
    C.CDLL(path, mode=C.RTLD_GLOBAL)
    return C.CDLL(so)


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
