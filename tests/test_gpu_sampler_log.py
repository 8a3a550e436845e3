"""-ln u of the FP32 sampler against 64 bits: no further off than CUDA's logf (for
u < 1/2) and log1pf of the exact complement, over all u and over each factor
of two of 1 - u; the words at the ends of the range and around powers of two."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))
SRC = os.path.join(os.path.dirname(HERE), "paper_1005_5405_gb300", "csrc")


@pytest.fixture(scope="module")
def errors(tmp_path_factory):
    nvcc = "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    so = str(tmp_path_factory.mktemp("neglog") / "neglog.so")
    subprocess.run([nvcc, "-gencode=arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "-cudart", "shared", "-I" + SRC, "-I" + os.path.join(os.path.dirname(HERE), "include"),
                    "-o", so, os.path.join(HERE, "_neglog_ref.cu")], check=True)
    lib = C.CDLL(so)

    def run(words):
        x = np.ascontiguousarray(words, dtype=np.uint32)
        a, b = np.empty(len(x), np.float32), np.empty(len(x), np.float32)
        assert lib.neglog_ref(len(x), *(C.c_void_p(v.ctypes.data) for v in (x, a, b))) == 0
        w = (2.0 ** 32 - 1 - x.astype(float) + 0.5) / 2.0 ** 32         # 1 - u, exact
        exact = np.where(w > 0.5, -np.log((x.astype(float) + 0.5) / 2.0 ** 32), -np.log1p(-w))
        return np.abs(a - exact) / exact, np.abs(b - exact) / exact

    return run


def test_over_all_u(errors):
    got, ref = errors(np.random.default_rng(1).integers(0, 2 ** 32, 1 << 23))
    assert got.max() <= ref.max() and np.sqrt(np.mean(got ** 2)) <= np.sqrt(np.mean(ref ** 2))


@pytest.mark.parametrize("k", range(1, 32))
def test_near_one(errors, k):
    """1 - u from 2^-(k+1) to 2^-k."""
    words = 2 ** 32 - 1 - np.unique(np.random.default_rng(k).integers(2 ** (31 - k), 2 ** (32 - k), 1 << 18))
    got, ref = errors(words)
    assert got.max() <= ref.max()


def test_ends_and_powers_of_two(errors):
    words = [2 ** k + d for k in range(33) for d in (-2, -1, 0, 1) if 0 <= 2 ** k + d < 2 ** 32]
    got, _ = errors(words)
    # Rounding of v and of the result (2^-24 each, 1.44 the condition at v = 1/2)
    # and an ulp of log1pf.
    assert got.max() <= (1.44 + 1 + 2) * 2.0 ** -24
