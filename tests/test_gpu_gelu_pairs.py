"""The packed GELU of the fused network kernels and its derivative against the single ones, bit for bit over every
float of the range that it is used for (|z| <= 13: 2.2e9 of them)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


def test_packed_gelu_has_the_single_ones_bits():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    out_dir = os.path.join(HERE, "cuda", "_build")
    os.makedirs(out_dir, exist_ok=True)
    so = os.path.join(out_dir, "libgelu_pairs_test.so")
    # the flags of the library's own build, as far as they bear on arithmetic
    subprocess.check_call(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "-shared",
                           "-Xcompiler", "-fPIC", "-o", so, os.path.join(HERE, "cuda", "gelu_pairs.cu")])
    compared, differ = ctypes.c_ulonglong(0), ctypes.c_ulonglong(0)
    assert ctypes.CDLL(so).gelu_pairs(ctypes.byref(compared), ctypes.byref(differ)) == 0
    assert compared.value == 2 * (int(np.float32(13.0).view(np.uint32)) + 1)
    assert differ.value == 0
