"""Device functions and kernels of the library by themselves, on operands that the public calls reach only at sizes too large
for a test."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    from paper_2205_03902_gb300 import build
    so = str(tmp_path_factory.mktemp("device") / "device_functions.so")
    subprocess.run([build.nvcc(), "-std=c++17", "-O3", build.ARCH, "-shared", "-Xcompiler", "-fPIC", "-I" + build.INCLUDE,
                    "-I" + build.CSRC, os.path.join(HERE, "device_functions.cu"), "-o", so], check=True)
    return ctypes.CDLL(so)


def ptr(t):
    return ctypes.c_void_p(t.data_ptr())


@pytest.mark.parametrize("value,pixels", [(9e17, 511), (9.9e17, 512), (2.5e17, 512), (1e-12, 512)])
def test_training_loss_of_many_pixels_of_one_thread(lib, value, pixels):
    # a thread of the largest image takes 512 pixels: their squares pass FP32's range where no pixel does
    P, blocks = 256 * pixels, 1
    pre = torch.zeros((P, 16), device="cuda")
    target = torch.full((P,), -value, device="cuda")
    g = torch.empty((P, 16), dtype=torch.bfloat16, device="cuda")
    part = torch.empty(blocks, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert lib.run_loss(ptr(pre), ptr(target), 1, ctypes.c_size_t(P), ctypes.c_float(1.0), ptr(g), ptr(part), blocks) == 0
    # FP64: 512 terms of a thread, 5 + 8 sums over the block, two roundings of the mean
    assert abs(part.item() / float(np.float32(value)) ** 2 - 1) < (512 + 15) * 2.0 ** -53
