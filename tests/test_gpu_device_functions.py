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


def residual(lib, a2, I, thr2=0.0, general=0):
    a2, I = torch.from_numpy(a2.astype(np.float32)).cuda(), torch.from_numpy(I.astype(np.float32)).cuda()
    out = torch.empty((a2.numel(), 2), device="cuda")
    torch.cuda.synchronize()
    assert lib.run_residual(ptr(a2), ptr(I), ctypes.c_float(thr2), a2.numel(), general, ptr(out)) == 0
    return out.cpu().numpy()


def operands(n, kind):
    rng = np.random.default_rng(n)
    if kind == "patterns":       # dark field to bright field, counts
        return (10.0 ** rng.uniform(-12, 4, n)).astype(np.float32), rng.poisson(10.0 ** rng.uniform(-2, 4, n)).astype(np.float32)
    if kind == "range":          # everything that is in range, and counts of 0
        a2 = np.ldexp(1 + rng.random(n), rng.integers(-100, 128, n)).astype(np.float32)
        I = np.ldexp(1 + rng.random(n), rng.integers(-149, 128, n)).astype(np.float32) * (rng.random(n) < 0.9)
        a2 = np.where(np.isfinite(a2), a2, np.float32(3.4e38))
        return a2, np.where(np.isfinite(I), I, np.float32(3.4e38)).astype(np.float32)
    k = np.arange(n)             # squares and their neighbours, where roots and quotients are exact or nearly so
    return (((k % 5003 + 1.0) ** 2).astype(np.float32) * np.float32(1 + 2.0 ** -23 * (k % 3 - 1))), ((k % 4099) ** 2).astype(np.float32)


@pytest.mark.parametrize("kind", ["patterns", "range", "squares"])
def test_residual_of_a_far_field_value(lib, kind):
    n = 1 << 20
    a2, I = operands(n, kind)
    out = residual(lib, a2, I).astype(np.float64)
    a, rt = np.sqrt(a2.astype(np.float64)), np.sqrt(I.astype(np.float64))
    q = rt / a
    # a, sqrt(I), their quotient and the difference, each rounded once: half an ulp is at most 2^-24 of the value
    u = 2.0 ** -24 * 1.001
    small = 2.0 ** -149
    assert (np.abs(out[:, 0] - (1 - q)) <= 3 * u * q + u * np.abs(1 - q) + 3 * small).all()
    fits = (rt - a) ** 2 < 3e38
    d = np.sqrt(out[fits, 1])
    e = np.abs(rt - a)[fits]
    assert (np.abs(d - e) <= u * (a + rt)[fits] + 2 * u * e + 2.0 ** -74).all()   # a square below 2^-148 is lost


def test_residual_of_a_far_field_value_of_zero(lib):
    I = np.concatenate([np.arange(4097.0), 10.0 ** np.linspace(-25, 37, 1000)])
    out = residual(lib, np.zeros(I.size), I, thr2=1e-10).astype(np.float64)
    assert (out[:, 0] == 1.0).all()
    assert (np.abs(out[:, 1] - I.astype(np.float32)) <= 3 * 2.0 ** -24 * 1.001 * I).all()   # the root, rounded once, squared


def test_residual_of_operands_out_of_range(lib):
    tiny = np.array([0.0, 1e-45, 1e-44, 1e-38, 7e-31, np.inf, np.nan])
    I = np.array([0.0, 1e-45, 1.0, 3e38, np.inf, np.nan, -1.0])
    a2, I = (x.ravel() for x in np.meshgrid(np.concatenate([tiny, [1.0, 3e38]]), I, indexing="ij"))
    for thr2 in (0.0, 1e-40, 1e-3):
        got, want = residual(lib, a2, I, thr2), residual(lib, a2, I, thr2, general=1)
        out = ~(((a2 == 0) | (a2 >= 2.0 ** -100)) & (a2 < np.inf) & (I >= 0) & (I < np.inf))
        assert np.array_equal(got[out], want[out], equal_nan=True)
        assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want))
