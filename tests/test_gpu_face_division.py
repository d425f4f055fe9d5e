"""The division of the face evaluation (gamma_face.cuh, div_) against the
quotient in FP64: an approximate reciprocal with a documented error of 2^-22 of
its value and one rounded product (2^-24) differ from it by less than 3e-7;
past 2^126 the reciprocal flushes to zero."""
import ctypes
import importlib.util
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = """
#include "gamma_face.cuh"
__global__ void k(const float* a, const float* b, float* q, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) q[i] = gk::div_(a[i], b[i]);
}
extern "C" int quotients(const float* a, const float* b, float* q, int n)
{
    k<<<(n + 255) / 256, 256>>>(a, b, q, n);
    return (int)cudaDeviceSynchronize();
}
"""


def test_quotients_are_within_the_documented_error(tmp_path):
    spec = importlib.util.spec_from_file_location("_b", os.path.join(ROOT, "paper_1012_1900_gb300", "_build.py"))
    build = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(build)
    src, lib = tmp_path / "q.cu", tmp_path / "q.so"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, "-shared", str(src), "-o", str(lib)],
                   check=True, capture_output=True)
    rng = np.random.default_rng(1)
    n = 1 << 20
    # divisors over all exponents, close to powers of two, and below 2
    b = np.exp2(rng.uniform(0, 126, n))
    b[: n // 4] = np.exp2(rng.integers(0, 126, n // 4)) * (1 + rng.integers(-2, 3, n // 4) * 2.0 ** -23)
    b[n // 4 : n // 2] = rng.uniform(1, 2, n // 4)
    b = np.clip(b, 1, 2.0 ** 126).astype(np.float32)
    # (dividends that keep the quotient a normal number)
    a = (rng.choice([-1.0, 1.0], n) * b.astype(np.float64) * np.exp2(rng.uniform(-60, 1, n))).astype(np.float32)
    b[-3:], a[-3:] = np.float32(2.0 ** 126) * np.float32(1.5), (1.0, -1e30, 0.0)
    ta, tb = torch.from_numpy(a).cuda(), torch.from_numpy(b).cuda()
    q = torch.empty_like(ta)
    f = ctypes.CDLL(str(lib)).quotients
    f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_int]
    torch.cuda.synchronize()
    assert f(ta.data_ptr(), tb.data_ptr(), q.data_ptr(), n) == 0
    q = q.cpu().numpy().astype(np.float64)
    want = a.astype(np.float64) / b.astype(np.float64)
    assert (q[-3:] == 0).all()
    err = np.abs(q - want)[:-3] / np.abs(want[:-3])
    assert err.max() <= 2.0 ** -22 + 2.0 ** -24 + 2.0 ** -46
