"""The device's double reciprocal (csrc/grf_point.cuh, approximate reciprocal and two Newton-Raphson steps)
against CUDA's correctly rounded one.

Bound: with the second step's remainder below 2^-70, the result differs from the correctly rounded one only
where the quotient lies within 2^-70 relative of a rounding boundary, and then by one unit in the last place.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

SRC = """
#include "grf_point.cuh"
__global__ void k(const double* x, double* own, double* cuda, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) { own[i] = grf::recip(x[i]); cuda[i] = __drcp_rn(x[i]); }
}
extern "C" int run(const double* x, double* own, double* cuda, int n) {
    k<<<(n + 255) / 256, 256>>>(x, own, cuda, n);
    return cudaDeviceSynchronize() == cudaSuccess && cudaGetLastError() == cudaSuccess ? 0 : 1;
}
"""


@pytest.mark.gpu
def test_reciprocal_against_the_correctly_rounded_one(tmp_path):
    torch = pytest.importorskip("torch")
    from paper_2309_06225_gb300 import build
    src, lib = tmp_path / "recip.cu", tmp_path / "recip.so"
    src.write_text(SRC)
    subprocess.check_call([build.NVCC] + build.ARCH + build.FLAGS + ["-shared", str(src), "-o", str(lib)])
    L = C.CDLL(os.fspath(lib))
    L.run.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p, C.c_int]
    rng = np.random.default_rng(11)
    n = 1 << 22
    x = rng.uniform(1.0, 2.0, n)
    x[: n // 2] *= 2.0 ** rng.integers(-1000, 1000, n // 2)
    x[:4096] = 1.0 + 2.0 ** -52 * np.arange(4096)          # just above and below powers of two
    x[4096:8192] = 2.0 - 2.0 ** -52 * (1 + np.arange(4096))
    x *= rng.choice([-1.0, 1.0], n)
    t = torch.from_numpy(x).cuda()
    own, ref = torch.empty_like(t), torch.empty_like(t)
    torch.cuda.synchronize()
    assert L.run(t.data_ptr(), own.data_ptr(), ref.data_ptr(), n) == 0
    ulps = np.abs(own.cpu().numpy().view(np.int64) - ref.cpu().numpy().view(np.int64))
    assert ulps.max() <= 1
    assert np.mean(ulps != 0) <= 2.0 ** -15                # 2^-70 against half a unit of 2^-53, and a margin of 2
