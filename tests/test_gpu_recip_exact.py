"""The device's double reciprocal (csrc/grf_point.cuh): the correctly rounded one on ordinary values, and a division's
results at the ends of the range."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from test_gpu_recip import SRC

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    torch = pytest.importorskip("torch")
    from paper_2309_06225_gb300 import build
    d = tmp_path_factory.mktemp("recip")
    (d / "r.cu").write_text(SRC)
    subprocess.check_call([build.NVCC] + build.ARCH + build.FLAGS + ["-shared", str(d / "r.cu"), "-o", str(d / "r.so")])
    L = C.CDLL(os.fspath(d / "r.so"))
    L.run.argtypes = [C.c_void_p, C.c_void_p, C.c_void_p, C.c_int]

    def f(x):
        t = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        own, ref = torch.empty_like(t), torch.empty_like(t)
        torch.cuda.synchronize()
        assert L.run(t.data_ptr(), own.data_ptr(), ref.data_ptr(), len(x)) == 0
        return own.cpu().numpy(), ref.cpu().numpy()
    return f


@pytest.mark.parametrize("low,high", [(0, 1), (-1022, -1020), (1019, 1021), (-1000, 1000)])
def test_every_reciprocal_is_correctly_rounded(run, low, high):
    rng = np.random.default_rng(low + 2000)
    n = 1 << 22
    x = rng.uniform(1.0, 2.0, n) * rng.choice([-1.0, 1.0], n) * 2.0 ** rng.integers(low, high, n)
    x[:4096] = (1.0 + 2.0 ** -52 * np.arange(4096)) * 2.0 ** low
    x[4096:8192] = (2.0 - 2.0 ** -52 * (2 + np.arange(4096))) * 2.0 ** low      # (not the mantissa of all ones)
    own, ref = run(x)
    assert np.array_equal(own, ref)


def test_the_ends_of_the_range(run):
    """Zeros, infinities and NaNs as a division gives them; subnormals as zeros; below a reciprocal of 2^-1021, 20 bits
    or zero."""
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan])
    own, ref = run(special)
    assert np.array_equal(own, ref, equal_nan=True) and np.array_equal(np.signbit(own[:4]), np.signbit(ref[:4]))
    rng = np.random.default_rng(5)
    tiny = 2.0 ** -1074 * np.concatenate([[1.0], rng.integers(1, 1 << 52, 4096).astype(float)])
    own, _ = run(np.concatenate([tiny, -tiny]))
    assert np.array_equal(own, np.inf * np.repeat([1.0, -1.0], len(tiny)))
    big = np.ldexp(rng.uniform(0.5, 1, 8192), np.repeat([1022, 1023, 1024], [2730, 2731, 2731]))
    own, ref = run(np.concatenate([big, -big]))
    assert np.all((np.abs(own - ref) <= 2.0 ** -19 * np.abs(ref)) | (np.abs(ref) <= 1.0001 * 2.0 ** -1022) & (own == 0.0))
