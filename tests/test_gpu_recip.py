"""FastMath::recip (wt_math_fast.cuh), the reciprocal of the fast policy's cells, against the division."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_1504_00731_gb300 import build

torch = pytest.importorskip("torch")

SRC = """
#include "wt_math_fast.cuh"
__global__ void k(const double* x, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = wt::FastMath::recip(x[i]);
}
extern "C" int run(const double* x, double* y, int n) {
  k<<<(n + 255) / 256, 256>>>(x, y, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def recip(tmp_path_factory):
    d = tmp_path_factory.mktemp("recip")
    (d / "recip.cu").write_text(SRC)
    so = str(d / "librecip.so")
    subprocess.run([build.NVCC, *build.COMMON, "-I", build.CSRC, "-shared", str(d / "recip.cu"), "-o", so], check=True)
    lib = ctypes.CDLL(so)

    def run(x):
        u = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        y = torch.empty_like(u)
        assert lib.run(ctypes.c_void_p(u.data_ptr()), ctypes.c_void_p(y.data_ptr()), u.numel()) == 0
        return y.cpu().numpy()

    return run


@pytest.mark.gpu
def test_recip_within_its_bound(recip):
    """Within 2^-52 of 1 / x over all magnitudes of either sign (the remainder 1 - x y rounded in long double,
    below 2^-63), and the division's own value outside [2^-1000, 2^1000]."""
    rng = np.random.default_rng(1)
    m = np.concatenate([rng.uniform(1, 2, 1 << 20), [1.0, np.nextafter(1, 2), np.nextafter(2, 1), 1.5], 1 + 2.0**-np.arange(1, 53)])
    x = np.ldexp(m, rng.integers(-999, 999, m.size)) * rng.choice([-1.0, 1.0], m.size)
    x = np.concatenate([x, m, np.ldexp(1.0, np.arange(-999, 1000))])
    e = np.abs(1 - x.astype(np.longdouble) * recip(x).astype(np.longdouble))
    assert e.max() <= 2.0**-52
    with np.errstate(all="ignore"):
        z = np.concatenate([np.ldexp(1.3, np.arange(-1074, -1001)), np.ldexp(1.3, np.arange(1001, 1024)),
                            [0.0, -0.0, np.inf, -np.inf, 5e-324, -5e-324, np.finfo(float).max]])
        assert np.array_equal(recip(z), 1 / z)
        assert np.isnan(recip(np.array([np.nan])))[0]
