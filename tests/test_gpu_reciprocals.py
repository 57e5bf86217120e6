"""The device's reciprocal and reciprocal square root (common.cuh) against correctly rounded values, over their
exponent range and beyond both of its ends."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1710_03757_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "common.cuh"
__global__ void k(const double* x, double* r, double* y, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  r[i] = mctrg::inv(x[i]);
  y[i] = mctrg::inv_sqrt(fabs(x[i]));
}
extern "C" int both(const double* x, double* r, double* y, int n) {
  k<<<(n + 255) / 256, 256>>>(x, r, y, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def both(tmp_path_factory):
    d = tmp_path_factory.mktemp("recip")
    (d / "k.cu").write_text(SOURCE)
    lib = str(d / "k.so")
    subprocess.run([build.nvcc()] + build.ARCH + ["-std=c++17", "-O3", "-shared", "-Xcompiler", "-fPIC", "-cudart", "static",
                    "-I" + build.CSRC, "-I" + os.path.join(build.ROOT, "include"), str(d / "k.cu"), "-o", lib], check=True)
    return ctypes.CDLL(lib).both


def _errors(both, x):
    """Relative errors of 1/x and 1/sqrt|x|, from exact residuals (1/x (1 + e) x - 1 = e)."""
    torch = pytest.importorskip("torch")
    xd = torch.tensor(x, device="cuda")
    r, y = torch.zeros_like(xd), torch.zeros_like(xd)
    assert both(ctypes.c_void_p(xd.data_ptr()), ctypes.c_void_p(r.data_ptr()), ctypes.c_void_p(y.data_ptr()), x.size) == 0
    # scaled by powers of two (exactly) so that nothing leaves the range
    m, e = np.frexp(x)
    half = e // 2
    t = np.ldexp(np.abs(m), e - 2 * half)                  # |x| = t 4^half
    rs, ys = np.ldexp(r.cpu().numpy(), e), np.ldexp(y.cpu().numpy(), half)
    if np.finfo(np.longdouble).nmant >= 112:               # quadruple: the residuals to 2^-110
        L = np.longdouble
        er = L(rs) * L(m) - 1
        ey = (L(ys) * L(ys) * L(t) - 1) / 2
        return np.abs(er).astype(float), np.abs(ey).astype(float)
    from fractions import Fraction as F
    er = [abs(float(F(float(a)) * F(float(b)) - 1)) for a, b in zip(rs, m)]
    ey = [abs(float((F(float(a)) ** 2 * F(float(b)) - 1) / 2)) for a, b in zip(ys, t)]
    return np.array(er), np.array(ey)


def _values(exponents, rng, per):
    m = np.concatenate([rng.uniform(1.0, 2.0, per), 1.0 + rng.integers(0, 64, per) * 2.0 ** -52,
                        2.0 - rng.integers(1, 64, per) * 2.0 ** -52])
    return np.ldexp(m, rng.choice(exponents, m.size)) * rng.choice([-1.0, 1.0], m.size)


def test_inside_the_range(both):
    x = _values(np.arange(-999, 1000), np.random.default_rng(1), 200000)
    er, ey = _errors(both, x)
    print("1/x: %.3f 2^-53, 1/sqrt: %.3f 2^-53" % (er.max() * 2.0 ** 53, ey.max() * 2.0 ** 53))
    assert er.max() <= 1.07 * 2.0 ** -53
    assert ey.max() <= 1.67 * 2.0 ** -53


def test_beyond_and_at_its_ends(both):
    # the functions take over: correctly rounded quotients, and roots within an ulp
    for ends in (np.arange(-1021, -1001), np.arange(1001, 1021), np.arange(-1004, -996), np.arange(996, 1004)):
        er, ey = _errors(both, _values(ends, np.random.default_rng(2), 2000))
        assert er.max() <= 1.07 * 2.0 ** -53 and ey.max() <= 2.0 ** -52
