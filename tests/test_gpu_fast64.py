"""quick_rcp and quick_rsqrt (csrc/fast64.cuh) over the whole exponent range.

Bounds, in units in the last place of the exact value.  With a start value good
to 2^-19 and e its residual: reciprocal, cut term e^3 <= 2^-57 and the final
rounding, 0.6; reciprocal square root, the rounding of x y moves e by 2^-53 and
the result by 2^-54 of itself, at most half a unit, and the final rounding, 1.1.
The library functions that take the ends of the range have 0.5 and 1.  Asserted:
1 and 1.5."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SRC = r"""
#include "fast64.cuh"
__global__ void k(const double* x, double* r, double* s, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    r[i] = peps::quick_rcp(x[i]);
    s[i] = peps::quick_rsqrt(x[i]);
  }
}
extern "C" int run(const double* x, double* r, double* s, int n) {
  k<<<(n + 255) / 256, 256>>>(x, r, s, n);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_1611_09467_gb300 import build
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    d = tmp_path_factory.mktemp("fast64")
    (d / "t.cu").write_text(SRC)
    so = d / "t.so"
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-I", build.CSRC, str(d / "t.cu"), "-o", str(so)],
                   check=True, capture_output=True)
    f = ctypes.CDLL(os.fspath(so)).run
    f.argtypes = [ctypes.c_void_p] * 3 + [ctypes.c_int]

    def call(x):
        xd = torch.from_numpy(x).cuda()
        r, s = torch.empty_like(xd), torch.empty_like(xd)
        torch.cuda.synchronize()
        assert f(xd.data_ptr(), r.data_ptr(), s.data_ptr(), len(x)) == 0
        return r.cpu().numpy(), s.cpu().numpy()
    return call


def ulps(got, exact):
    """Distance in units in the last place of the double nearest to `exact` (long double)."""
    near = exact.astype(np.float64)
    assert np.isfinite(near).all() and np.isfinite(got).all()
    return float((np.abs(got.astype(np.longdouble) - exact) / np.spacing(np.abs(near)).astype(np.longdouble)).max())


@pytest.mark.parametrize("lo,hi", [(-1074, -1021), (-1021, -702), (-702, -698), (-698, 698), (698, 702), (702, 1024), (-2, 3)])
def test_errors_by_exponent(run, lo, hi):
    """Random mantissas at exponents lo <= e < hi: subnormal numbers, both sides of
    the lines at 2^-700 and 2^700, the middle and the top."""
    assert np.finfo(np.longdouble).nmant >= 63
    rng = np.random.default_rng(abs(lo) * 3000 + abs(hi))
    n = 400000
    x = np.ldexp(1.0 + rng.random(n), rng.integers(lo, hi, n))
    x[: n // 8] = np.ldexp(1.0, rng.integers(lo, hi, n // 8))
    x[n // 8: n // 4] = np.nextafter(x[n // 8: n // 4], np.inf)
    x = x[np.isfinite(x) & (x > 0)]
    r, s = run(x)
    X = x.astype(np.longdouble)
    ok = x > 2.0 ** -1022          # below, the reciprocal overflows
    e_r, e_s = ulps(r[ok], 1 / X[ok]) if ok.any() else 0.0, ulps(s, 1 / np.sqrt(X))
    rn, _ = run(-x)
    print(f"2^[{lo}, {hi}): reciprocal {e_r:.3f} ulp, inverse square root {e_s:.3f} ulp")
    assert np.array_equal(rn, -r)
    assert e_r <= 1.0 and e_s <= 1.5


def test_special_values(run):
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, -1.0, -2.0 ** -800, 2.0 ** -1074])
    r, s = run(x)
    with np.errstate(all="ignore"):
        assert np.array_equal(r, 1.0 / x, equal_nan=True) and np.array_equal(np.signbit(r[:4]), [False, True, False, True])
    assert np.array_equal(s, [np.inf, -np.inf, 0.0, np.nan, np.nan, np.nan, np.nan, 2.0 ** 537], equal_nan=True)
