"""The division-free Sturm count (csrc/sturm64.cuh) against the quotient form in
exact arithmetic, on the host: the header is compiled with the host compiler and
plain definitions of the CUDA names it uses."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1611_09467_gb300", "csrc")

SHIM = r"""
#pragma once
#include <cmath>
#include <cstdint>
#include <cstring>
#include <algorithm>
using std::fma; using std::fmax; using std::max; using std::min;
#define __device__
#define __forceinline__ inline
#define __noinline__
inline int __double2hiint(double x) { int64_t b; std::memcpy(&b, &x, 8); return (int)(b >> 32); }
inline int __double2loint(double x) { int64_t b; std::memcpy(&b, &x, 8); return (int)b; }
inline double __hiloint2double(int h, int l) {
  const int64_t b = (int64_t)(((uint64_t)(uint32_t)h << 32) | (uint32_t)l);
  double x; std::memcpy(&x, &b, 8); return x;
}
inline int __all_sync(unsigned, int p) { return p; }
inline unsigned __ballot_sync(unsigned, int p) { return p ? 1u : 0u; }
inline int __popc(unsigned x) { return __builtin_popcount(x); }
"""


@pytest.fixture(scope="module")
def count(tmp_path_factory):
    d = tmp_path_factory.mktemp("sturm")
    (d / "cuda_runtime.h").write_text(SHIM)
    (d / "t.cpp").write_text('#include "cuda_runtime.h"\n#include "sturm64.cuh"\nextern "C" int count(const double* t2, '
                             "int n2, double x) { return peps::sturm_count_minors(t2, n2, x); }\n")
    so = d / "t.so"
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", str(d), "-I", CSRC,
                    str(d / "t.cpp"), "-o", str(so)], check=True)
    f = ctypes.CDLL(str(so)).count
    f.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_double]

    def call(t2, x):
        a = np.asarray(t2, dtype=np.float64)
        return f(a.ctypes.data, len(a) + 1, x)
    return call


def quotient_count(t2, x):
    """Pivots of T - x in exact arithmetic, a zero one clamped to a tiny negative value."""
    q, n = -Fraction(x), 0
    for i in range(len(t2) + 1):
        if i:
            q = -Fraction(x) - Fraction(t2[i - 1]) / q
        if q == 0:
            q = Fraction(-1, 1 << 2000)
        n += q < 0
    return n


def test_decoupled_blocks_with_a_root_at_the_point(count):
    """A zero minor followed by a zero off-diagonal: eigenvalues -2, -2, -1, 1, 2, 2
    have four at or below 1."""
    assert quotient_count([1, 0, 4, 0, 4], 1) == 4
    assert count([1.0, 0.0, 4.0, 0.0, 4.0], 1.0) == 4


def test_counts_equal_the_quotient_form(count):
    """Random decoupled and coupled matrices whose minors are exact in double
    (dyadic entries, up to 24 rows), counted at points that are roots of
    many of their blocks, and past the row count between two scalings."""
    rng = np.random.default_rng(17)
    vals, points = [0.0, 0.0, 0.25, 1.0], [0.5, 1.0, 0.25, 2.0]
    for _ in range(20000):
        t2 = [float(v) for v in rng.choice(vals, size=rng.integers(1, 24))]
        x = float(rng.choice(points))
        assert count(t2, x) == quotient_count(t2, x), (t2, x)


def test_counts_of_generic_matrices(count):
    """Random matrices without ties against the eigenvalues themselves."""
    rng = np.random.default_rng(18)
    for _ in range(500):
        n = int(rng.integers(2, 72))
        t = rng.uniform(0, 1.99, n - 1) * rng.choice([1.0, 1.0, 1e-9], size=n - 1)
        x = float(rng.uniform(0.01, 3.5))
        ev = np.linalg.eigvalsh(np.diag(t, 1) + np.diag(t, -1))
        if np.abs(ev - x).min() > 1e-9:
            assert count(t * t, x) == int((ev < x).sum())
