"""The fixed-point digits of the digit-slice contractions, compiled for the host from the
kernels' own header: each value's digit word is its nearest integer multiple of the line's
unit, halves away from zero, for both signs."""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_18221_gb300", "csrc")

SHIM = r"""
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
using std::min;
#define __device__
#define __forceinline__ inline
template <class A, class B> static inline A bits(B b) { A a; std::memcpy(&a, &b, sizeof(a)); return a; }
static inline int __double2hiint(double x) { return (int)(bits<uint64_t>(x) >> 32); }
static inline int __double2loint(double x) { return (int)(uint32_t)bits<uint64_t>(x); }
static inline double __hiloint2double(int hi, int lo) { return bits<double>(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo); }
static inline double __ll2double_rn(long long v) { return (double)v; }
static inline double __longlong_as_double(long long v) { return bits<double>(v); }
static inline int __clzll(long long v) { return __builtin_clzll((unsigned long long)v); }
#include "fx_digits.cuh"
extern "C" void digits(const double* u, const int* el, long long* x, int n) {
    for (int i = 0; i < n; i++) x[i] = (long long)(gk::digit_word(u[i], el[i], 4u) - gk::DIG_BIAS);
}
"""


@pytest.fixture(scope="module")
def digits(tmp_path_factory):
    import ctypes
    d = tmp_path_factory.mktemp("digits")
    (d / "d.cpp").write_text(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, str(d / "d.cpp"), "-o", str(d / "d.so")],
                   check=True)
    fn = ctypes.CDLL(str(d / "d.so")).digits

    def run(u, el):
        u, el = np.ascontiguousarray(u, np.float64), np.ascontiguousarray(el, np.int32)
        x = np.empty(u.size, np.int64)
        fn(u.ctypes.data_as(ctypes.c_void_p), el.ctypes.data_as(ctypes.c_void_p), x.ctypes.data_as(ctypes.c_void_p), u.size)
        return x
    return run


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("shift", [0, 1, 2, 3, 20, 52, 53, 54, 55, 60, 2000])
def test_nearest_integer(digits, sign, shift):
    """A value of exponent e on a line of exponent EL = e + shift: X = u 2^(1076 - EL), rounded."""
    rng = np.random.default_rng(shift)
    m = rng.integers(2 ** 52, 2 ** 53, 4000, dtype=np.int64)
    m[:4] = [2 ** 52, 2 ** 52 + 1, 2 ** 53 - 1, 2 ** 52 + 2 ** 51]
    k = min(shift, 53)
    half = (m >> k << k) | (1 << max(k - 2, 0))      # about and exactly half a unit, where k >= 2
    m = np.concatenate([m, half, np.bitwise_or(half, 1)])
    e = 30 if shift == 2000 else 1000
    u = sign * np.ldexp(m.astype(np.float64), e - 1075)
    got = digits(u, np.full(u.size, e + shift))
    # exactly: |X| = 2 m / 2^shift, to the nearest, halves up in magnitude
    want = [int(sign) * ((2 * int(v) * 2 + (1 << shift)) >> (shift + 1)) for v in m]
    assert got.tolist() == want


def test_zero_and_subnormal(digits):
    u = np.array([0.0, -0.0, 5e-324, -2e-308])
    assert digits(u, np.array([1023, 1023, 40, 40])).tolist() == [0, 0, 0, 0]
