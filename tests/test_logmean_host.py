"""The log means' polynomials and the FP64 form's two-part series on the host: the
coefficients read from the headers against artanh with 40 digits, and the
header's own functions, compiled as plain C++ with the few device intrinsics
they use written out, so that their rounding can be compared with exact
arithmetic.
"""
import ctypes
import os
import re
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2604_02125_gb300", "csrc", "crkfr_physics.cuh")

SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>
template <class T, class S> static T bits_as(S s) { T t; std::memcpy(&t, &s, sizeof(t)); return t; }
#define __host__
#define __device__
#define __noinline__
#define __forceinline__ inline
#define __double2hiint(x) ((int)(bits_as<uint64_t>((double)(x)) >> 32))
#define __double2loint(x) ((int)(uint32_t)bits_as<uint64_t>((double)(x)))
#define __hiloint2double(h, l) bits_as<double>(((uint64_t)(uint32_t)(h) << 32) | (uint32_t)(l))
#define __longlong_as_double(i) bits_as<double>((int64_t)(i))
#define __float_as_int(f) bits_as<int32_t>((float)(f))
#define __float_as_uint(f) bits_as<uint32_t>((float)(f))
#define __uint_as_float(u) bits_as<float>((uint32_t)(u))
#define __fma_rn std::fma
#define __fmaf_rn std::fmaf
#define __fmul_rn(a, b) ((float)(a) * (float)(b))
#define __fadd_rn(a, b) ((float)(a) + (float)(b))
#define __dmul_rn(a, b) ((double)(a) * (double)(b))
#define __funnelshift_l(lo, hi, s) ((uint32_t)(((((uint64_t)(hi)) << 32 | (uint32_t)(lo)) << (s)) >> 32))
#define __funnelshift_r(lo, hi, s) ((uint32_t)((((uint64_t)(hi)) << 32 | (uint32_t)(lo)) >> (s)))
// the reciprocal units: 23 bits in FP32, 20 bits in FP64; sign and magnitude of
// the error from the bits of x; out-of-range operands as documented for .ftz
static float unit_rcp(const char*, float x) { return (1.0f / x) * (1.0f + ((int)(bits_as<uint32_t>(x) % 3) - 1) * 1.1920929e-7f); }
static double unit_rcp(const char*, double x) {
  if (std::fabs(x) < 2.2250738585072014e-308) return std::copysign(INFINITY, x);
  if (std::fabs(x) > 4.4942328371557898e307) return std::copysign(0.0, x);
  return (1.0 / x) * (1.0 + ((int)(bits_as<uint64_t>(x) % 2001) - 1000) * 9.5e-10);
}
#define asm(...) r = unit_rcp(#__VA_ARGS__, x)
#include HEADER
extern "C" void units(int n, const double* d, const double* s, double* iF4, double* F) {
  for (int k = 0; k < n; ++k) {
    // 1/(4 F) and F as logmean_pair takes them
    double rs2, H1, T2;
    crk::logmean_pair(s[k] + d[k], s[k] - d[k], s[k] + d[k], s[k] - d[k], H1, T2, rs2);
    iF4[k] = H1 / (2.0 * s[k]);
    F[k] = T2 / rs2;
  }
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("logmean")
    src, lib = str(d / "shim.cpp"), str(d / "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I/usr/local/cuda/include",
                    "-DHEADER=\"%s\"" % HEADER, src, "-o", lib], check=True)
    return ctypes.CDLL(lib)


def _call(fn, *arrays):
    out = [np.empty_like(arrays[0]) for _ in range(2)]
    fn(len(arrays[0]), *[a.ctypes.data_as(ctypes.c_void_p) for a in list(arrays) + out])
    return out


def _series(u):
    """(1/F, F) of u = (d/s)^2 <= 2^-11: the sixth power leaves less than 2^-66."""
    inv = [Fraction(1), Fraction(-1, 3), Fraction(-4, 45), Fraction(-44, 945), Fraction(-428, 14175),
           Fraction(-10196, 467775)]
    return sum(c * u ** k for k, c in enumerate(inv)), sum(u ** k / (2 * k + 1) for k in range(7))


@pytest.mark.parametrize("fmax", [2.0 ** -8, 2.0 ** -11, 2.0 ** -15])
def test_two_part_series_is_rounded_once(host, fmax):
    """u < 2^-16: the part beyond 1 is at most u/3 and off by 2^-45 of itself, below
    2^-62; its low words add a few 2^-60.  So 1/(4F) in [1/8, 1/4] lies within half a
    step of 2^-55, and F in [1, 2) within half a step of 2^-52, of the exact value and
    2^-59 of the unit more.  s is a power of two, so the products with s and 1/(2s)
    that the call makes of them are exact."""
    rng = np.random.default_rng(7)
    s = 2.0 ** rng.integers(-3, 4, 6000).astype(np.float64)
    d = np.round(s * fmax * rng.uniform(-1.0, 1.0, 6000) * 2.0 ** 49) / 2.0 ** 49   # s +- d exact
    assert np.all((s + d) - s == d) and np.all(s - (s - d) == d)
    iF4, F = _call(host.units, d, s)
    for k in range(len(s)):
        u = (Fraction(d[k]) / Fraction(s[k])) ** 2
        e_inv, e_F = _series(u)
        assert abs(4 * Fraction(iF4[k]) - e_inv) <= Fraction(1, 2 ** 54) + Fraction(1, 2 ** 59), (k, float(u))
        assert abs(Fraction(F[k]) - e_F) <= Fraction(1, 2 ** 53) + Fraction(1, 2 ** 59), (k, float(u))


@pytest.mark.parametrize("e", [-1021, -1017, -1000, -897, -896, -895, -894, 1020, 1021, 1022])
def test_sums_at_the_ends_of_the_range(host, e):
    """Equal and nearly equal values whose sum 2^(e+1) lies at either end of the FP64
    range, where the exponent field of a zero difference is not small beside the
    sum's and the reciprocal unit takes operands or results for zero.  Two roundings, and
    the subnormal result's own beyond 2^1022."""
    s = np.full(3, 2.0 ** e)
    d = s * np.array([0.0, 2.0 ** -20, -2.0 ** -12]) if e > -900 else np.zeros(3)
    iF4, F = _call(host.units, d, s)
    for k in range(3):
        e_inv, e_F = _series((Fraction(d[k]) / Fraction(s[k])) ** 2)
        assert abs(4 * Fraction(iF4[k]) - e_inv) <= Fraction(1, 2 ** 52), (e, k, iF4[k])
        assert abs(Fraction(F[k]) - e_F) <= Fraction(1, 2 ** 50), (e, k, F[k])


def _coefficients(path, head):
    """c0, c1, ... of the nested polynomial c0 + u (c1 + u (c2 + ...)) in the function that starts with head,
    rounded as its suffix says."""
    with open(path) as f:
        body = f.read().split(head, 1)[1].split("}", 1)[0]
    expr = " ".join(re.findall(r"(?:c[0-3]\([^)]*\)|return [^;]*;)", body))
    vals = []
    for factor, num, single in re.findall(r"(-?0\.25f \* )?(-?\d+\.\d+)(f?)", expr):
        v = float(np.float32(num)) if single else float(num)
        vals.append(float(np.float32(-0.25) * np.float32(v)) if factor else v)
    return vals if "c3(" not in expr else vals[::-1]


@pytest.mark.parametrize("head,umax,kind,bound", [
    ("double series_F(double u) {", 1 / 16, "F", 1.8e-17), ("double series_invF(double u) {", 1 / 16, "invF", 3.1e-18),
    ("float series_F(float u) {", 0.05, "F", 1.2e-8), ("float series_invF(float u) {", 0.05, "invF", 3.7e-9),
    ("float series_invF4(float u) {", 0.05, "invF4", 3.7e-9 / 4),
    ("f2 series_F(f2 u) {", 0.05, "F", 1.2e-8), ("f2 series_invF4(f2 u) {", 0.05, "invF4", 3.7e-9 / 4)])
def test_polynomial_errors(head, umax, kind, bound):
    """The errors stated beside the polynomials, in exact arithmetic."""
    mp = pytest.importorskip("mpmath")
    path = HEADER.replace("physics", "f2") if "f2 " in head else HEADER
    with mp.workdps(40):
        c = [mp.mpf(x) for x in _coefficients(path, head)]
        assert len(c) == (9 if umax > 0.06 else 4), c
        worst = mp.mpf(0)
        for k in range(1, 801):
            u = mp.mpf(umax) * (1 - mp.cos(mp.pi * k / 800)) / 2
            F = mp.atanh(mp.sqrt(u)) / mp.sqrt(u)
            exact = {"F": F, "invF": 1 / F, "invF4": 1 / (4 * F)}[kind]
            worst = max(worst, abs(mp.polyval(c[::-1], u) - exact))
        assert bound / 2 < worst < bound, worst
