"""The device functions that replace FP64 operations by work on bit fields,
compiled from their own source text for the CPU (the CUDA intrinsics they use
have one meaning each) and compared with what they stand for: quotients by a
divisor known ahead with IEEE division, the scaled FP32 residual with the FP64
product narrowed once, 1/s of a power of two with the division, and the rounding
of the learned features with the divided-out quotient."""
import ctypes
import os
import re
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2502_05279_gb300", "csrc")

SHIM = r"""
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __forceinline__ inline
#define __noinline__
template <class A, class B> static A as(B b) { A a; std::memcpy(&a, &b, sizeof a); return a; }
static int __double2hiint(double d) { return (int)(as<uint64_t>(d) >> 32); }
static int __double2loint(double d) { return (int)(uint32_t)as<uint64_t>(d); }
static double __hiloint2double(int h, int l) { return as<double>(((uint64_t)(uint32_t)h << 32) | (uint32_t)l); }
static float __uint_as_float(unsigned u) { return as<float>(u); }
static unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
  return (unsigned)((((uint64_t)hi << 32) | lo) << s >> 32);
}
static double __fma_rn(double a, double b, double c) { return std::fma(a, b, c); }
static float __double2float_rn(double d) { return (float)d; }
static double rmul(double a, double b) { return a * b; }
static double rdiv(double a, double b) { return a / b; }
"""

LOOPS = r"""
extern "C" {
void quot_many(long n, const double* s, const double* m, double* out) {
  for (long k = 0; k < n; ++k) {
    double yl;
    const double y = quot_recip(m[k], &yl);
    out[k] = quot(s[k], m[k], y, yl);
  }
}
void narrow_many(long n, const double* r, double scale, float* out) {
  const double inv = pow2_inverse(scale);
  const int bias = narrow_bias(inv);
  for (long k = 0; k < n; ++k) out[k] = narrow_scaled(r[k], inv, bias);
}
void pow2_many(long n, const double* s, double* out) { for (long k = 0; k < n; ++k) out[k] = pow2_inverse(s[k]); }
void feature_many(long n, const double* q, const double* s, const double* o, float* out) {
  for (long k = 0; k < n; ++k) out[k] = feature_round(q[k], s[k], o[k]);
}
}
"""

FUNCTIONS = {"common.cuh": ["quot_slow", "quot", "quot_recip"],
             "cycle_device.cuh": ["narrow_scaled_slow", "pow2_inverse", "narrow_bias", "narrow_scaled"],
             "learned_device.cuh": ["feature_slow", "feature_round"]}


def source_of(text, name):
    m = re.search(rf"^(?:static )?__device__ [^\n;]*\b{name}\([^;{{]*\) \{{", text, re.M)
    end = re.search(r"\}$" if "\n" not in text[m.start():text.index("}", m.end())] else r"^\}", text[m.end():], re.M)
    return text[m.start():m.end() + end.end()]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    src = SHIM + "constexpr int NARROW_NEVER = -65536;\n"
    for name, functions in FUNCTIONS.items():
        text = open(os.path.join(CSRC, name)).read()
        src += "\n".join(source_of(text, f) for f in functions) + "\n"
        if name == "cycle_device.cuh":
            assert "constexpr int NARROW_NEVER = -65536;" in text
    d = tmp_path_factory.mktemp("bits")
    (d / "bits.cc").write_text(src + LOOPS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-fPIC", "-shared", "-o", str(d / "bits.so"),
                    str(d / "bits.cc")], check=True)
    return ctypes.CDLL(str(d / "bits.so"))


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def same(a, b):
    """The same bits, any NaN for any other."""
    u = np.uint64 if a.dtype == np.float64 else np.uint32
    return ((a.view(u) == b.view(u)) | (np.isnan(a) & np.isnan(b))).all()


def doubles(rng, n, lo, hi):
    """Random mantissas (a quarter with all ones or all zeros but the last bits) at biased exponents lo .. hi."""
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    few = rng.integers(0, 8, n, dtype=np.uint64)
    kind = rng.integers(0, 8, n)
    m = np.where(kind == 0, few, np.where(kind == 1, np.uint64((1 << 52) - 1) - few, m))
    e = rng.integers(lo, hi + 1, n).astype(np.uint64)
    return ((rng.integers(0, 2, n).astype(np.uint64) << np.uint64(63)) | (e << np.uint64(52)) | m).view(np.float64)


SPECIAL = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.0 ** -1022, -2.0 ** -1030, 2.0 ** 1023,
                    np.finfo(np.float64).max, 1.0, -1.0] + [2.0 ** k for k in (-201, -200, -199, 199, 200, 201, -624,
                                                                             -623, -622, 622, 623, 624)])


def test_quotients_are_divisions(lib):
    rng = np.random.default_rng(3)
    s = [doubles(rng, 400_000, 1013, 1033), doubles(rng, 400_000, 0, 2047), doubles(rng, 200_000, 395, 405),
         doubles(rng, 200_000, 1640, 1652)]
    m = [doubles(rng, 400_000, 1013, 1033), doubles(rng, 400_000, 0, 2047), doubles(rng, 200_000, 818, 1228),
         doubles(rng, 200_000, 818, 1228)]
    # numerators whose quotient lies next to a double or next to the middle of two
    d = doubles(rng, 400_000, 820, 1226)
    q = doubles(rng, 400_000, 1000, 1040)
    near = q * d
    for k in (0, 1, -1, 2, -2):
        s.append((near.view(np.int64) + k).view(np.float64))
        m.append(d)
    half = (q.view(np.int64) & ~np.int64((1 << 27) - 1)).view(np.float64)      # 26-bit q: (q + ulp/2) d is exact in parts
    mid = half * d + np.ldexp(np.spacing(half), -1) * d
    for k in (0, 1, -1):
        s.append((mid.view(np.int64) + k).view(np.float64))
        m.append(d)
    a, b = np.meshgrid(SPECIAL, SPECIAL)
    s.append(a.ravel())
    m.append(b.ravel())
    s, m = np.ascontiguousarray(np.concatenate(s)), np.ascontiguousarray(np.concatenate(m))
    got = np.empty_like(s)
    lib.quot_many(ctypes.c_long(s.size), ptr(s), ptr(m), ptr(got))
    with np.errstate(all="ignore"):
        assert same(got, s / m)


@pytest.mark.parametrize("k", [-1022, -1000, -897, -896, -300, -20, 0, 5, 300, 896, 897, 1023])
def test_narrowed_residual(lib, k):
    rng = np.random.default_rng(k + 2000)
    r = np.concatenate([doubles(rng, 200_000, max(0, 1023 + k - 160), min(2047, max(0, 1023 + k + 160))),
                        doubles(rng, 50_000, 0, 2047), SPECIAL])
    tie = (r.view(np.uint64) & ~np.uint64((1 << 29) - 1)) | np.uint64(1 << 28)    # exact ties, and one bit beside
    r = np.concatenate([r, tie.view(np.float64), (tie + np.uint64(1)).view(np.float64), (tie - np.uint64(1)).view(np.float64)])
    scale = 2.0 ** k
    got = np.empty(r.size, np.float32)
    lib.narrow_many(ctypes.c_long(r.size), ptr(r), ctypes.c_double(scale), ptr(got))
    with np.errstate(all="ignore"):
        assert same(got, (r * (np.float64(1.0) / scale)).astype(np.float32))


def test_inverse_of_a_power_of_two(lib):
    s = np.concatenate([2.0 ** np.arange(-1074, 1024, dtype=np.float64), SPECIAL, [3.0, 0.1, -2.0]])
    got = np.empty_like(s)
    lib.pow2_many(ctypes.c_long(s.size), ptr(s), ptr(got))
    with np.errstate(all="ignore"):
        assert same(got, 1.0 / s)


def test_feature_rounding(lib):
    """q within 2^-37 of s / o (relative) rounds as the quotient itself."""
    rng = np.random.default_rng(9)
    s, o = doubles(rng, 600_000, 900, 1146), doubles(rng, 600_000, 1000, 1046)
    # quotients next to a float or to the middle of two floats
    f = (s.view(np.uint64) & ~np.uint64((1 << 28) - 1)).view(np.float64)
    s = np.concatenate([s, f * o, f * o, SPECIAL])
    o = np.concatenate([o, o, np.nextafter(o, 0), np.full(SPECIAL.size, 3.0)])
    with np.errstate(all="ignore"):
        want = (s / o).astype(np.float32)
        for rel in (0.0, 2.0 ** -37, -2.0 ** -37):
            q = np.ascontiguousarray((s / o) * (1.0 + rel))
            got = np.empty(s.size, np.float32)
            lib.feature_many(ctypes.c_long(s.size), ptr(q), ptr(s), ptr(o), ptr(got))
            assert same(got, want)
