"""The integer arithmetic of the rate-of-spread path against IEEE-754.

``csrc/c2f_exact.cuh`` compiles as plain C++: division and square root must return the
correctly rounded binary64 result (numpy's) over their stated range, for any
starting estimate within two units of binary32 (the GPU's approximate
reciprocals are within one).  Arguments sit where the algorithms can go wrong:
significands next to 1 and 2 and with few bits set, exponents at the ends of
the range, quotients and roots next to a rounding boundary.
"""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1905_09317_gb300", "csrc")
SOURCE = r"""
static float g_scale = 1.0f;
#define C2F_HOST_ESTIMATE_SCALE g_scale
#include "c2f_exact.cuh"
extern "C" void steps(const double *r, long n, int log, double *q, double *e, unsigned char *ok) {
  for (long i = 0; i < n; ++i) {
    bool exact;
    q[i] = log ? c2f::log_steps(r[i], &exact) : c2f::exp_steps(r[i], &exact);
    ok[i] = exact;
    if (log)
      e[i] = std::fma(std::fma(std::fma(std::fma(-1.0 / 6, r[i], 1.0 / 5), r[i], -0.25), r[i], 1.0 / 3), r[i], -0.5);
    else
      e[i] = std::fma(std::fma(std::fma(1.0 / 120, r[i], 1.0 / 24), r[i], 1.0 / 6), r[i], 0.5);
  }
}
extern "C" void products(const double *a, const double *b, long n, double *p, double *d, unsigned char *ok) {
  for (long i = 0; i < n; ++i) {
    p[i] = c2f::mul_mid(a[i], b[i]);
    ok[i] = c2f::mid_range(c2f::bits_of(a[i])) && c2f::mid_range(c2f::bits_of(b[i]));
    d[i] = c2f::below_one(c2f::bits_of(a[i])) ? c2f::one_minus(a[i]) : 1.0 - a[i];
  }
}
extern "C" void run(const double *a, const double *b, long n, int ulps, double *q, double *s, unsigned char *ok) {
  g_scale = 1.0f + ulps * 0x1p-23f;
  for (long i = 0; i < n; ++i) {
    q[i] = c2f::div_mid(a[i], b[i]);
    s[i] = c2f::sqrt_mid(a[i]);
    ok[i] = c2f::mid_range(c2f::bits_of(a[i])) && c2f::mid_range(c2f::bits_of(b[i]));
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("exact")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC, str(d / "t.cpp"),
                    "-o", str(d / "t.so")], check=True)
    return C.CDLL(str(d / "t.so"))


def _values(rng, n, span):
    m = rng.integers(0, 1 << 52, n, dtype=np.uint64)
    kind = rng.integers(0, 6, n)
    few = rng.integers(0, 256, n, dtype=np.uint64)
    m = np.where(kind == 0, few, m)                                    # next to 1
    m = np.where(kind == 1, np.uint64((1 << 52) - 1) - few, m)         # next to 2
    m = np.where(kind == 2, m & ~np.uint64((1 << 32) - 1), m)          # few bits
    m = np.where(kind == 3, few << np.uint64(44), m)
    e = (1023 + rng.integers(-span, span + 1, n)).astype(np.uint64)
    return ((e << np.uint64(52)) | m).view(np.float64)


@pytest.mark.parametrize("ulps", [-2, 0, 2])
@pytest.mark.parametrize("span", [1, 499])
def test_division_and_root_are_correctly_rounded(lib, ulps, span):
    rng = np.random.default_rng(1000 * span + ulps + 2)
    n = 400_000
    a, b = _values(rng, n, span), _values(rng, n, span)
    half = n // 2   # quotients and roots next to a boundary: products and squares, one unit either side
    step = rng.integers(-1, 2, half)
    a[:half] = (np.sqrt(np.abs(a[:half])) * np.sqrt(np.abs(b[:half]))) if span == 499 else a[:half] * b[:half]
    a[:half // 2] = b[:half // 2] * b[:half // 2] if span == 1 else a[:half // 2]
    a[:half] = (a[:half].view(np.int64) + step).view(np.float64)
    q, s, ok = np.empty(n), np.empty(n), np.empty(n, dtype=np.uint8)
    lib.run(a.ctypes.data_as(C.c_void_p), b.ctypes.data_as(C.c_void_p), C.c_long(n), C.c_int(ulps),
            q.ctypes.data_as(C.c_void_p), s.ctypes.data_as(C.c_void_p), ok.ctypes.data_as(C.c_void_p))
    use = ok.astype(bool)
    assert use.mean() > 0.99
    assert np.array_equal(q[use], (a / b)[use])
    assert np.array_equal(s[use], np.sqrt(a)[use])


def test_exp_and_log_steps_equal_fused_multiply_adds(lib):
    """Where they say so, the integer Horner steps are the FP64 ones: c + q r rounded at every step."""
    rng = np.random.default_rng(3)
    n = 200_000
    r = rng.uniform(-0.00542, 0.00542, n)
    r[: n // 4] = np.ldexp(r[: n // 4], -rng.integers(0, 12, n // 4))
    r[:7] = [0.0, -0.0, 2.0 ** -18, -2.0 ** -18, 2.0 ** -8, -2.0 ** -8, 2.0 ** -40]
    q, e, ok = np.empty(n), np.empty(n), np.empty(n, dtype=np.uint8)
    for which in (0, 1):   # exp, log
        lib.steps(r.ctypes.data_as(C.c_void_p), C.c_long(n), C.c_int(which), q.ctypes.data_as(C.c_void_p),
                  e.ctypes.data_as(C.c_void_p), ok.ctypes.data_as(C.c_void_p))
        use = ok.astype(bool)
        big = np.abs(r) > 2.0 ** -17.9
        assert use[big & ((r > 0) | (which == 0))].mean() > 0.999
        assert np.array_equal(q[use], e[use])


@pytest.mark.parametrize("span", [1, 499])
def test_product_and_one_minus_are_correctly_rounded(lib, span):
    rng = np.random.default_rng(span)
    n = 400_000
    a, b = _values(rng, n, span), _values(rng, n, span)
    a[: n // 2] = np.where(rng.random(n // 2) < 0.5, 1.0 - np.ldexp(rng.random(n // 2), -rng.integers(0, 53, n // 2)),
                           np.ldexp(1.0 + np.round(rng.random(n // 2) * 8) / 8, -rng.integers(1, 60, n // 2)))
    p, d, ok = np.empty(n), np.empty(n), np.empty(n, dtype=np.uint8)
    lib.products(a.ctypes.data_as(C.c_void_p), b.ctypes.data_as(C.c_void_p), C.c_long(n), p.ctypes.data_as(C.c_void_p),
                 d.ctypes.data_as(C.c_void_p), ok.ctypes.data_as(C.c_void_p))
    use = ok.astype(bool)
    assert use.mean() > 0.9
    assert np.array_equal(p[use], (a * b)[use])
    assert np.array_equal(d, 1.0 - a)
