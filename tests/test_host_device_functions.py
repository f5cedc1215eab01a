"""The kernels' digit splits, level-word conversion and double-word scalars, run on
the CPU: the functions' own source is cut out of the headers and compiled with g++
(no contraction), CUDA's intrinsics given by their definitions, so what is checked is
what the kernels run.  The approximate root and reciprocal instructions are given as
the exact value with a relative error that the caller chooses within the documented
bounds of rsqrt.approx.f32 (2^-22.9) and rcp.approx.f32 (2^-23).
"""
import ctypes
import os
import re
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1708_06290_gb300", "csrc")
f32, LD = np.float32, np.longdouble

PRE = r'''
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __host__
#define __forceinline__ inline
struct uint4 { unsigned x, y, z, w; };
static uint4 make_uint4(unsigned a, unsigned b, unsigned c, unsigned d) { return uint4{a, b, c, d}; }
template <class A, class B> static A bits(B b) { A a; static_assert(sizeof(A) == sizeof(B), ""); std::memcpy(&a, &b, sizeof a); return a; }
static long long __double_as_longlong(double x) { return bits<long long>(x); }
static double __longlong_as_double(long long x) { return bits<double>(x); }
static int __double2hiint(double x) { return (int)(bits<long long>(x) >> 32); }
static unsigned __float_as_uint(float x) { return bits<unsigned>(x); }
static float __uint_as_float(unsigned x) { return bits<float>(x); }
static float __fmul_rn(float a, float b) { return a * b; }
static float __fadd_rn(float a, float b) { return a + b; }
static int __clzll(long long x) { return __builtin_clzll((unsigned long long)x); }
static unsigned __byte_perm(unsigned a, unsigned b, unsigned s) {
  const unsigned long long v = ((unsigned long long)b << 32) | a;
  unsigned r = 0;
  for (int i = 0; i < 4; ++i) r |= (unsigned)((v >> (8 * ((s >> (4 * i)) & 7))) & 0xff) << (8 * i);
  return r;
}
static double seed_err = 0.0;
static float seed_rsqrt(float x) { return (float)((1.0 + seed_err) / std::sqrt((double)x)); }
static float seed_rcp(float x) { return (float)((1.0 + seed_err) / (double)x); }
constexpr int kDigits = 8, kBadExp = 0x40000000;
'''
POST = r'''
extern "C" {
int s_exp(double x) { return scale_exp_hi(abs_hi(x)); }
void s_digits8(double x, int E, int* d) {
  unsigned short u[kDigits];
  digits8(x, E, u);
  for (int l = 0; l < kDigits; ++l) d[l] = (int)__uint_as_float((unsigned)u[l] << 16);
}
int s_exp_f(float x) { return scale_exp_f(x); }
void s_digits7(const float* hi, const float* lo, int E, int* d) {
  float h[8], l[8];
  std::memcpy(h, hi, sizeof h);
  std::memcpy(l, lo, sizeof l);
  uint4 o[7];
  digits7_oct(h, l, digit_scale(E), o);
  for (int k = 0; k < 7; ++k) {
    const unsigned p[4] = {o[k].x, o[k].y, o[k].z, o[k].w};
    for (int e = 0; e < 8; ++e) d[8 * k + e] = (int)__uint_as_float((e & 1 ? p[e / 2] >> 16 : p[e / 2] & 0xffff) << 16);
  }
}
double s_words(int nw, const long long* w, int e) { return nw == 2 ? words_to_double<2>(w, e) : words_to_double<3>(w, e); }
void s_dw(int n, double err, const float* x, float* root, float* rcp) {
  seed_err = err;
  for (int i = 0; i < n; ++i) {
    const dw v{x[2 * i], x[2 * i + 1]}, r = dw_sqrt_fast(v), q = dw_rcp_fast(v);
    root[2 * i] = r.hi; root[2 * i + 1] = r.lo; rcp[2 * i] = q.hi; rcp[2 * i + 1] = q.lo;
  }
}
void s_add_ord(int n, const float* x, const float* y, float* s) {
  for (int i = 0; i < n; ++i) {
    const dw v = dw_add_ord(dw{x[2 * i], x[2 * i + 1]}, dw{y[2 * i], y[2 * i + 1]});
    s[2 * i] = v.hi; s[2 * i + 1] = v.lo;
  }
}
}
'''


def cut(header, name, struct=False):
    """Source of the function (with its template line) or struct `name`."""
    src = open(os.path.join(CSRC, header)).read()
    pat = r"^struct %s \{" if struct else r"^(template <[^\n]*>\n)?(static )?__device__ __forceinline__ [\w ]+\b%s\("
    m = re.search(pat % name, src, re.M)
    assert m, (header, name)
    i = src.index("{", m.end() - 1)
    depth, j = 1, i + 1
    while depth:
        depth += {"{": 1, "}": -1}.get(src[j], 0)
        j += 1
    return src[m.start():j] + (";\n" if struct else "\n")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    body = cut("dfloat.cuh", "dw", struct=True)
    for header, names in (("dfloat.cuh", ["dw_fast", "dw_add"]),
                          ("panel.cuh", ["dw_sqrt_fast", "dw_rcp_fast", "dw_add_ord"]),
                          ("tc_common.cuh", ["abs_hi", "scale_exp_hi", "digits8", "scale_exp_f", "digit_scale",
                                             "digits7_oct"]),
                          ("reduce_tc.cu", ["words_to_double"])):
        body += "".join(cut(header, n) for n in names)
    body, k = re.subn(r'asm\("(rsqrt|rcp)\.approx\.f32 %0, %1;" : "=f"\((\w)\) : "f"\(([\w.]+)\)\);',
                      r"\2 = seed_\1(\3);", body)
    assert k == 2
    d = tmp_path_factory.mktemp("dev")
    (d / "f.cpp").write_text(PRE + body + POST)
    so = str(d / "f.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-w", "-shared", "-fPIC", "-o", so,
                    str(d / "f.cpp")], check=True)
    L = ctypes.CDLL(so)
    L.s_words.restype = ctypes.c_double
    L.s_exp.argtypes = [ctypes.c_double]
    L.s_exp_f.argtypes = [ctypes.c_float]
    return L


def p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


# ---- eight digits of a double ------------------------------------------------
def digits8(lib, x, E):
    d = np.zeros(8, np.int32)
    lib.s_digits8(ctypes.c_double(x), E, p(d))
    return d


def test_digits8_round_to_nearest(lib):
    rng = np.random.default_rng(61)
    # at the top of the row's range the value fits without rounding: no carry past 2^56
    edge = [np.nextafter(1.0, 0), 1.0, np.nextafter(2.0, 0), 0.5, 2.0 ** -3 - 2.0 ** -56, 2.0 ** -4 - 2.0 ** -57, 5e-324, 0.0]
    vals = list(rng.standard_normal(300)) + list(rng.standard_normal(300) * 10.0 ** rng.uniform(-20, 0, 300)) + edge
    for x in vals + [-v for v in edge]:
        E0 = lib.s_exp(x)
        assert abs(x) < 2.0 ** E0 and (x == 0 or E0 == -1022 or abs(x) >= 2.0 ** (E0 - 1))
        for E in (E0, 1, 4):
            if abs(x) >= 2.0 ** E:
                continue
            d = digits8(lib, x, E)
            s = -1 if x < 0 else 1
            assert all(0 <= s * int(v) <= 127 for v in d)
            val = sum(Fraction(int(v)) * Fraction(2) ** (E - 7 * (l + 1)) for l, v in enumerate(d))
            err = abs(val - Fraction(float(x)))
            assert err <= Fraction(2) ** (E - 57)
            if E == E0 and E > -900:
                assert err == 0  # 53 bits under 56
    assert not digits8(lib, np.inf, lib.s_exp(np.inf)).any() and not digits8(lib, 1.0, lib.s_exp(np.nan)).any()


# ---- seven digits of a double-float value ------------------------------------
def digits7(lib, hi, lo, E):
    d = np.zeros((7, 8), np.int32)
    lib.s_digits7(p(f32(hi)), p(f32(lo)), E, p(d))
    return d


def test_digits7_of_pairs(lib):
    rng = np.random.default_rng(62)
    for k in range(300):
        x = rng.standard_normal(8) * 10.0 ** rng.uniform(-8, 0, 8) * 10.0 ** rng.uniform(-6, 6)
        if k < 4:  # the top of the range, both signs
            x[:] = [2 - 2.0 ** -24, -2 + 2.0 ** -24, 2 - 2.0 ** -20, 1.0, -1.0, 1.99609375, 1 + 2.0 ** -23, 0.0]
        hi = f32(x)
        lo = f32(x - hi.astype(float))
        E = lib.s_exp_f(float(np.abs(hi).max()))
        assert np.abs(hi).max() < 2.0 ** E
        d = digits7(lib, hi, lo, E)
        assert np.abs(d[0]).max() <= 128 and np.abs(d[1:]).max() <= 80
        for e in range(8):
            v = Fraction(float(hi[e])) + Fraction(float(lo[e]))
            got = sum(Fraction(int(d[l, e])) * Fraction(2) ** (E - 7 * (l + 1)) for l in range(7))
            assert abs(got - v) <= Fraction(2) ** (E - 50)
    assert not digits7(lib, np.ones(8), np.zeros(8), lib.s_exp_f(np.inf)).any()
    # level sums of one 128-deep window stay exact in FP32: H's digits up to 127 against these
    assert 128 * 127 * (128 + 6 * 80) < 2 ** 24


def test_shifts_of_a_group_share_its_columns():
    """32 real columns: 32 / cs shifts of cs columns, cs = 2m rounded up to a power of two;
    levels of shift l of Z2 P2 at columns 7 cs l + cs lv."""
    for m in range(1, 17):
        cs = 2
        while cs < 2 * m:
            cs *= 2
        S = 32 // cs
        assert S >= 1 and S * cs == 32 and cs >= 2 * m
        seen = {7 * cs * l + cs * lv + c for l in range(S) for lv in range(7) for c in range(cs)}
        assert len(seen) == 7 * 32 and max(seen) < 256


# ---- level words -------------------------------------------------------------
def test_words_to_double_rounds_once(lib):
    rng = np.random.default_rng(63)
    for k in range(4000):
        nw = 2 + k % 2
        w = [int(v) for v in rng.integers(-2 ** 62, 2 ** 62, nw) >> rng.integers(0, 62, nw)]
        e = int(rng.integers(-300, 300))
        if k % 7 == 0:  # a tie, and one unit to either side of it
            w = [int(2 ** 53 + 2 * rng.integers(0, 100) + 1), 0] + [int(rng.integers(-1, 2))] * (nw - 2)
            w[1] = w[1] if nw == 3 else int(rng.integers(-1, 2))
            w[0] <<= 0
        if k % 11 == 0:
            w[0] = 0
        exact = sum(Fraction(v) * Fraction(2) ** (e - 28 * q) for q, v in enumerate(w))
        got = lib.s_words(nw, p(np.array(w, np.int64)), e)
        assert got == exact.numerator / exact.denominator, (w, e)  # Python rounds a quotient to nearest even
    assert lib.s_words(3, p(np.zeros(3, np.int64)), 5) == 0.0


# ---- double-word scalars -----------------------------------------------------
def fma(a, b, c):
    return f32(LD(a) * LD(b) + LD(c))


def fast(a, b):
    s = f32(a + b)
    return s, f32(b - f32(s - a))


@pytest.mark.parametrize("err", [0.0, 1.0, -1.0, 0.7])
def test_root_and_reciprocal_from_the_worst_seeds(lib, err):
    """No less accurate than one correction on IEEE quotient and root, at seeds off by the
    documented bound."""
    rng = np.random.default_rng(64)
    n = 1 << 18
    hi = f32(rng.uniform(1.0, 4.0, n))
    hi, lo = fast(hi, f32(hi.astype(float) * rng.uniform(-2.0 ** -25, 2.0 ** -25, n)))
    X = LD(hi) + LD(lo)
    x = np.ascontiguousarray(np.stack([hi, lo], 1))
    root, rcp = np.zeros_like(x), np.zeros_like(x)
    s = np.sqrt(hi)
    q = f32(f32(1) / hi)
    ieee = (fast(s, f32(f32(fma(-s, s, hi) + lo) / f32(f32(2) * s))),
            fast(q, f32(f32(fma(-q, hi, f32(1)) + fma(-q, lo, f32(0))) / hi)))
    for which, bound, exact in ((0, 2.0 ** -22.9, np.sqrt(X)), (1, 2.0 ** -23, 1 / X)):
        lib.s_dw(n, ctypes.c_double(err * bound), p(x), p(root), p(rcp))
        g = (root, rcp)[which]
        e = np.abs((LD(g[:, 0]) + LD(g[:, 1]) - exact) / exact).astype(float)
        o = np.abs((LD(ieee[which][0]) + LD(ieee[which][1]) - exact) / exact).astype(float)
        assert e.max() <= o.max() and (e ** 2).mean() <= (o ** 2).mean()


def test_ordered_sum(lib):
    rng = np.random.default_rng(65)
    n = 20000
    a = rng.uniform(1, 2, n) * 2.0 ** rng.integers(0, 10, n)
    b = a * rng.uniform(0, 1, n)
    pair = lambda v: np.ascontiguousarray(np.stack([f32(v), f32(v - f32(v).astype(float))], 1))  # noqa: E731
    x, y, s = pair(a), pair(b), np.zeros((n, 2), f32)
    lib.s_add_ord(n, p(x), p(y), p(s))
    ex = LD(x).sum(1) + LD(y).sum(1)
    # roundings of the two low additions: 2^-24 of 2^-23 of the sum, twice
    assert (np.abs((LD(s).sum(1) - ex) / ex) <= 2.0 ** -46).all()
