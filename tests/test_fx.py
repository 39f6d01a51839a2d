"""The fixed-point arithmetic of the FP64 link tables (csrc/fx.cuh), compiled for the
host and compared with extended-precision references: the fraction of a turn of an
angle, its sine and cosine, and the conversions between doubles and scaled integers.
Bounds from the header: a fraction is cut at 2^-64 of a turn (two units allowed: the
truncation and the 96-bit 1 / 2 pi), sine and cosine to 2^-60, conversions to half a unit.
"""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2508_16298_gb300", "csrc")
NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"

SRC = r"""
#include "fx_gauss.cuh"
using namespace hqmc;
extern "C" {
void turns(const double* th, long long* o, int n) { for (int i = 0; i < n; ++i) o[i] = fx_turns(th[i]); }
void cossin(const long long* f, long long* o, int n) {
  longlong2 tab[256];
  for (int k = 0; k < 256; ++k) tab[k] = fx_table_angle(k, kFxEighth);
  for (int i = 0; i < n; ++i) { const longlong2 r = fx_cossin(f[i], tab); o[2 * i] = r.x; o[2 * i + 1] = r.y; }
}
void gauss(const long long* a, const long long* b, double* o, int n) {
  longlong2 tab[512];
  for (int k = 0; k < 256; ++k) tab[k] = fx_table_angle(k, kFxEighth);
  fx_log_table(tab + 256);
  for (int i = 0; i < n; ++i) { const double2 r = fx_gauss(a[i], b[i], tab); o[2 * i] = r.x; o[2 * i + 1] = r.y; }
}
void to_double(const long long* v, int e, double* o, int n) { for (int i = 0; i < n; ++i) o[i] = fx_to_double_normal(v[i], e); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("fx")
    src, so = str(d / "fx.cu"), str(d / "fx.so")
    open(src, "w").write(SRC)
    subprocess.check_call([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                           "-I" + CSRC, src, "-o", so])
    return ctypes.CDLL(so)


def ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


# pi to 60 digits
PI = Fraction(3141592653589793238462643383279502884197169399375105820974944, 10 ** 60)


def angles():
    g = np.random.default_rng(11)
    special = [0.0, -0.0, np.pi, -np.pi, np.pi / 2, np.pi / 256, 3 * np.pi / 256, 5e-324, 2.0 ** 27, -(2.0 ** 27) + 1e-8]
    return np.concatenate([g.uniform(-np.pi, np.pi, 300), g.uniform(-40, 40, 300), g.uniform(-2e8, 2e8, 100),
                           10.0 ** g.uniform(-25, 0, 100), special])


def test_turns(lib):
    th = angles()
    f = np.empty(len(th), np.int64)
    lib.turns(ptr(th), ptr(f), len(th))
    for t, v in zip(th, f):
        x = Fraction(float(t)) / (2 * PI) - Fraction(int(v), 2 ** 64)
        x -= round(x)
        assert abs(x) * 2 ** 64 <= 2, (t, float(x * 2 ** 64))


def test_sine_and_cosine(lib):
    g = np.random.default_rng(12)
    k = np.arange(-256, 256, dtype=np.int64) << 55  # table angles and the midpoints between them
    f = np.concatenate([k, k + 1, k - 1, g.integers(-2 ** 63, 2 ** 63, 500)])
    o = np.empty((len(f), 2), np.int64)
    lib.cossin(ptr(f), ptr(o), len(f))

    def cos_sin(x):  # x in turns: Taylor series in exact rationals (|angle| <= pi, 40 terms: below 1e-28)
        a = (2 * PI * x).limit_denominator(10 ** 40)
        c = s = Fraction(0)
        term = Fraction(1)
        for n in range(40):
            if n % 2 == 0:
                c += term if n % 4 == 0 else -term
            else:
                s += term if n % 4 == 1 else -term
            term = (term * a / (n + 1)).limit_denominator(10 ** 40)
        return c, s

    for v, (c, s) in zip(f[::3], o[::3]):
        rc, rs = cos_sin(Fraction(int(v), 2 ** 64))
        assert abs(Fraction(int(c), 2 ** 62) - rc) < Fraction(1, 2 ** 60), int(v)
        assert abs(Fraction(int(s), 2 ** 62) - rs) < Fraction(1, 2 ** 60), int(v)


def test_to_double_rounds_to_nearest_even(lib):
    g = np.random.default_rng(13)
    v = g.integers(-2 ** 62, 2 ** 62, 4000) >> g.integers(0, 62, 4000)
    ties = (g.integers(2 ** 52, 2 ** 53, 200) << 9) + 2 ** 8  # halfway between two doubles
    v = np.concatenate([v, ties, -ties, [0, 1, -1, 2 ** 62 - 1, -(2 ** 62)]]).astype(np.int64)
    o = np.empty(len(v))
    lib.to_double(ptr(v), -64, ptr(o), len(v))
    assert all(float(int(a)) * 2.0 ** -64 == b for a, b in zip(v, o))


def test_gauss_pairs(lib):
    """csrc/fx_gauss.cuh: sqrt(-ln v) (cos, sin) at every table interval's edge, next to v = 1
    and v = 0 and at random, against 60 digits: absolute error 2^-56 of max(1, modulus) (the
    header's bound) plus the rounding of the result."""
    mpmath = pytest.importorskip("mpmath")
    g = np.random.default_rng(14)
    i = np.arange(257, dtype=np.int64)
    n = np.concatenate([g.integers(1, 2 ** 53 - 2 ** 39, 1500), 1 << np.arange(53), np.arange(1, 20),
                        *[((256 + i) << s) + d for s in (44, 43, 30) for d in (-1, 0, 1)]])
    a = 2 ** 53 - n[(n > 0) & (n <= 2 ** 53 - 2 ** 39)]
    b = g.integers(0, 2 ** 53, len(a))
    b[:8] = np.arange(8) << 50
    o = np.empty((len(a), 2))
    lib.gauss(ptr(a), ptr(b), ptr(o), len(a))
    with mpmath.workdps(60):
        for ai, bi, (x, y) in zip(a, b, o):
            r = mpmath.sqrt(-mpmath.log(1 - mpmath.mpf(int(ai)) / 2 ** 53))
            w = 2 * mpmath.pi * mpmath.mpf(int(bi)) / 2 ** 53
            for v, e in ((x, r * mpmath.cos(w)), (y, r * mpmath.sin(w))):
                assert abs(mpmath.mpf(float(v)) - e) < 2.0 ** -56 * max(1, r) + 2.0 ** -53 * abs(e), (int(ai), int(bi))


PRODUCTS = r"""
#include "fx.cuh"
using namespace hqmc;
extern "C" {
// u b and conj(u) b, then (-u) b and conj(-u) b as the force's step back forms them
void products(const long long* u, const long long* b, long long* o, int n) {
  for (int i = 0; i < n; ++i) {
    const longlong2 z = make_longlong2(0, 0), x = make_longlong2(b[2 * i], b[2 * i + 1]);
    const int4 k = fx_link_limbs(u[2 * i], u[2 * i + 1]), m = make_int4(-k.x, -k.y, -k.z, -k.w);
    const longlong2 r[4] = {cfma(z, k, x), cfmac(z, k, x), cfma(z, m, x), cfmac(z, m, x)};
    for (int j = 0; j < 4; ++j) { o[8 * i + 2 * j] = r[j].x; o[8 * i + 2 * j + 1] = r[j].y; }
  }
}
}
"""


@pytest.fixture(scope="module")
def products_lib(tmp_path_factory):
    return compile_host(tmp_path_factory, PRODUCTS)


def compile_host(tmp_path_factory, text):
    if not os.path.exists(NVCC):
        pytest.skip("nvcc not found")
    d = tmp_path_factory.mktemp("fx")
    src, so = str(d / "fx.cu"), str(d / "fx.so")
    open(src, "w").write(text)
    subprocess.check_call([NVCC, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-shared", "-Xcompiler", "-fPIC",
                           "-I" + CSRC, src, "-o", so])
    return ctypes.CDLL(so)


def test_link_products_at_the_ends_of_the_low_limb(products_lib):
    """A link's low limb at -2^31, next to it and at 2^31 - 1: u b, conj(u) b and their
    negatives against exact integers.  A product is within 2 units: 1/2 of rounding, 1/4 for
    each product of two low limbs, and |b| 2^-64 < 1/2 for each component moved by a unit."""
    lows = [-2 ** 31, -2 ** 31 + 1, -1, 0, 1, 2 ** 31 - 1]
    highs = [0x1199999A, -0x0CCCCCCD, 0x4CCCCCCC, 0]
    b = [(2 ** 58 + 12345, -2 ** 59 + 2 ** 31), (-3 * 2 ** 57, 2 ** 60 - 1), (2 ** 31, -2 ** 31)]
    cases = [(h * 2 ** 32 + lo, h2 * 2 ** 32 + l2, x, y) for h in highs for lo in lows for h2 in highs[:2] for l2 in lows
             for x, y in b]
    u = np.array([c[:2] for c in cases], dtype=np.int64)
    v = np.array([c[2:] for c in cases], dtype=np.int64)
    o = np.empty((len(cases), 4, 2), np.int64)
    products_lib.products(ptr(u), ptr(v), ptr(o), len(cases))
    for (ur, ui, x, y), r in zip(cases, o):
        for (sr, si), (pr, pi) in zip(((1, 1), (1, -1), (-1, -1), (-1, 1)), r):
            er, ei = sr * ur * x - si * ui * y, sr * ur * y + si * ui * x
            assert abs(Fraction(er, 2 ** 64) - int(pr)) <= 2 and abs(Fraction(ei, 2 ** 64) - int(pi)) <= 2, (ur, ui, x, y)


PRODUCT_SUMS = r"""
#include "fx.cuh"
extern "C" void im(const long long* d, const long long* u, int shift, long long* o, int n) {
  for (int i = 0; i < n; ++i)
    o[i] = hqmc::fx_im(make_longlong2(d[2 * i], d[2 * i + 1]), make_longlong2(u[2 * i], u[2 * i + 1]), shift);
}
"""


def test_product_sums_at_the_ends_of_the_low_limb(tmp_path_factory):
    """The force's d.x u.y - d.y u.x with low words 2^31, next to it and 2^31 - 1 in every
    place, against exact integers.  In units of 2^(64 - shift): 1/2 of rounding and two
    high words cut by up to 1 of 2^32 each, so within 1."""
    lib = compile_host(tmp_path_factory, PRODUCT_SUMS)
    lows = [2 ** 31, 2 ** 31 + 1, 2 ** 31 - 1, 0]
    hi = [2 ** 24 + 1, -2 ** 25, 3, -1]
    cases = [[(h * 2 ** 32 + x) for h, x in zip(hi[k:] + hi[:k], (a, b, c, d))]
             for k in range(4) for a in lows for b in lows for c in lows for d in lows]
    q = np.array(cases, dtype=np.int64)
    d, u = np.ascontiguousarray(q[:, :2]), np.ascontiguousarray(q[:, 2:])
    for shift in (4, 10):  # sums of high limbs below 2^51: no shift above 11 (fx_force_scales)
        o = np.empty(len(q), np.int64)
        lib.im(ptr(d), ptr(u), shift, ptr(o), len(q))
        for (dx, dy, ux, uy), r in zip(cases, o):
            assert abs(Fraction(dx * uy - dy * ux, 2 ** (64 - shift)) - int(r)) <= 1, (dx, dy, ux, uy)


TO_DOUBLE = r"""
#include "fx.cuh"
extern "C" void to_double_any(const long long* v, const int* e, double* o, int n) {
  for (int i = 0; i < n; ++i) o[i] = hqmc::fx_to_double(v[i], e[i]);
}
"""


def test_to_double_at_any_exponent(tmp_path_factory):
    """v 2^e for the exponents of a slice and of a product of two slices: rounded as FP64 rounds
    it where v has 53 bits (one rounding, subnormal results included), zero below the range
    and infinite above it."""
    lib = compile_host(tmp_path_factory, TO_DOUBLE)
    g = np.random.default_rng(15)
    vs = np.concatenate([g.integers(-2 ** 53, 2 ** 53, 20), [0, 1, -1, 12345, 2 ** 60, -(2 ** 62)]])
    es = [-4300, -2400, -2100, -1800, -1700, -1600, -1500, -1301, -1300, -1200, -1138, -1137, -1100, -1074, -1000, -801, -800,
          -799, -60, 0, 799, 800, 801, 960, 1000, 1023, 1024, 1100, 1101, 1500, 1600, 1934, 2100]
    v = np.repeat(vs, len(es)).astype(np.int64)
    e = np.tile(es, len(vs)).astype(np.int32)
    o = np.empty(len(v))
    lib.to_double_any(ptr(v), ptr(e), ptr(o), len(v))
    with np.errstate(over="ignore", under="ignore"):
        want = np.ldexp(v.astype(np.float64), e)
    bad = ~(o == want)
    assert not np.any(bad), list(zip(v[bad], e[bad], o[bad], want[bad]))[:5]
