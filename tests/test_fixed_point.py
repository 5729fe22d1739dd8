"""The fixed-point arithmetic of the FP64 update (csrc/su3_fixed.cuh), compiled
for the host: its functions against 60-digit decimal values, its product sums
against exact integers.

Tolerances (units 2^-60, derived): a logarithm is a table value and a series
rounded to 2^-57 (4 units) plus z times the rounding of ln 2 in units 2^-57
(z <= 32: 128 units); sine and cosine carry the 2^-41 rounding of d^2 (2^-42
x 2^-4.6 x 2^-10.7 = 2^-57.3, 7 units) and of the last coefficients, with
five products of at most 4 dropped units each: 32 units in all; a reciprocal
square root three truncations below 2 units.
"""
import ctypes
import os
import random
import shutil
import subprocess
from decimal import Decimal, getcontext

import pytest

getcontext().prec = 60
HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_0904_0642_gb300", "csrc")

SOURCE = r"""
#include "su3_fixed.cuh"
using namespace su3g;
extern "C" {
int64_t t_log(uint32_t w) { return neg_log_fx(w); }
void t_trig(uint32_t w, int half, int64_t *o) { trig_fx(w, half, o[0], o[1]); }
int64_t t_rsqrt(int64_t n) { return rsqrt_fx(fx_split(n)); }
int64_t t_of(double x) { return fx_val(fx_of(x)); }
double t_to(int64_t v, int e) { return dbl_of(v, e); }
int64_t t_neg(int64_t v) { return fx_val(fx_neg(fx_split(v))); }
int t_range(double re, double im) { FxRange r; fc_of(re, im, r); return r.ok(); }
int64_t t_dot(const int64_t *a, const int64_t *b, int n) {
  FxAcc s = {0, kHalf60};
  for (int i = 0; i < n; ++i) fmac(s, fx_split(a[i]), fx_split(b[i]));
  return fold60(s);
}
}
"""


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fx")
    src, so = d / "fx.cpp", d / "fx.so"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(so)], check=True)
    L = ctypes.CDLL(str(so))
    i64, u32, i32, dbl = ctypes.c_int64, ctypes.c_uint32, ctypes.c_int, ctypes.c_double
    for name, res, args in [("t_log", i64, [u32]), ("t_trig", None, [u32, i32, ctypes.POINTER(i64)]),
                            ("t_rsqrt", i64, [i64]), ("t_of", i64, [dbl]), ("t_to", dbl, [i64, i32]),
                            ("t_neg", i64, [i64]), ("t_range", i32, [dbl, dbl]),
                            ("t_dot", i64, [ctypes.POINTER(i64), ctypes.POINTER(i64), i32])]:
        f = getattr(L, name)
        f.restype, f.argtypes = res, args
    return L


def _words():
    rng = random.Random(3)
    edges = [0, 1, 2, 3, 2 ** 31 - 1, 2 ** 31, 2 ** 32 - 1, 2 ** 32 - 2, 2 ** 24 - 1, 2 ** 24, 2 ** 25]
    return edges + [1 << k for k in range(32)] + [rng.getrandbits(32) for _ in range(400)]


def _sincos(t):
    s, c, term, n = Decimal(0), Decimal(0), Decimal(1), 0
    while abs(term) > Decimal(10) ** -45:
        sign = 1 if n % 4 < 2 else -1
        if n % 2:
            s += sign * term
        else:
            c += sign * term
        n += 1
        term = term * t / n
    return s, c


def test_logarithm(fx):
    for w in _words():
        u = (Decimal(w) + Decimal("0.5")) / 2 ** 32
        assert abs(Decimal(fx.t_log(w)) / 2 ** 57 + u.ln()) * 2 ** 60 < 132, w


def test_sine_cosine(fx):
    pi = Decimal("3.14159265358979323846264338327950288419716939937510582097494")
    out = (ctypes.c_int64 * 2)()
    for w in _words()[:200]:
        for half in (0, 1):
            s, c = _sincos(2 * pi * (Decimal(w) + Decimal(half) / 2) / 2 ** 32)
            fx.t_trig(w, half, out)
            assert max(abs(out[0] - c * 2 ** 60), abs(out[1] - s * 2 ** 60)) < 32, (w, half)


def test_reciprocal_square_root(fx):
    rng = random.Random(5)
    for n in [2 ** 58, 2 ** 60, 2 ** 62 - 1] + [rng.randrange(2 ** 58, 2 ** 62) for _ in range(500)]:
        want = 1 / (Decimal(n) / 2 ** 60).sqrt() * 2 ** 60
        assert abs(fx.t_rsqrt(n) - want) < 6, n


def test_conversions_and_range(fx):
    rng = random.Random(7)
    for x in [0.0, -0.0, 1.0, -1.0, 2.0 ** -28, 2.0 ** -29, -2.0 ** -30, 1e-310, 1.0625] + [
            rng.uniform(-1, 1) * 2.0 ** -rng.randrange(70) for _ in range(500)]:
        v = fx.t_of(x)
        assert abs(Decimal(v) - Decimal(x) * 2 ** 60) <= 1, x
        if abs(v) >= 2 ** 20:
            assert abs(Decimal(fx.t_to(v, 60)) * 2 ** 60 - v) <= Decimal(abs(v)) / 2 ** 53
    assert fx.t_to(0, 60) == 0.0 and fx.t_to(2 ** 60, 60) == 1.0 and fx.t_to(-(2 ** 60), 60) == -1.0
    for v in (-2 ** 31, 2 ** 31, -2 ** 60, 2 ** 60, 5 * 2 ** 32 - 2 ** 31, 0):
        assert fx.t_neg(v) == -v
    inf, nan = float("inf"), float("nan")
    assert all(fx.t_range(a, b) for a, b in ((1.0, -1.0), (0.0, -0.0), (-1.0625, 1.0625)))
    assert not any(fx.t_range(a, b) for a, b in ((1.07, 0.0), (0.0, -1.07), (inf, 0.0), (0.0, -inf), (nan, 0.0),
                                                 (0.0, -nan), (1e300, 0.0)))


@pytest.mark.parametrize("low", [2 ** 31 - 1, -2 ** 31, None])
def test_products_do_not_wrap(fx, low):
    """Six products of elements at the range limit, with the low limbs at
    either end: the sum equals the integer sum less the dropped products."""
    rng = random.Random(11)
    lim = int(1.0625 * 2 ** 28)
    for _ in range(200):
        limbs = [[((rng.choice((-lim, lim)), low) if low is not None else
                   (rng.randrange(-lim, lim), rng.randrange(-2 ** 31, 2 ** 31))) for _ in range(6)] for _ in range(2)]
        vals = [[h * 2 ** 32 + l for h, l in side] for side in limbs]
        arr = [(ctypes.c_int64 * 6)(*side) for side in vals]
        t = sum(((ha * hb) << 32) + ha * lb + la * hb for (ha, la), (hb, lb) in zip(*limbs)) + (1 << 27)
        assert fx.t_dot(arr[0], arr[1], 6) == t >> 28
