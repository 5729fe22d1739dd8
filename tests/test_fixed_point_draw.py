"""The quaternion norm, the draw and the re-unitarisation in fixed point
(csrc/su3_fixed.cuh), compiled for the host, against 60-digit decimal values.

Tolerances (units 2^-60, derived).  A product sum drops at most 4 units per
real product and rounds by one half; a reciprocal square root is within 6
units of its argument's (test_fixed_point.py).
  norm: the sum of four squares 16.5 at most (without the low products that
    norm_fx adds); |a| 16.5 / 2 sqrt(n) + 6 n + 4.5 < 40 for n in [1/4, 4); the
    inverse 16.5 / (2 n^1.5) + 6 <= 72, and the direction 72 + 4.5 < 80.
  X: relative, 36 of the inverse, 4.5 / (1/4) and 4.5 / (1/8) of the two
    products < 100; one unit of the final shift.
  rho^2 = X (2 - X): 4.5 x 2^4 of the product (X = Q 2^e, e <= 4), and twice
    the square root's 16: < 128.
  quaternion product: 4 x 4 + 1/2 < 17.
  Gram-Schmidt of rows with squared norms in [0.6, 1.6]: first row 40, inner
    product 140, second row before its norm 250 and after it 2300, third row
    twice two products of those < 2^13.
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
ONE = 2 ** 60

SOURCE = r"""
#include "su3_fixed.cuh"
using namespace su3g;
extern "C" {
// o: v[4], y, kappa, s
int t_norm(const int64_t *a, int64_t *o) {
  FxNorm n = {};
  int32_t large = 0;
  const bool ok = norm_fx<false>(a, n, large);
  // the same mark beside a count
  FxNorm m = {};
  int32_t count = 762;
  if (norm_fx<true>(a, m, count) != ok || (count < 0) != (large < 0) || (count & INT32_MAX) != 762) return -1;
  const int st = large < 0 ? 2 : ok;
  for (int q = 0; q < 4; ++q) o[q] = fx_val(n.v[q]);
  o[4] = fx_val(n.y);
  o[5] = n.kappa;
  o[6] = n.s;
  return st;
}
// o: X, x[4]
int t_draw(const int64_t *a, int64_t L, int64_t u4sq, int64_t m, int e, const int64_t *dir, int64_t *o) {
  FxNorm n;
  int32_t large = 0;
  if (!norm_fx<false>(a, n, large) || large < 0) return -1;
  Proposal p = {};
  const int st = (int)propose_fx(L, u4sq, n, InvBeta{m, e}, p);
  if (st != kAccepted) return st;
  const Direction d = {fx_split(dir[0]), fx_split(dir[1]), fx_split(dir[2]), fx_split(dir[3])};
  Fx x[4];
  direction_fx(p, d, x);
  o[0] = p.X;
  for (int q = 0; q < 4; ++q) o[1 + q] = fx_val(x[q]);
  return st;
}
void t_quat(const int64_t *x, const int64_t *v, int64_t *o) {
  Fx a[4], b[4], r[4];
  for (int q = 0; q < 4; ++q) {
    a[q] = fx_split(x[q]);
    b[q] = fx_split(v[q]);
  }
  quat_fx(a, b, r);
  for (int q = 0; q < 4; ++q) o[q] = fx_val(r[q]);
}
int t_reunit(int64_t *m) {
  FM3 f;
  for (int i = 0; i < 9; ++i) f.e[i / 3][i % 3] = {fx_split(m[2 * i]), fx_split(m[2 * i + 1])};
  FxRange rg;
  if (!reunit_f<false>(f, rg) || !rg.ok()) return 0;
  for (int i = 0; i < 9; ++i) {
    m[2 * i] = fx_val(f.e[i / 3][i % 3].re);
    m[2 * i + 1] = fx_val(f.e[i / 3][i % 3].im);
  }
  return 1;
}
}
"""
VANISHES, NORMED, TOO_LARGE = 0, 1, 2


@pytest.fixture(scope="module")
def fx(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fxd")
    src, so = d / "fxd.cpp", d / "fxd.so"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-O2", "-std=c++17", "-Wno-unknown-pragmas", "-shared", "-fPIC", "-I", CSRC, str(src), "-o",
                    str(so)], check=True)
    return ctypes.CDLL(str(so))


def arr(v):
    return (ctypes.c_int64 * len(v))(*v)


def norm(fx, a):
    """(status, v, y, kappa, s) of a in units 2^-57."""
    o = arr([0] * 7)
    st = fx.t_norm(arr(a), o)
    return st, list(o[:4]), o[4], o[5], o[6]


def projections(rng, count, lo, hi):
    """Projections (units 2^-57) of norm 2^lo .. 2^hi, single components among them."""
    for i in range(count):
        g = [rng.gauss(0, 1) for _ in range(4)]
        if i % 5 == 0:
            g = [g[q] if q == i // 5 % 4 else 0.0 for q in range(4)]
        size = 2.0 ** rng.uniform(lo, hi) / sum(x * x for x in g) ** 0.5
        yield [int(x * size * 2 ** 57) for x in g]


def test_norm(fx):
    assert norm(fx, [0, 0, 0, 0])[0] == VANISHES
    for a in projections(random.Random(1), 2000, -40, 2.999):
        k = sum(Decimal(x) ** 2 for x in a).sqrt()  # units 2^-57
        st, v, _, kappa, s = norm(fx, a)
        assert st == NORMED, a
        # k = kappa 2^(3 - s): the difference in units of kappa
        assert abs(Decimal(kappa) - k * 2 ** s) < 40, a
        assert max(abs(Decimal(x) - Decimal(y) / k * ONE) for x, y in zip(v, a)) < 80, a


def test_norm_of_eight_and_more_is_refused(fx):
    """SU(3) links have |a| <= 6; links that pass the range check without
    being unitary reach more, up to the 64 of the units."""
    for a in projections(random.Random(2), 2000, 3.001, 5.6):
        assert norm(fx, a)[0] == TOO_LARGE, a
    for x in (7.9, 8.1, 13.4, 31.0, 60.0):
        for q in range(4):
            a = [0] * 4
            a[q] = int(x * 2 ** 57)
            want = NORMED if x < 8 else TOO_LARGE
            assert norm(fx, a)[0] == want and norm(fx, [-t for t in a])[0] == want
    # no component of 8, the norm beyond
    assert norm(fx, [int(4.1 * 2 ** 57)] * 4)[0] == TOO_LARGE
    assert norm(fx, [int(3.9 * 2 ** 57)] * 4)[0] == NORMED


def test_draw(fx):
    rng = random.Random(3)
    accepted = 0
    for a in projections(rng, 3000, -6, 2.9):
        k = sum(Decimal(x) ** 2 for x in a).sqrt() / 2 ** 57
        beta = 2.0 ** rng.uniform(-3, 6)
        m, e = 1.5 / beta, 0
        while m >= 1:
            m, e = m / 2, e + 1
        while m < 0.5:
            m, e = m * 2, e - 1
        mi = int(m * ONE)
        L = int(2.0 ** rng.uniform(-11.9, 5.4) * 2 ** 57)
        X = Decimal(L) / 2 ** 57 * Decimal(mi) / ONE * Decimal(2) ** e / k
        u4sq = rng.randrange(ONE)
        edge = 1 - X / 2 - Decimal(u4sq) / ONE
        if abs(edge) < Decimal(2) ** -40:
            continue
        # theta = 0: the third component is the length
        o = arr([0] * 5)
        st = fx.t_draw(arr(a), ctypes.c_int64(L), ctypes.c_int64(u4sq), ctypes.c_int64(mi), e, arr([0, ONE, ONE, 0]), o)
        assert st == (1 if edge > 0 else 0), (a, beta, L)
        if st != 1:
            continue
        accepted += 1
        assert abs(Decimal(o[0]) - X * ONE) <= 100 * X + 1
        assert o[1] == ONE - o[0] and o[2] == 0 and o[3] == 0
        got = Decimal(o[0]) / ONE
        assert abs((Decimal(o[4]) / ONE) ** 2 - got * (2 - got)) * ONE < 128
    assert accepted > 500


def test_quaternion_product(fx):
    rng = random.Random(4)
    for _ in range(500):
        x, v = ([int(t * ONE) for t in unit(rng)] for _ in range(2))
        o = arr([0] * 4)
        fx.t_quat(arr(x), arr(v), o)
        (x0, x1, x2, x3), (v0, v1, v2, v3) = x, v
        want = [x0 * v0 + x1 * v1 + x2 * v2 + x3 * v3, -x0 * v1 + v0 * x1 + x2 * v3 - x3 * v2,
                -x0 * v2 + v0 * x2 + x3 * v1 - x1 * v3, -x0 * v3 + v0 * x3 + x1 * v2 - x2 * v1]
        assert max(abs(Decimal(a) - Decimal(b) / ONE) for a, b in zip(o, want)) < 17


def unit(rng):
    g = [rng.gauss(0, 1) for _ in range(4)]
    n = sum(t * t for t in g) ** 0.5
    return [t / n for t in g]


def cmul(a, b):
    return a[0] * b[0] - a[1] * b[1], a[0] * b[1] + a[1] * b[0]


def test_reunitarisation(fx):
    rng = random.Random(5)
    done = 0
    for _ in range(1000):
        rows = [[complex(rng.gauss(0, 1), rng.gauss(0, 1)) for _ in range(3)] for _ in range(2)]
        size = [abs(sum(abs(z) ** 2 for z in r)) ** 0.5 for r in rows]
        inner = sum(p.conjugate() * q for p, q in zip(*rows)) / size[0] / size[1]
        if abs(inner) > 0.3:
            continue
        rows = [[z / s * rng.uniform(0.85, 1.15) for z in r] for r, s in zip(rows, size)]
        m = [int(t * ONE) for r in rows for z in r for t in (z.real, z.imag)]
        if max(map(abs, m)) > ONE:
            continue
        a, b = ([(Decimal(m[6 * i + 2 * k]) / ONE, Decimal(m[6 * i + 2 * k + 1]) / ONE) for k in range(3)]
                for i in range(2))
        s = 1 / sum(x * x + y * y for x, y in a).sqrt()
        a = [(x * s, y * s) for x, y in a]
        q = [sum(t) for t in zip(*(cmul((x, -y), z) for (x, y), z in zip(a, b)))]
        b = [(z[0] - w[0], z[1] - w[1]) for z, w in zip(b, (cmul(q, z) for z in a))]
        s = 1 / sum(x * x + y * y for x, y in b).sqrt()
        b = [(x * s, y * s) for x, y in b]
        c = []
        for k in range(3):
            p, r = cmul(a[(k + 1) % 3], b[(k + 2) % 3]), cmul(a[(k + 2) % 3], b[(k + 1) % 3])
            c.append((p[0] - r[0], -(p[1] - r[1])))
        got = arr(m + [0] * 6)
        assert fx.t_reunit(got) == 1
        want = [t for row in (a, b, c) for z in row for t in z]
        assert max(abs(Decimal(g) - w * ONE) for g, w in zip(got, want)) < 2 ** 13
        done += 1
    assert done > 100
