"""The integer form of the operator's arithmetic (csrc/mg_fix64.cuh), compiled for the host,
against exact rational arithmetic: stencils of one binade, of near and far binades, of both
signs, with zeros, at binade edges, and values that it has to refuse."""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cmath>
#include "mg_fix64.cuh"
using namespace mg;
static double g_err;  // relative error of the reciprocal square root's approximation
namespace mg { float fix_rsqrt(float x) { return (float)((1 + g_err) / std::sqrt((double)x)); } }
extern "C" {
double root(double q, double err) { g_err = err; return sqrt_fix_normal(q); }
// 18 neighbours and the centre; face, M without the centre, lap with it
int forms(const double* v, double* face, double* M, double* lap) {
  long long b[18], w[19];
  for (int k = 0; k < 18; ++k) b[k] = fix_bits(v[k]);
  for (int k = 0; k < 19; ++k) w[k] = fix_bits(v[k]);
  FixRef r, t;
  if (!fix_align(b, r) || !fix_align(w, t)) return 0;
  typedef unsigned long long u;
  const u sx = (u)b[0] + b[1], sy = (u)b[2] + b[3], sz = (u)b[4] + b[5];
  *face = fix_signed((long long)(sx + sy + sz - (u)r.off6), r);
  const long long a[3] = {(long long)(sx - sy), (long long)(sx - sz), (long long)(sy - sz)};
  long long c[3];
  for (int k = 0; k < 3; ++k)
    c[k] = (long long)(((u)b[6 + 4 * k] + b[7 + 4 * k]) - ((u)b[8 + 4 * k] + b[9 + 4 * k]));
  int sh;
  unsigned top;
  const u N = fix_quad(a, c, sh, top);
  *M = fix_double(N, 64 - 2 * sh + 2 * r.ue);
  *lap = fix_signed((long long)((u)w[0] + w[1] + w[2] + w[3] + w[4] + w[5] - 6 * (u)w[18]), t);
  return 1;
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fix64")
    src, so = d / "fix64.cpp", d / "fix64.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1303_0008_gb300", "csrc"), str(src), "-o", str(so)],
                   check=True)
    L = ctypes.CDLL(str(so))
    L.root.restype = ctypes.c_double
    L.root.argtypes = [ctypes.c_double, ctypes.c_double]
    return L


def forms(L, v):
    out = [ctypes.c_double() for _ in range(3)]
    ok = L.forms((ctypes.c_double * 19)(*v), *(ctypes.byref(o) for o in out))
    return ok, [o.value for o in out]


OFFSETS = [(1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
           (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
           (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1), (0, 0, 0)]


def stencil(kind, rng):
    base = math.ldexp(1 + rng.random(), int(rng.integers(-60, 60))) * rng.choice([-1, 1])
    g = rng.standard_normal(3)
    lin = np.array([np.dot(g, o) for o in OFFSETS])
    noise = rng.standard_normal(19)
    if kind == "smooth":
        return base * (1 + 1e-3 * lin + 1e-5 * noise)
    if kind == "flat":
        return base * (1 + 1e-15 * noise)
    if kind == "edge":  # around a power of two
        return math.copysign(2.0 ** round(math.log2(abs(base))), base) * (1 + 1e-2 * lin)
    if kind == "signs":
        return base * (0.05 * lin + 1e-3 * noise)
    if kind == "rough":
        return base * noise
    if kind == "zeros":
        return base * noise * (rng.random(19) < 0.5)
    if kind == "far":  # one large value, the others down to 2^-80 of it
        return base * noise * 2.0 ** -rng.integers(0, 80, 19)
    if kind == "checker":  # the largest sums: faces against the centre
        return base * (2 - 2.0 ** -52) * np.where(np.arange(19) < 6, 1.0, -1.0)
    return base * np.where(rng.random(19) < 0.5, 1.0, 1 - 2.0 ** -53)  # "ulp"


@pytest.mark.parametrize("kind", ["smooth", "flat", "edge", "signs", "rough", "zeros", "far", "ulp",
                                  "checker"])
def test_forms(lib, kind):
    rng = np.random.default_rng(5)
    for _ in range(400):
        v = [float(x) for x in stencil(kind, rng)]
        if not any(v):
            continue
        ok, (face, M, lap) = forms(lib, v)
        assert ok
        F = [Fraction(x) for x in v]
        s = [F[0] + F[1], F[2] + F[3], F[4] + F[5]]
        a = [s[0] - s[1], s[0] - s[2], s[1] - s[2]]
        c = [F[6 + 4 * k] + F[7 + 4 * k] - F[8 + 4 * k] - F[9 + 4 * k] for k in range(3)]
        big = max(abs(x) for x in v)
        # one rounding of the result, and one unit 2^-59 for each value below 2^-7 of the largest
        unit = Fraction(big) * Fraction(1, 2 ** 58)
        for got, want, terms in ((face, sum(s), 6), (lap, sum(s) - 6 * F[18], 12)):
            assert abs(Fraction(got) - want) <= abs(want) * Fraction(1, 2 ** 53) + terms * unit
        want = sum(x * x for x in a) + Fraction(3, 8) * sum(x * x for x in c)
        # M is a square and enters through its root, next to values as large as `big`.  Its
        # own error: 2^-53 and a rounding; where all second differences are below 2^32
        # units of the last place, N counts in 2^4 squared units and is off by up to 4.  On
        # top, each of its six terms has values cut off at a unit.
        ulp = Fraction(math.ulp(big))
        root = Fraction(math.sqrt(float(want)))
        cut = 16 * unit
        assert abs(Fraction(M) - want) <= want * Fraction(1, 2 ** 52) + 64 * ulp * ulp + \
            cut * (2 * root + cut), (kind, v)


def test_refused_values(lib):
    rng = np.random.default_rng(1)
    base = list(1 + 1e-3 * rng.standard_normal(19))
    for bad in (math.inf, -math.inf, math.nan, 1e200, 1.7e308):
        v = list(base)
        v[7] = bad
        assert forms(lib, v)[0] == 0
    assert forms(lib, [0.0] * 19)[0] == 0
    assert forms(lib, [1e-200 * x for x in base])[0] == 0
    assert forms(lib, [5e-324] * 19)[0] == 0
    # within the range of exponents
    assert forms(lib, [1e-110 * x for x in base])[0] == 1
    assert forms(lib, [1e130 * x for x in base])[0] == 1


def test_square_root(lib):
    rng = np.random.default_rng(2)
    qs = [math.ldexp(1 + rng.random(), int(e)) for e in rng.integers(-1000, 1000, 4000)]
    for e in range(-6, 7):
        for x in (1.0, 1 + 2.0 ** -52, 2 - 2.0 ** -52, 1.5):
            qs.append(math.ldexp(x, e))
    qs += [2.2250738585072014e-308, 1.7976931348623157e308]
    for k, q in enumerate(qs):
        s = lib.root(q, (-1, 0, 1)[k % 3] * 2.0 ** -22)
        # nearest, up to 2^-8 of a unit in the last place: |s - sqrt q| <= (1/2 + 2^-8) ulp
        half = Fraction(math.ulp(s)) * (Fraction(1, 2) + Fraction(1, 256))
        lo, hi = Fraction(s) - half, Fraction(s) + half
        assert lo * lo <= Fraction(q) <= hi * hi
