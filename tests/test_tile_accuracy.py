"""Precision of the integers that stand for FP64 values in a shared-memory tile
(csrc/mg_fix64.cuh), compiled for the host: a colour update and a defect of every cell of tiles
whose amplitude falls off, in units of 2^-53 of their largest term, against extended precision
and beside the same expressions in FP64."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <algorithm>
#include <cmath>
#include "mg_fix64.cuh"
using namespace mg;
namespace mg { float fix_rsqrt(float x) { return (float)(1.0 / std::sqrt((double)x)); } }
typedef long double Q;
typedef long long ll;
typedef unsigned long long u64;

// The forms of one stencil of tile integers v[0 ... 18] (the last the centre): the face sum and
// half of its difference to six centres; false: the unit does not resolve the stencil.
static bool forms(const ll* v, unsigned small, bool defect, ll& face, u64& N, int& sh) {
  const u64* u = (const u64*)v;
  const u64 sx = u[0] + u[1], sy = u[2] + u[3], sz = u[4] + u[5];
  face = defect ? ((ll)(sx + sy + sz) >> 1) - 3 * v[18] : (ll)(sx + sy + sz);
  const ll a[3] = {(ll)(sx - sy), (ll)(sx - sz), (ll)(sy - sz)};
  ll c[3];
  for (int k = 0; k < 3; ++k)
    c[k] = (ll)((u[6 + 4 * k] + u[7 + 4 * k]) - (u[8 + 4 * k] + u[9 + 4 * k]));
  unsigned tq, mag = 0;
  N = fix_quad(a, c, sh, tq);
  for (int k = 0; k < 6; ++k) mag |= tile_mag(v[k]);
  const bool low = defect ? tile_mag(v[18]) < kTileSmallCentre : tile_mag(face) < (small << 3);
  return tq != 0 && face != 0 && !(low && tq < (small << 3) && mag < small);
}

// p: a tile and its shell, X x Y x Z; src: the source term.  Per inner cell the error of the
// update (defect: of h^2 times the defect) in units of 2^-53 of the largest term, in the tile
// form and in FP64, -1 where the tile leaves the cell to another path.
extern "C" void errors(const double* p, const double* src, int X, int Y, int Z, double e1,
                       double h2, double k2, int defect, unsigned small, double* tile,
                       double* fp) {
  int em = 0;
  for (int o = 0; o < X * Y * Z; ++o) em = std::max(em, fix_hi(fix_bits(p[o])) & 0x7ff00000);
  const int ue = (em >> 20) - 1082;
  const double c0 = defect ? -h2 * k2 : -h2 * k2 / 6;  // of the root
  for (int z = 1; z < Z - 1; ++z)
    for (int y = 1; y < Y - 1; ++y)
      for (int x = 1; x < X - 1; ++x) {
        const int o = x + X * (y + Y * z), dx = 1, dy = X, dz = X * Y;
        const int at[19] = {o + dx,      o - dx,      o + dy,      o - dy,      o + dz,
                            o - dz,      o + dx + dy, o - dx - dy, o + dx - dy, o - dx + dy,
                            o + dx + dz, o - dx - dz, o + dx - dz, o - dx + dz, o + dy + dz,
                            o - dy - dz, o + dy - dz, o - dy + dz, o};
        double v[19];
        for (int k = 0; k < 19; ++k) v[k] = p[at[k]];
        // extended precision
        const Q qx = (Q)v[0] + v[1], qy = (Q)v[2] + v[3], qz = (Q)v[4] + v[5];
        Q M = (qx - qy) * (qx - qy) + (qx - qz) * (qx - qz) + (qy - qz) * (qy - qz);
        for (int k = 0; k < 3; ++k) {
          const Q c = (Q)v[6 + 4 * k] + v[7 + 4 * k] - v[8 + 4 * k] - v[9 + 4 * k];
          M += Q(0.375) * c * c;
        }
        const Q root = (Q)c0 * sqrtl((Q)src[o] + (Q)e1 * M);
        const Q lin = defect ? qx + qy + qz - 6 * (Q)v[18] : (qx + qy + qz) / 6;
        const Q want = lin + root - (Q)c0;
        Q big = std::max(fabsl(root), fabsl((Q)c0));
        for (int k = 0; k < 6; ++k) big = std::max(big, fabsl((Q)v[k]) / (defect ? 1 : 6));
        if (defect) big = std::max(big, 6 * fabsl((Q)v[18]));
        auto err = [&](double got) { return (double)(fabsl((Q)got - want) / big * 0x1p53L); };
        auto finish = [&](double face, double m) {
          const double r = std::fma(c0, std::sqrt(std::fma(e1, m, src[o])), -c0);
          return defect ? face + r : std::fma(face, 1.0 / 6.0, r);
        };
        // FP64
        const double sx = v[0] + v[1], sy = v[2] + v[3], sz = v[4] + v[5];
        double c[3];
        for (int k = 0; k < 3; ++k) c[k] = (v[6 + 4 * k] + v[7 + 4 * k]) - (v[8 + 4 * k] + v[9 + 4 * k]);
        const double d[3] = {sx - sy, sx - sz, sy - sz};
        const double A = std::fma(d[0], d[0], std::fma(d[1], d[1], d[2] * d[2]));
        const double B = std::fma(c[0], c[0], std::fma(c[1], c[1], c[2] * c[2]));
        const double sum = sx + sy + sz;
        fp[o] = err(finish(defect ? sum - 6.0 * v[18] : sum, std::fma(0.375, B, A)));
        // the tile
        ll t[19], face;
        for (int k = 0; k < 19; ++k) t[k] = tile_convert(fix_bits(v[k]), em);
        u64 N;
        int sh;
        if (forms(t, small, defect, face, N, sh))
          tile[o] = err(finish(fix_signed(face, FixRef{0, defect ? ue + 1 : ue, false}),
                               fix_double(N, 64 - 2 * sh + 2 * ue)));
        else
          tile[o] = -1;
      }
}
extern "C" long long convert(double x, int em) { return tile_convert(fix_bits(x), em << 20); }
extern "C" unsigned bound(int defect) { return defect ? kTileSmallDefect : kTileSmall; }
"""

X, Y, Z = 34, 18, 10


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("tile")
    src, so = d / "tile.cpp", d / "tile.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1303_0008_gb300", "csrc"), str(src), "-o", str(so)],
                   check=True)
    L = ctypes.CDLL(str(so))
    L.convert.restype = ctypes.c_longlong
    L.convert.argtypes = [ctypes.c_double, ctypes.c_int]
    return L


def field(kind, rng, defect):
    x, y, z = np.arange(X), np.arange(Y)[:, None], np.arange(Z)[:, None, None]
    noise = rng.standard_normal((Z, Y, X))
    if kind == "noise":
        return noise
    if kind == "falling":
        return noise * np.exp(-0.15 * x - 0.1 * y)
    if kind == "steep":
        return noise * np.exp(-0.5 * x - 0.3 * y)
    if kind == "crossing":
        return (x - 19 + 0.3 * y) * 0.06 + 0.002 * noise
    # "edge": one value of every 27 just above the bound, the others below it
    e = np.where((x % 3 == 1) & (y % 3 == 1) & (z % 3 == 1), -6, -8 - rng.integers(0, 4, noise.shape))
    e = e + defect
    v = np.ldexp(1 + rng.random(noise.shape), e) * np.where(rng.random(noise.shape) < 0.5, -1, 1)
    v[Z // 2, Y // 2, X // 2] = 1.5
    return v


def measure(L, kind, amp, defect, small):
    n, alpha = 128, 0.3
    c3 = 8 / 3 * alpha
    tile, fp = [], []
    for seed in range(40):
        rng = np.random.default_rng(seed)
        p = np.ascontiguousarray(amp * field(kind, rng, defect))
        src = 1 + c3 * rng.uniform(-0.3, 3.0, p.shape)
        out = [np.full(p.shape, -1.0) for _ in range(2)]
        args = [a.ctypes.data_as(ctypes.POINTER(ctypes.c_double)) for a in (p, src, *out)]
        L.errors(args[0], args[1], X, Y, Z, ctypes.c_double(c3 * alpha * n ** 4 / 3),
                 ctypes.c_double(1 / n ** 2), ctypes.c_double(2 / c3), defect,
                 ctypes.c_uint(small), args[2], args[3])
        took = out[0] >= 0
        tile.append(out[0][took])
        fp.append(out[1][took])
    return np.concatenate(tile), np.concatenate(fp)


def rms(e):
    return float(np.sqrt(np.mean(e * e)))


@pytest.mark.parametrize("defect", [0, 1])
@pytest.mark.parametrize("amp", [1e-3, 1.0])
@pytest.mark.parametrize("kind", ["noise", "falling", "steep", "crossing", "edge"])
def test_no_further_off_than_fp64(lib, kind, amp, defect):
    tile, fp = measure(lib, kind, amp, defect, lib.bound(defect))
    assert tile.size > 1000
    assert rms(tile) <= rms(fp), (rms(tile), rms(fp))
    assert tile.max() <= fp.max(), (tile.max(), fp.max())


@pytest.mark.parametrize("defect", [0, 1])
def test_the_bound_on_small_stencils_is_needed(lib, defect):
    """Without it (a planted mistake) the steep tiles' cells are far off."""
    tile, fp = measure(lib, "steep", 1.0, defect, 0)
    assert tile.max() > 10 * fp.max()


def test_conversion_is_to_nearest(lib):
    rng = np.random.default_rng(4)
    for _ in range(4000):
        x = float(np.ldexp(1 + rng.random(), int(-rng.integers(0, 64))) * rng.choice([-1, 1]))
        got, exact = lib.convert(x, 1023), x * 2.0 ** 59  # exact: a power of two
        assert abs(got - exact) <= 0.5 if abs(exact) < 2 ** 52 else got == int(exact)
    assert lib.convert(0.0, 1023) == 0 and lib.convert(-0.0, 1023) == 0
