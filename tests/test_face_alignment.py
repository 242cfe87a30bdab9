"""Face sums of the integer form (csrc/mg_fix64.cuh) where values across a cell's edges are far
larger than those across its faces: the linear form aligns the latter alone, the conjugate one
leaves such cells to FP64.  Compiled for the host, against exact rational arithmetic."""
import ctypes
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
namespace mg { float fix_rsqrt(float x) { return (float)(1.0 / std::sqrt((double)x)); } }
template <int NV>
static int face(const double* v, int near, double* out) {
  long long b[NV];
  for (int k = 0; k < NV; ++k) b[k] = fix_bits(v[(NV & 1) && k == NV - 1 ? 18 : k]);
  FixRef r;
  if (!fix_align(b, r, near != 0)) return 0;
  unsigned long long s = 0;
  for (int k = 0; k < 6; ++k) s += b[k];
  *out = fix_signed((long long)(s - ((NV & 1) ? 6 * (unsigned long long)b[NV - 1] : r.off6)), r);
  return 1;
}
// six faces, twelve edges, the centre
extern "C" int sum(int nv, const double* v, int near, double* out) {
  return nv == 6 ? face<6>(v, near, out) : nv == 7 ? face<7>(v, near, out)
       : nv == 18 ? face<18>(v, near, out) : face<19>(v, near, out);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("faces")
    src, so = d / "faces.cpp", d / "faces.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1303_0008_gb300", "csrc"), str(src), "-o", str(so)],
                   check=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("nv,near", [(6, 0), (7, 0), (18, 1), (19, 1)])
@pytest.mark.parametrize("centre", ["as the faces", "as the edges"])
def test_face_sums(lib, nv, near, centre):
    rng = np.random.default_rng(3)
    err, err64, taken = [], [], 0
    for t in range(4000):
        v = rng.standard_normal(19)
        v[6:18] *= 2.0 ** (t % 40)
        if centre == "as the edges":
            v[18] *= 2.0 ** (t % 40)
        out = ctypes.c_double()
        ok = lib.sum(nv, (ctypes.c_double * 19)(*v), near, ctypes.byref(out))
        assert ok or near
        if not ok:
            continue
        taken += 1
        got = out.value
        want = sum(Fraction(x) for x in v[:6])
        fp = (v[0] + v[1]) + (v[2] + v[3]) + (v[4] + v[5])
        big = np.abs(v[:6]).max()
        if nv & 1:
            want -= 6 * Fraction(v[18])
            fp = fp - 6.0 * v[18]
            big = max(big, 6 * abs(v[18]))
        err.append(float(abs(Fraction(got) - want)) / (2.0 ** -53 * big))
        err64.append(float(abs(Fraction(fp) - want)) / (2.0 ** -53 * big))
    assert taken >= 400
    # one rounding of the sum, and values cut off (twice the unit of the faces' 2^-6)
    assert max(err) <= 6 + 6
    assert np.sqrt(np.mean(np.square(err))) <= np.sqrt(np.mean(np.square(err64)))
