// The operator's double-precision arithmetic on the integer and FP32 pipes.
//
// GB300 retires 2 FP64 lane-operations per SM and clock, so one FP64 warp instruction
// holds its scheduler's FP64 unit for 64 cycles; an integer one takes 1 to 2.  A cell of
// the operator needs 18 neighbours, 14 additions, six squares and a square root, about 33
// FP64 instructions.  Here everything but three fused multiply-adds runs in 64-bit
// integers:
//   fix_align   the neighbours as integers of one unit.  Values of one sign and binade
//               (the usual case: the field varies by a few percent over a stencil) need
//               no conversion at all: their bit patterns differ by exactly the
//               differences of their significands.  Values of one sign and near
//               binades are shifted up, exactly; others are shifted to the largest
//               exponent, with 6 or 7 more bits below, and cut off there (2^-58 or 2^-59 of
//               the largest).
//   sums        exact sums of those integers (FP64 rounds each to half a unit in its last
//               place), so exact sums of the values in the first two forms.
//   fix_quad    the quadratic form of Sigma_d as a 62-bit integer, error below 2^-53 of it;
//               where all second differences are below 2^32 units it counts in 2^4 squared
//               units and is off by up to four of those.
//   sqrt_fix    square root to about 2^-61 (half a unit in the last place and 2^-8 of one at
//               most) from the FP32 reciprocal square root and two exact integer residuals.
//   fix_double  back to FP64, rounded once.
// A cell's error is below that of its FP64 form (tests/test_tile_accuracy.py: 0.5 to 0.95 of
// it, rms).
// Cells whose values have no such form (all zero, infinities, NaN, exponents whose
// squares leave the FP64 range) keep the FP64 code.  Every function depends on its arguments
// alone, so all kernels that update a cell give the same bits.
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#include <cuda_runtime.h>
#define MG_HD __host__ __device__ __forceinline__
#else
#define MG_HD inline
#endif

namespace mg {

MG_HD long long fix_bits(double x) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(x);
#else
  long long b;
  std::memcpy(&b, &x, 8);
  return b;
#endif
}

MG_HD double fix_from_bits(long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double x;
  std::memcpy(&x, &b, 8);
  return x;
#endif
}

MG_HD int fix_hi(long long b) { return (int)(b >> 32); }

MG_HD int fix_clz32(unsigned x) {
#ifdef __CUDA_ARCH__
  return __clz((int)x);
#else
  return x ? __builtin_clz(x) : 32;
#endif
}

MG_HD int fix_clz64(unsigned long long x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

MG_HD float fix_float(unsigned b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float x;
  std::memcpy(&x, &b, 4);
  return x;
#endif
}

// Shifts by 0 ... 31 of the 64-bit value hi:lo, word by word: the 64-bit operators cost
// two to three times as many instructions where the amount is not known.
MG_HD unsigned fix_shl_hi(unsigned lo, unsigned hi, int s) {
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, s);
#else
  return (unsigned)((((unsigned long long)hi << 32 | lo) << s) >> 32);
#endif
}
MG_HD unsigned fix_shr_lo(unsigned lo, unsigned hi, int s) {
#ifdef __CUDA_ARCH__
  return __funnelshift_r(lo, hi, s);
#else
  return (unsigned)(((unsigned long long)hi << 32 | lo) >> s);
#endif
}
MG_HD unsigned long long fix_words(unsigned lo, unsigned hi) {
  return (unsigned long long)hi << 32 | lo;
}

#ifdef __CUDA_ARCH__
__device__ __forceinline__ float fix_rsqrt(float x) {
  float y;
  asm("rsqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ int fix_rint(float x) { return __float2int_rn(x); }
#else
float fix_rsqrt(float x);  // host checks provide one with the error of the device's
inline int fix_rint(float x) {
  return x >= 2147483648.f ? 2147483647 : (int)__builtin_llrint((double)x);
}
#endif

// How the integers of a stencil read: value = (-1)^neg (integer - offset) 2^ue, where the
// offset cancels in every difference; off6 is six times it.
struct FixRef {
  long long off6;
  int ue;
  bool neg;
};

// Exponent fields whose squares, scaled by any shift of fix_quad, stay normal doubles.
constexpr int kFixMinExp = 640, kFixMaxExp = 1470;

// Replace the bit patterns b[] by integers of one unit; false when the values have no
// such form (b is then unchanged).
//
// The first six are those across the cell's faces; NV = 18 adds the twelve across its edges;
// NV = 7 and 19 have the centre last, of which six are subtracted.  Without a centre the
// largest stays below 2^60, for sums of six, with one below 2^59.
//
// near: also false where values across the edges would cut off more of the others than FP64
// does (the sums of those stand alone unless the squares of all enter beside them at the
// weight of the square-root form).
template <int NV>
MG_HD bool fix_align(long long (&b)[NV], FixRef& r, bool near = false) {
  constexpr bool kCentre = NV == 7 || NV == 19;
  constexpr int kUp = kCentre ? 6 : 7;  // bits above a significand
  const int h0 = fix_hi(b[0]);
  int diff = 0;
#pragma unroll
  for (int k = 1; k < NV; ++k) diff |= fix_hi(b[k]) ^ h0;
  const unsigned se = (unsigned)h0 >> 20;  // sign and exponent
  const int e0 = (int)(se & 0x7ffu);
  if ((diff & (int)0xfff00000) == 0 && e0 >= kFixMinExp && e0 <= kFixMaxExp) {
    r.off6 = (long long)((unsigned long long)(6u * (se - 1u)) << 52);
    r.ue = e0 - 1075;
    r.neg = h0 < 0;
    return true;
  }
  if (diff >= 0 && e0 >= kFixMinExp + 3 && e0 <= kFixMaxExp - 7) {
    // one sign: significands shifted up from three binades below the first value's
    const unsigned lo = se - 3u;
    unsigned d[NV], far = 0;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      d[k] = ((unsigned)fix_hi(b[k]) >> 20) - lo;
      far = d[k] > far ? d[k] : far;
    }
    if (far <= (unsigned)kUp) {
#pragma unroll
      for (int k = 0; k < NV; ++k)
        b[k] = (long long)((((unsigned long long)b[k] & 0xfffffffffffffULL) | 0x10000000000000ULL)
                           << d[k]);
      r.off6 = 0;
      r.ue = e0 - 1078;
      r.neg = h0 < 0;
      return true;
    }
  }
  int em = 0;
  auto largest = [&](int k) {
    const int e = fix_hi(b[k]) & 0x7ff00000;
    em = e > em ? e : em;
  };
#pragma unroll
  for (int k = 0; k < 6; ++k) largest(k);
  if (kCentre) largest(NV - 1);
  const int ef = em;
#pragma unroll
  for (int k = 6; k < NV; ++k) largest(k);
  if (em < (kFixMinExp << 20) || em > (kFixMaxExp << 20)) return false;
  if (near && em - ef > ((kUp - 2) << 20)) return false;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const int h = fix_hi(b[k]);
    int d = (em - (h & 0x7ff00000)) >> 20;
    d = d > 63 ? 63 : d;
    const long long s = b[k] >> 63;
    const unsigned long long m =
        (((unsigned long long)b[k] & 0xfffffffffffffULL) | 0x10000000000000ULL) << kUp;
    b[k] = (long long)((m >> d) ^ (unsigned long long)s) - s;
  }
  r.off6 = 0;
  r.ue = (em >> 20) - 1075 - kUp;
  r.neg = false;
  return true;
}

// (hi:lo + 2^9) 2^-10, the significand of a double with its leading bit at 2^62 rounded,
// under the exponent field be (less one: the leading bit adds it) and the sign bit.
MG_HD double fix_pack(unsigned lo, unsigned hi, int be, unsigned sign) {
  const unsigned long long t = fix_words(lo, hi) + 0x200ULL;
  const unsigned th = (unsigned)(t >> 32);
  return fix_from_bits((long long)fix_words(fix_shr_lo((unsigned)t, th, 10),
                                            ((th >> 10) + ((unsigned)be << 20)) | sign));
}

// m 2^e rounded to nearest, 2^32 <= m < 2^63; the result has to be a normal double.
MG_HD double fix_double_top(unsigned long long m, int e, unsigned sign = 0) {
  const unsigned lo = (unsigned)m, hi = (unsigned)(m >> 32);
  const int s = fix_clz32(hi) - 1;  // to bit 62
  return fix_pack(lo << s, fix_shl_hi(lo, hi, s), e - s + (10 + 52 + 1023 - 1), sign);
}

// The same for any m < 2^63.
MG_HD double fix_double(unsigned long long m, int e, unsigned sign = 0) {
  const bool up = (m >> 32) == 0;
  const double r = fix_double_top(up ? m << 31 : m, up ? e - 31 : e, sign);
  return m == 0 ? 0.0 : r;
}

MG_HD double fix_signed(long long v, const FixRef& r) {
  const unsigned n = (unsigned)(fix_hi(v) >> 31);
  const unsigned long long f = fix_words(n, n);
  return fix_double(((unsigned long long)v ^ f) - f, r.ue,
                    (n ^ (r.neg ? 0xffffffffu : 0u)) & 0x80000000u);
}

// Sum a^2 + (3/8) sum c^2 = N 2^(64 - 2 sh) of integers below 2^62 (top: their high words
// or-ed, signs removed): each value is shifted so that the largest lies in [2^61, 2^62)
// and split as h 2^32 + l with -2^31 <= l < 2^31; h^2 and h l are exact, l^2 (a quarter
// of a unit of N at most) is left out.  The shift ends at 30: N of (1, 1, 0) is 0, of
// (3, 3, 0) 16 for 18.
MG_HD unsigned long long fix_quad(const long long (&a)[3], const long long (&c)[3], int& sh,
                                  unsigned& top) {
  top = 0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int ha = fix_hi(a[k]), hc = fix_hi(c[k]);
    top |= (unsigned)(ha ^ (ha >> 31));
    top |= (unsigned)(hc ^ (hc >> 31));
  }
  sh = fix_clz32(top) - 2;
  auto form = [&](const long long (&v)[3]) {
    long long hh = 0, hl = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const unsigned lo = (unsigned)v[k], xl = lo << sh;
      const int h = (int)(fix_shl_hi(lo, (unsigned)fix_hi(v[k]), sh) + (xl >> 31));
      hh += (long long)h * h;
      hl += (long long)h * (int)xl;
    }
    return (unsigned long long)(hh + (hl >> 31));  // never negative
  };
  return form(a) + ((3ULL * form(c)) >> 3);
}

// Whether q is a normal double above 0.
MG_HD bool fix_normal(double q) {
  return ((unsigned)(fix_bits(q) >> 32) >> 20) - 1u < 2046u;
}

// sqrt(q) of a normal q > 0.  With Q = q scaled by an even power of two into
// [2^60, 2^62): s0 = Q rsqrt(Q) in FP32 as an integer (error 2^-22 of s0), then twice
// the residual Q - s^2 over 2 s0, in FP32: 2^-43, then below 2^-60.
MG_HD double sqrt_fix_normal(double q) {
  const long long b = fix_bits(q);
  const unsigned lo = (unsigned)b, hi = (unsigned)(b >> 32);
  const int e = (int)(hi >> 20);
  const int odd = (e & 1) ^ 1;  // of the unbiased exponent
  const unsigned mh = (hi & 0xfffffu) | 0x100000u;
  const unsigned long long Q = fix_words(lo << (8 + odd), fix_shl_hi(lo, mh, 8 + odd));
  const float f = fix_float((fix_shl_hi(lo, hi, 3) & 0x7fffffu) + 0x3f800000u +
                            ((unsigned)odd << 23));  // Q / 2^60 cut to 24 bits
  const float y = fix_rsqrt(f);
  const int s0 = fix_rint(f * y * 1073741824.f);
  const long long r0 = (long long)Q - (long long)s0 * s0;
  const unsigned r0l = (unsigned)r0, r0h = (unsigned)(r0 >> 32);
  // d0: units of 2^-16; the residual left is (2^32 r0 - 2^17 s0 d0 - d0^2)
  const int d0 = fix_rint((float)(int)fix_shr_lo(r0l, r0h, 12) * (y * 0.125f));
  const long long u = (long long)fix_words(r0l << 15, fix_shl_hi(r0l, r0h, 15)) -
                      (long long)s0 * d0;
  const long long dd = (long long)d0 * d0;
  const int r1 = (int)(fix_shr_lo((unsigned)u, (unsigned)(u >> 32), 5) -
                       fix_shr_lo((unsigned)dd, (unsigned)(dd >> 32), 22));
  const int d1 = fix_rint((float)r1 * (y * 0.001953125f));  // units of 2^-32
  const long long t = (long long)d0 * 65536 + d1;
  // s0 2^32 + t in [2^62, 2^63)
  return fix_pack((unsigned)t, (unsigned)s0 + (unsigned)(t >> 32),
                  ((e - 1023 - odd) >> 1) + 1022, 0);
}

// x >> d for any d >= 0, with copies of the sign from 63 on.
MG_HD long long fix_sar(long long x, int d) {
#ifdef __CUDA_ARCH__
  asm("shr.s64 %0, %0, %1;" : "+l"(x) : "r"(d));
  return x;
#else
  return x >> (d < 63 ? d : 63);
#endif
}

// b as an integer of the unit 2^-59 of a tile (mg_tile64.cuh) whose exponent field (in place)
// is em, rounded to nearest: the significand up by 8 bits, with its sign (the complement: one
// unit off), down by the difference of the exponents to twice the unit's resolution, and the
// last bit rounded, which takes the complement's unit back too.
MG_HD long long tile_convert(long long b, int em) {
  const int h = fix_hi(b);
  const unsigned s = (unsigned)(h >> 31);
  const unsigned lo = (unsigned)b, mh = (unsigned)((h & 0xfffff) | 0x100000);
  const long long t = fix_sar((long long)fix_words((lo << 8) ^ s, fix_shl_hi(lo, mh, 8) ^ s),
                              (em - (h & 0x7ff00000)) >> 20);
  return (t + 1) >> 1;
}

// The high word of a tile value's magnitude, and the bounds that one of the six across a cell's
// faces has to reach, or the unit would be too coarse for the cell: 2^-7 of the tile's range
// for an update, where six rounded values count a sixth each, and 2^-6 for a defect, to which
// the centre adds six times its own rounding.  A defect's centre of 2^-8 of the range will do
// too: it is exact, and six times it is the largest term.
MG_HD unsigned tile_mag(long long v) { return (unsigned)(fix_hi(v) ^ (fix_hi(v) >> 31)); }
constexpr unsigned kTileSmall = 1u << 21, kTileSmallDefect = 1u << 22,
                   kTileSmallCentre = 1u << 20;

#ifdef __CUDACC__
static __device__ __noinline__ float fix_to_float_rare(double x) { return (float)x; }

// (float)x, rounded to nearest even: the conversion instruction runs on the FP64 pipe.
__device__ __forceinline__ float fix_to_float(double x) {
  const int hi = __double2hiint(x);
  const unsigned lo = (unsigned)__double2loint(x);
  const unsigned h = ((unsigned)hi & 0x7fffffffu) - 0x38000000u;  // exponent bias 1023 -> 127
  if (h - 0x00100000u >= 0x0fe00000u) return fix_to_float_rare(x);  // not a normal float
  unsigned r = __funnelshift_l(lo, h, 3);
  r += ((lo << 3) + (r & 1u)) > 0x80000000u ? 1u : 0u;
  return __uint_as_float(r | ((unsigned)hi & 0x80000000u));
}
#endif

}  // namespace mg
