// Tiles of a periodic FP64 field in shared memory as integers of one unit (mg_fix64.cuh).
//
// A cell's operator reads 18 neighbours, and bringing them to one unit costs about as
// many instructions as the rest of the update: on the 256^3 lognormal workloads four
// stencils in ten cross a binade of the field or its sign.  A CTA therefore loads a tile
// of 32 x 16 x 8 cells and its shell (34 x 18 x 10 = 6120 values, 49 KB, four CTAs per
// SM), finds the largest exponent, and converts each value once, to a unit 2^-59 of it.
// Then no cell converts anything: 1.5 conversions per cell instead of 18 or 19.
//
// A value lost below the unit is less than an FP64 addition loses as long as the stencil
// holds a value within 2^-6 of the tile's largest; tile_small finds the others, which take
// their values from memory (cells at a zero of the field in a steep tile, about none).
// Tiles without such a unit (infinities, NaN, extreme exponents) go cell by cell too.
#pragma once

#include "mg_bodies64.cuh"

namespace mg {

// Levels from this side on run in tiles (a rule on the side alone, so that every caller
// gives a level the same bits).  Smaller ones have too few tiles to fill the GPU twice:
// at 96 a colour stage takes 14.0 us in 216 tiles and 12.9 us cell by cell, at 112 14.4
// against 16.8 us, at 128 15.8 against 19.6 us.
constexpr int kTileMinSide = 112;

constexpr int kTileX = 32, kTileY = 16, kTileZ = 8;
// A row holds the even x (x0 ... x0 + 32), then the odd ones (x0 - 1 ... x0 + 31), so that
// the cells of a colour, at every other x, read contiguously.
constexpr int kTileRow = 34, kTilePlane = kTileRow * (kTileY + 2);
constexpr int kTileWords = kTilePlane * (kTileZ + 2);

__host__ __device__ inline dim3 tile_grid(int n) {
  return dim3((unsigned)(n + kTileX - 1) / kTileX, (unsigned)(n + kTileY - 1) / kTileY,
              (unsigned)(n + kTileZ - 1) / kTileZ);
}

struct TileShared {
  long long v[kTileWords];
  int em[8];
  double scalar;
};

// b as an integer of the unit 2^-59 of a tile whose exponent field (in place) is em: the
// significand up by 7 bits, with its sign (the complement: one unit off), down by the
// difference of the exponents.
__device__ __forceinline__ long long tile_convert(long long b, int em) {
  const int h = fix_hi(b);
  const int d = min((em - (h & 0x7ff00000)) >> 20, 63);
  const unsigned s = (unsigned)(h >> 31);
  const unsigned lo = (unsigned)b, mh = (unsigned)((h & 0xfffff) | 0x100000);
  return (long long)fix_words((lo << 7) ^ s, fix_shl_hi(lo, mh, 7) ^ s) >> d;
}

// The largest high word of |values|, read as FP32 numbers (their order is that of the
// words; NaN patterns, from exponent field 0x7f8 on, win).
__device__ __forceinline__ float tile_max(float m, long long b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(m), "f"(fabsf(__int_as_float(fix_hi(b)))));
  return r;
}

// Which values of a tile a thread (of 256) loads, and where they go.  For a stage of a
// colour, the cells of that colour are left out: the launch is writing them, and a stencil
// never reads them.  A row with (y + z) of the colour's parity holds its cells at every
// other x, and only the 17 others are read ("half" rows, two per warp load); of the rows
// between, all 34 are.  Each of the ten planes has nine of both kinds: 19 loads per thread
// for 4590 values, where the whole box would take 25.
//   0 ... 9     full row `w` of each plane
//   10 ... 14   half rows 0 ... 7, two per warp, of five planes
//   15, 16      the ninth rows
//   17, 18      the ends x0 - 1 and x0 + 32 of the rows
struct TileMap {
  int g[2], gh, ge[2], gl[2];  // offsets in the n x n plane
  int s[2], sh, se[2], sl[2];  // places in the tile
  int ze, zl[2];               // planes of 16, 17, 18 (-1: none)
};

__device__ __forceinline__ TileMap tile_map(int n, int x0, int y0, int colour) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  auto wrap = [n](int v) { return v < 0 ? v + n : (v >= n ? v - n : v); };
  auto gxy = [&](int x, int y) { return wrap(y0 - 1 + y) * n + wrap(x0 + x); };
  // Tile row (y, z) is that of cell y0 - 1 + y, z0 - 1 + z (origins are even)
  const int cy = (colour >> 1) & 1, cx = (colour ^ 1) & 1;
  auto full = [&](int r, int z) { return 2 * r + ((z + cy + 1) & 1); };
  auto half = [&](int r, int z) { return 2 * r + ((z + cy) & 1); };
  auto npar = [&](int z) { return (cx + z + 1) & 1; };  // parity of x read in a half row
  auto place = [](int x, int y, int z) {
    return z * kTilePlane + y * kTileRow + ((x & 1) ? 18 + (x >> 1) : x >> 1);
  };
  TileMap T;
#pragma unroll
  for (int z = 0; z < 2; ++z) {
    T.g[z] = gxy(lane, full(w, z));
    T.s[z] = place(lane, full(w, z), z);
  }
  {
    const int z = w >> 2, y = half(2 * (w & 3) + (lane >> 4), z), x = 2 * (lane & 15) - npar(z);
    T.gh = gxy(x, y);
    T.sh = place(x, y, z);
  }
  T.ge[0] = gxy(lane, full(8, w));
  T.se[0] = place(lane, full(8, w), w);
  {
    // full rows of planes 8 and 9 (warps 0, 1), half rows of two planes (warps 2 to 6)
    const bool f = w < 2;
    const int z = f ? 8 + w : 2 * (w - 2) + (lane >> 4);
    const int y = f ? full(8, z) : half(8, z), x = f ? lane : 2 * (lane & 15) - npar(z);
    T.ze = w < 7 ? z : -1;
    T.ge[1] = gxy(x, y);
    T.se[1] = place(x, y, z);
  }
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    // both ends of the 90 full rows, one of the 90 half rows
    const int e = threadIdx.x + 256 * s;
    const bool f = e < 180;
    const int row = f ? e >> 1 : e - 180, z = row / 9, r = row - 9 * z;
    const int y = f ? full(r, z) : half(r, z);
    const int x = f ? ((e & 1) ? 32 : -1) : (npar(z) ? 31 : 32);
    T.zl[s] = e < 270 ? z : -1;
    T.gl[s] = gxy(x, y);
    T.sl[s] = place(x, y, z);
  }
  return T;
}

// Load and convert the tile on planes z0 - 1 ... z0 + 8 (all 256 threads); ue: its unit is
// 2^ue.  False (for every thread): it has none.
__device__ __forceinline__ bool tile_load(int n, const double* __restrict__ phi, int z0,
                                          const TileMap& T, TileShared& S, int& ue) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int n2 = n * n;
  auto zoff = [&](int z) {
    const int k = z0 - 1 + z;
    return (k < 0 ? k + n : (k >= n ? k - n : k)) * n2;
  };
  auto rd = [&](int q) { return __double_as_longlong(phi[q]); };
  long long v[19];
  if (z0 > 0 && z0 + kTileZ < n) {
    // no plane wraps
    const double* p[3] = {phi + (z0 - 1) * n2 + T.g[0], phi + (z0 - 1) * n2 + T.g[1],
                          phi + (z0 - 1 + (w >> 2)) * n2 + T.gh};
#pragma unroll
    for (int z = 0; z < 10; ++z) v[z] = __double_as_longlong(p[z & 1][(long long)z * n2]);
#pragma unroll
    for (int q = 0; q < 5; ++q) v[10 + q] = __double_as_longlong(p[2][(long long)(2 * q) * n2]);
  } else {
#pragma unroll
    for (int z = 0; z < 10; ++z) v[z] = rd(zoff(z) + T.g[z & 1]);
#pragma unroll
    for (int q = 0; q < 5; ++q) v[10 + q] = rd(zoff(2 * q + (w >> 2)) + T.gh);
  }
  v[15] = rd(zoff(w) + T.ge[0]);
  v[16] = T.ze >= 0 ? rd(zoff(T.ze) + T.ge[1]) : 0;
  v[17] = rd(zoff(T.zl[0]) + T.gl[0]);
  v[18] = T.zl[1] >= 0 ? rd(zoff(T.zl[1]) + T.gl[1]) : 0;
  float fm = 0.f;
#pragma unroll
  for (int k = 0; k < 19; ++k) fm = tile_max(fm, v[k]);
  int em = __reduce_max_sync(0xffffffffu, __float_as_int(fm) & 0x7fffffff);
  if (lane == 0) S.em[w] = em;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 8; ++k) em = max(em, S.em[k]);
  if (em < (kFixMinExp << 20) || em >= ((kFixMaxExp + 1) << 20)) {
    long long any = em;
#pragma unroll
    for (int k = 0; k < 19; ++k) any |= v[k] << 1;
    // a tile of zeros has every unit
    if (__syncthreads_or(any != 0)) return false;
    em = 1023 << 20;
  }
  em &= 0x7ff00000;
  ue = (em >> 20) - 1082;
#pragma unroll
  for (int z = 0; z < 10; ++z)
    S.v[T.s[z & 1] + (z & ~1) * kTilePlane] = tile_convert(v[z], em);
#pragma unroll
  for (int q = 0; q < 5; ++q) S.v[T.sh + 2 * q * kTilePlane] = tile_convert(v[10 + q], em);
  S.v[T.se[0]] = tile_convert(v[15], em);
  if (T.ze >= 0) S.v[T.se[1]] = tile_convert(v[16], em);
  S.v[T.sl[0]] = tile_convert(v[17], em);
  if (T.zl[1] >= 0) S.v[T.sl[1]] = tile_convert(v[18], em);
  __syncthreads();
  return true;
}

// The forms of a cell where a value of theirs is small: face, M from N and sh of fix_quad.
// In FP64 where no value around the cell (at place o of `row`, its x - 1 at l) reaches
// 2^-7 of the unit's range, so that FP64 could resolve the stencil better.
struct TileForms {
  double face, M;
};
static __device__ __noinline__ TileForms tile_forms_small(long long face, unsigned long long N,
                                                          int e, int ue, const long long* row,
                                                          int o, int l, const double* at,
                                                          NbrOff nbr) {
  auto mag = [](long long v) { return (unsigned)(fix_hi(v) ^ (fix_hi(v) >> 31)); };
  const unsigned top = mag(row[l]) | mag(row[l + 1]) | mag(row[o + kTileRow]) |
                       mag(row[o - kTileRow]) | mag(row[o + kTilePlane]) |
                       mag(row[o - kTilePlane]);
  TileForms r;
  if (top < (1u << 21)) {
    stencil_forms_fp64(at, nbr, 18, &r.face, &r.M);
  } else {
    r.face = fix_signed(face, FixRef{0, ue, false});
    r.M = fix_double(N, e);
  }
  return r;
}

// A colour stage on the tile at (x0, y0, z0) (256 threads): four cells per thread, on
// planes two apart.  From plane to plane a cell takes over what the plane between them
// gives both: the value itself and the differences across it in x and y (13 loads per cell
// instead of 18).
//
// Per stage, 512^3: 2076 us in FP64, 765 us with the integers formed cell by cell, 560 us
// in tiles; 256^3: 262, 110, 78 us; 128^3: 35.8, 19.6, 16.4 us.  What bounds it now is
// instruction issue (about 470 per 32 cells, two thirds of the slots used, the integer
// pipe 70 % busy) with the tile's loads in front: 37 us of the 78 are the load alone, whose
// 205 MB read and 40 MB written at 256^3 would take 36 us at the measured copy rate.
// Tiles 16 planes deep, or several tiles per CTA one after the other, gained 1 % at 512^3
// and lost at 256^3.
template <bool F>
__device__ __forceinline__ void b_smooth_tile64(int n, double* __restrict__ phi,
                                                const double* __restrict__ src,
                                                const double* __restrict__ f,
                                                const LevelScalars* __restrict__ sc,
                                                const OpConst64& c, int colour, int x0, int y0,
                                                int z0, TileShared& S) {
  if (threadIdx.x == 0) S.scalar = smooth_scalar64(sc, c);
  const TileMap T = tile_map(n, x0, y0, colour);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int p = w & 1, jj = (w >> 1) * 2 + (lane >> 4), m = lane & 15;
  const int px = (colour ^ p) & 1, py = ((colour >> 1) ^ p) & 1;
  const int i = x0 + 2 * m + px, j = y0 + 2 * jj + py;
  const int o = px ? 18 + m : m, l = px ? m : 17 + m;
  const int n2 = n * n;
  typedef unsigned long long u64;
  int ue;
  const bool ok = tile_load(n, phi, z0, T, S, ue);
  if (i >= n || j >= n) return;
  const double s_c = S.scalar;
  int id = (z0 + p) * n2 + j * n + i;
  if (!ok) {
    for (int k = z0 + p; k < z0 + kTileZ && k < n; k += 2)
      cell_smooth64_at(n, phi, src, f, s_c, c, i, j, k);
    return;
  }
  const long long* row = S.v + (p + 1) * kTilePlane + (2 * jj + py + 1) * kTileRow;
  auto at = [&](int q) { return (u64)row[q]; };
  u64 cz = at(o - kTilePlane), dx = at(l + 1 - kTilePlane) - at(l - kTilePlane),
      dy = at(o + kTileRow - kTilePlane) - at(o - kTileRow - kTilePlane);
#pragma unroll 1
  for (int k = z0 + p; k < z0 + kTileZ && k < n; k += 2, id += 2 * n2, row += 2 * kTilePlane) {
    const double sv = src[id];
    const double fv = F ? f[id] : 0.0;
    const u64 sx = at(l) + at(l + 1), sy = at(o + kTileRow) + at(o - kTileRow);
    const u64 cz1 = at(o + kTilePlane), dx1 = at(l + 1 + kTilePlane) - at(l + kTilePlane),
              dy1 = at(o + kTileRow + kTilePlane) - at(o - kTileRow + kTilePlane);
    const u64 sz = cz + cz1;
    const long long face = (long long)(sx + sy + sz);
    u64 N = 0;
    int sh = 0;
    unsigned tq = 1;
    if (c.mode != OP_LINEAR) {
      const long long a[3] = {(long long)(sx - sy), (long long)(sx - sz), (long long)(sy - sz)};
      const long long cc[3] = {(long long)((at(l + 1 + kTileRow) + at(l - kTileRow)) -
                                           (at(l + 1 - kTileRow) + at(l + kTileRow))),
                               (long long)(dx1 - dx), (long long)(dy1 - dy)};
      N = fix_quad(a, cc, sh, tq);
    }
    cz = cz1;
    dx = dx1;
    dy = dy1;
    const int qe = 64 - 2 * sh + 2 * ue;
    const unsigned fs = (unsigned)(fix_hi(face) >> 31);
    const u64 fm = ((u64)face ^ fix_words(fs, fs)) - fix_words(fs, fs);
    const unsigned ft = (unsigned)(fm >> 32);
    double fd, M;
    if (min(ft, tq) != 0 && (ft | tq) >= (1u << 24)) {
      fd = fix_double_top(fm, ue, fs & 0x80000000u);
      M = fix_double_top(N, qe);
    } else {
      const TileForms t = tile_forms_small(face, N, qe, ue, row, o, l, phi + id,
                                           nbr_offsets(i, j, k, n));
      fd = t.face;
      M = t.M;
    }
    double acc = F ? fma(fv, -c.h2_6, s_c) : s_c;
    if (c.mode == OP_SQRT) {
      acc = fma(c.upd_s, sqrt_clamped_fix(fma(c.e1, M, sv)), acc);
    } else {
      double q;
      bool g;
      acc = fma(-c.h2_6, root_of_M(M, sv, c, q, g), acc);
    }
    const double v = fma(fd, 1.0 / 6.0, acc);
    if (not_one(c.omega))
      relax64(phi + id, v, c.omega);
    else
      phi[id] = v;
  }
}

}  // namespace mg
