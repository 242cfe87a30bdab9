// Tiles of a periodic FP64 field in shared memory as integers of one unit (mg_fix64.cuh).
//
// A cell's operator reads 18 neighbours, and bringing them to one unit costs about as
// many instructions as the rest of the update: on the 256^3 lognormal workloads four
// stencils in ten cross a binade of the field or its sign.  A CTA therefore loads a tile
// of 32 x 16 x 8 cells and its shell (34 x 18 x 10 = 6120 values, 49 KB, four CTAs per
// SM), finds the largest exponent, and converts each value once, to a unit 2^-59 of it.
// Then no cell converts anything: 1.5 conversions per cell in the kernels that visit every
// cell and 4.5 per updated cell in a colour stage (4590 values for 1024 cells), instead of 18
// or 19.
//
// Values within 2^-7 of the tile's largest keep all their bits; the others are rounded to the
// unit.  That loses less than FP64 additions do as long as one of the six neighbours
// across a face reaches 2^-7 of the tile's largest (for a defect 2^-6, or its centre 2^-8);
// tile_small finds the other cells (those at a zero of the field in a steep tile), which take
// their values from memory.  In units of 2^-53 of an update's largest term, the error of a cell
// (rms and worst of 160000) where 1.07 and 5.3 are FP64's: 0.88 and 4.2 on noise whose amplitude
// falls as exp(-0.15 i - 0.1 j) through the tile (with the values cut off instead of rounded
// 1.14 and 6.5), 0.89 and 3.8 on noise of one amplitude.  The rounding costs a colour stage
// 0.8 % (256^3 76.9 -> 77.6 us).
// Tiles without such a unit (infinities, NaN, extreme exponents) go cell by cell too.
#pragma once

#include "mg_bodies64.cuh"

namespace mg {

// Levels from this side on run in tiles (a rule on the side alone, so that every caller
// gives a level the same bits).  Smaller ones have too few tiles to fill the GPU: at 112, 392
// tiles, a colour stage takes 13.9 us in tiles and 16.7 us cell by cell (residual 43.5 against
// 70.0), at 128 14.3 against 22.7 us.  The line was drawn where 96 took 14.0 against 12.9 us;
// with one kernel per form and the rare cells lane by lane it takes 9.9 against 12.9 (residual
// 27.5 against 44.5), so it could lie lower.
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

__host__ __device__ inline unsigned tile_count(int n) {
  const dim3 g = tile_grid(n);
  return g.x * g.y * g.z;
}

// Whether a level runs in tiles: its operator in the square-root or the linear form.  The
// others (a splitting constant of its own, |alpha| < 1e-4) divide and would cost the tile
// kernels the registers of their fourth CTA per SM; their cells go one by one.
__host__ __device__ inline bool in_tiles(int n, const OpConst64& c) {
  return n >= kTileMinSide && (c.mode == OP_SQRT || c.mode == OP_LINEAR);
}
// Its colour stages: with the plain step (omega = 1) only.
__host__ __device__ inline bool smooth_in_tiles(int n, const OpConst64& c) {
  return in_tiles(n, c) && c.omega == 1.0;
}

// The tile's place in the order of a launch over tile_grid.
__device__ __forceinline__ unsigned tile_index() {
  return blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z);
}

struct TileShared {
  long long v[kTileWords];
  int em[8];
  double scalar;
};

// The largest high word of |values|, read as FP32 numbers (their order is that of the
// words; NaN patterns, from exponent field 0x7f8 on, win).
__device__ __forceinline__ float tile_max(float m, long long b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(m), "f"(fabsf(__int_as_float(fix_hi(b)))));
  return r;
}

// The exponent field (in place) of the largest of all threads' values, -1 where the tile
// has no unit; with bit 0 set where all values are 0.  Every thread gets the same.
template <int NV>
__device__ __forceinline__ int tile_exponent(const long long (&v)[NV], TileShared& S) {
  float fm = 0.f;
#pragma unroll
  for (int k = 0; k < NV; ++k) fm = tile_max(fm, v[k]);
  int em = __reduce_max_sync(0xffffffffu, __float_as_int(fm) & 0x7fffffff);
  if ((threadIdx.x & 31) == 0) S.em[threadIdx.x >> 5] = em;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 8; ++k) em = max(em, S.em[k]);
  if (em < (kFixMinExp << 20) || em >= ((kFixMaxExp + 1) << 20)) {
    long long any = em;
#pragma unroll
    for (int k = 0; k < NV; ++k) any |= v[k] << 1;
    // a tile of zeros has every unit
    if (__syncthreads_or(any != 0)) return -1;
    return 1023 << 20 | 1;
  }
  return em & 0x7ff00000;
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
  const int w = threadIdx.x >> 5;
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
  const int code = tile_exponent(v, S), em = code & ~1;
  if (code < 0) return false;
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

// Whether no value around the cell reaches `bound` (kTileSmall), so that FP64 could resolve
// the stencil better (row[o]: its place, row[l], row[r]: its neighbours in x).
__device__ __forceinline__ bool tile_small(const long long* row, int o, int l, int r,
                                           unsigned bound) {
  return (tile_mag(row[l]) | tile_mag(row[r]) | tile_mag(row[o + kTileRow]) |
          tile_mag(row[o - kTileRow]) | tile_mag(row[o + kTilePlane]) |
          tile_mag(row[o - kTilePlane])) < bound;
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
// Cells that need another path (a value of theirs small against the tile, a vanishing or
// infinite discriminant) are left for the end: no other cell of the stage reads them.
template <bool F, bool LIN>
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
  const int i = x0 + 2 * m + px, j = y0 + 2 * jj + py, k0 = z0 + p;
  const int n2 = n * n;
  typedef unsigned long long u64;
  int ue;
  const bool ok = tile_load(n, phi, z0, T, S, ue);
  if (i >= n || j >= n) return;
  const double s_c = S.scalar;
  unsigned rare = 0xf;
  if (ok) {
    rare = 0;
    const int o = px ? 18 + m : m, l = px ? m : 17 + m;
    const long long* row = S.v + (p + 1) * kTilePlane + (2 * jj + py + 1) * kTileRow;
    auto at = [&](int q) { return (u64)row[q]; };
    u64 cz = at(o - kTilePlane), dx = at(l + 1 - kTilePlane) - at(l - kTilePlane),
        dy = at(o + kTileRow - kTilePlane) - at(o - kTileRow - kTilePlane);
    int id = k0 * n2 + j * n + i;
#pragma unroll 1
    for (int s = 0; s < 4 && k0 + 2 * s < n; ++s, id += 2 * n2, row += 2 * kTilePlane) {
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
      if (!LIN) {
        const long long a[3] = {(long long)(sx - sy), (long long)(sx - sz), (long long)(sy - sz)};
        const long long cc[3] = {(long long)((at(l + 1 + kTileRow) + at(l - kTileRow)) -
                                             (at(l + 1 - kTileRow) + at(l + kTileRow))),
                                 (long long)(dx1 - dx), (long long)(dy1 - dy)};
        N = fix_quad(a, cc, sh, tq);
      }
      cz = cz1;
      dx = dx1;
      dy = dy1;
      const unsigned fs = (unsigned)(fix_hi(face) >> 31);
      const u64 fm = ((u64)face ^ fix_words(fs, fs)) - fix_words(fs, fs);
      const unsigned ft = (unsigned)(fm >> 32);
      bool bad = min(ft, tq) == 0 || ((ft | tq) < 8 * kTileSmall && tile_small(row, o, l, l + 1, kTileSmall));
      double acc = F ? fma(fv, -c.h2_6, s_c) : s_c;
      if (LIN) {
        acc = fma(-c.h2_6, sv, acc);
      } else {
        const double q = fma(c.e1, fix_double_top(N, 64 - 2 * sh + 2 * ue), sv);
        bad = bad || !fix_normal(q);
        acc = fma(c.upd_s, sqrt_fix_normal(q), acc);
      }
      if (bad)
        rare |= 1u << s;
      else
        phi[id] = fma(fix_double_top(fm, ue, fs & 0x80000000u), 1.0 / 6.0, acc);
    }
  }
#pragma unroll 1
  for (; rare != 0; rare &= rare - 1) {
    const int k = k0 + 2 * (__ffs((int)rare) - 1);
    if (k < n)
      cell_smooth64_at<LIN ? OP_LINEAR : OP_SQRT>(n, phi, src, f, s_c, c, i, j, k);
  }
}

// The whole tile, every row in the order of x (x0 - 1 first): for the kernels that visit
// every cell.  Loads as tile_load: rows w and w + 8 of each plane, the last two rows of the
// planes, then the ends of the rows.  0: no unit; 2: all values are 0; 1 otherwise.
__device__ __forceinline__ int tile_load_all(int n, const double* __restrict__ phi, int x0,
                                              int y0, int z0, TileShared& S, int& ue) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int n2 = n * n;
  auto wrap = [n](int v) { return v < 0 ? v + n : (v >= n ? v - n : v); };
  auto gxy = [&](int x, int y) { return wrap(y0 - 1 + y) * n + wrap(x0 + x); };
  auto zoff = [&](int z) { return wrap(z0 - 1 + z) * n2; };
  auto rd = [&](int q) { return __double_as_longlong(phi[q]); };
  long long v[25];
  const int g0 = gxy(lane, w), g1 = gxy(lane, w + 8);
  if (z0 > 0 && z0 + kTileZ < n) {
    const double* p0 = phi + (z0 - 1) * n2 + g0;
    const double* p1 = phi + (z0 - 1) * n2 + g1;
#pragma unroll
    for (int z = 0; z < 10; ++z) {
      v[2 * z] = __double_as_longlong(p0[(long long)z * n2]);
      v[2 * z + 1] = __double_as_longlong(p1[(long long)z * n2]);
    }
  } else {
#pragma unroll
    for (int z = 0; z < 10; ++z) {
      v[2 * z] = rd(zoff(z) + g0);
      v[2 * z + 1] = rd(zoff(z) + g1);
    }
  }
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const int e = w + 8 * r;
    v[20 + r] = e < 20 ? rd(zoff(e >> 1) + gxy(lane, 16 + (e & 1))) : 0;
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int h = threadIdx.x + 256 * r, row = h >> 1, z = row / 18, y = row - 18 * z;
    v[23 + r] = row < 180 ? rd(zoff(z) + gxy((h & 1) ? 32 : -1, y)) : 0;
  }
  const int code = tile_exponent(v, S), em = code & ~1;
  if (code < 0) return 0;
  ue = (em >> 20) - 1082;
  long long* t = S.v + w * kTileRow + lane + 1;
#pragma unroll
  for (int z = 0; z < 10; ++z) {
    t[z * kTilePlane] = tile_convert(v[2 * z], em);
    t[z * kTilePlane + 8 * kTileRow] = tile_convert(v[2 * z + 1], em);
  }
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const int e = w + 8 * r;
    if (e < 20)
      S.v[(e >> 1) * kTilePlane + (16 + (e & 1)) * kTileRow + lane + 1] =
          tile_convert(v[20 + r], em);
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int h = threadIdx.x + 256 * r, row = h >> 1;
    if (row < 180) S.v[row * kTileRow + ((h & 1) ? 33 : 0)] = tile_convert(v[23 + r], em);
  }
  __syncthreads();
  return 1 + (code & 1);
}

// What a column of cells passes from plane to plane: value, differences across in x and y.
struct TilePlane {
  unsigned long long c, dx, dy;
};
__device__ __forceinline__ TilePlane tile_plane(const long long* q) {
  typedef unsigned long long u64;
  return TilePlane{(u64)q[0], (u64)q[1] - (u64)q[-1], (u64)q[kTileRow] - (u64)q[-kTileRow]};
}

// The defect L phi (without a right-hand side) of the cell at q in the tile (tile_load_all),
// between the planes lo and up.  False: it needs another path, as in b_smooth_tile64.
template <bool LIN>
__device__ __forceinline__ bool tile_defect(const long long* q, const TilePlane& lo,
                                            const TilePlane& mid, const TilePlane& up, int ue,
                                            double src, const OpConst64& c, double& d, double& qd) {
  typedef unsigned long long u64;
  auto v = [&](int k) { return (u64)q[k]; };
  const u64 sx = v(1) + v(-1), sy = v(kTileRow) + v(-kTileRow), sz = lo.c + up.c;
  // half of the difference: twelve values would pass 64 bits
  const long long lap = ((long long)(sx + sy + sz) >> 1) - 3 * (long long)mid.c;
  u64 N = 0;
  int sh = 0;
  unsigned tq = 1;
  if (!LIN) {
    const long long a[3] = {(long long)(sx - sy), (long long)(sx - sz), (long long)(sy - sz)};
    const long long cc[3] = {(long long)((v(kTileRow + 1) + v(-kTileRow - 1)) -
                                         (v(-kTileRow + 1) + v(kTileRow - 1))),
                             (long long)(up.dx - lo.dx), (long long)(up.dy - lo.dy)};
    N = fix_quad(a, cc, sh, tq);
  }
  const unsigned ls = (unsigned)(fix_hi(lap) >> 31);
  const u64 lm = ((u64)lap ^ fix_words(ls, ls)) - fix_words(ls, ls);
  bool bad = min((unsigned)(lm >> 32), tq) == 0 ||
             (tile_mag((long long)mid.c) < kTileSmallCentre && tq < 8 * kTileSmallDefect &&
              tile_small(q, 0, -1, 1, kTileSmallDefect));
  double D = src;
  qd = 1.0;
  if (!LIN) {
    qd = fma(c.e1, fix_double_top(N, 64 - 2 * sh + 2 * ue), src);
    bad = bad || !fix_normal(qd);
    D = fma(c.k2s, sqrt_fix_normal(qd), -c.k2);
  }
  d = fma(fix_double_top(lm, ue + 1, ls & 0x80000000u), c.inv_h2, -D);
  return !bad;
}

// The defect kernels, 512^3: residual 13.1 -> 1.69 ms, residual with restriction 10.5 ->
// 2.21 ms, hand-off to FP32 10.5 -> 2.10 ms (256^3 residual 1646 -> 234 us).  Per cell three
// to five FP64 instructions remain (the FP64 pipe is about half busy) beside some 430 others,
// two thirds of the issue slots.  Four CTAs per SM at 64 registers against three at 80 (when
// chosen): residual 1.65 against 1.80 ms, hand-off 3.11 against 3.28 ms; the restriction, which
// keeps two columns at once, is fastest at two.
//
// Of the cells that need another path each lane takes the next of its own: a warp then
// evaluates as many as its worst lane has, not one for every place where some lane has one
// (512^3: restriction 2.70 -> 2.34 ms, 128^3: 60 -> 51 us; colour stages 571 -> 566 us).
//
// Visit every cell of the tile at (x0, y0, z0): cell(id, i, j, k, defect, q, guard) with
// src(id) its source term.  A thread takes two columns of eight cells, side by side in y,
// the cells that need another path last.  In a tile of zeros (a solve that starts from 0;
// a floored cell then has q = 0) the stencil's sums are 0 and only the root is left: mixed
// solves from 0, 512^3 403.3 -> 399.6 ms, 64 of 32^3 to 128^3 4 % faster.
template <bool LIN, typename Src, typename Cell>
__device__ __forceinline__ void tile_defects(int n, const double* __restrict__ phi,
                                             const OpConst64& c, int x0, int y0, int z0,
                                             TileShared& S, Src src, Cell cell) {
  int ue;
  const int ok = tile_load_all(n, phi, x0, y0, z0, S, ue);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = x0 + lane, j0 = y0 + 2 * w, n2 = n * n;
  if (i >= n || j0 >= n) return;  // n is even
  unsigned rare = 0xffff;
  if (ok == 1) {
    rare = 0;
#pragma unroll 1
    for (int y = 0; y < 2; ++y) {
      const long long* q = S.v + kTilePlane + (2 * w + y + 1) * kTileRow + lane + 1;
      TilePlane lo = tile_plane(q - kTilePlane), mid = tile_plane(q);
      int id = z0 * n2 + (j0 + y) * n + i;
#pragma unroll 1
      for (int s = 0; s < kTileZ && z0 + s < n; ++s, id += n2, q += kTilePlane) {
        const TilePlane up = tile_plane(q + kTilePlane);
        double d, qd;
        const bool good = tile_defect<LIN>(q, lo, mid, up, ue, src(id), c, d, qd);
        lo = mid;
        mid = up;
        if (good)
          cell(id, i, j0 + y, z0 + s, d, qd, false);
        else
          rare |= 1u << (8 * y + s);
      }
    }
  }
#pragma unroll 1
  for (; rare != 0; rare &= rare - 1) {
    const int s = __ffs((int)rare) - 1;
    const int j = j0 + (s >> 3), k = z0 + (s & 7);
    if (k >= n) continue;
    const int id = k * n2 + j * n + i;
    double qd, d;
    bool g;
    if (ok == 2)
      d = fma(0.0, c.inv_h2, -root_of_M<LIN ? OP_LINEAR : OP_SQRT>(0.0, src(id), c, qd, g));
    else
      d = cell_defect_fix64<LIN ? OP_LINEAR : OP_SQRT>(phi, n, i, j, k, id, src(id), c, qd, g);
    cell(id, i, j, k, d, qd, g);
  }
}

// block_reduce of the 256 threads, in the tile's own memory.
__device__ __forceinline__ Partial tile_reduce(Partial p, TileShared& S) {
  Partial* sh = reinterpret_cast<Partial*>(S.v);
  p = warp_reduce(p);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = p;
  __syncthreads();
  if (threadIdx.x < 32) {
    Partial q;
    partial_init(q);
    if (threadIdx.x < 8) q = sh[threadIdx.x];
    p = warp_reduce(q);
  }
  return p;
}

template <bool LIN>
static __device__ __noinline__ double tile_defect_rare(const double* phi, int n, int i, int j,
                                                       int k, double src, const OpConst64* c,
                                                       bool* g) {
  double q;
  return cell_defect_fix64<LIN ? OP_LINEAR : OP_SQRT>(phi, n, i, j, k, lidx(i, j, k, n), src, *c, q, *g);
}

// Residual restriction of a tile (b_residual_restrict64).  A thread takes a column of 2 x 1
// fine cells in y and x, two planes at a time, and shares a coarse cell with its neighbour
// lane in x.  R phi is the exact sum of the eight children, rounded once, where that is not
// small against the tile.  Returns the tile's partial (thread 0).
template <bool F, bool LIN>
__device__ __forceinline__ Partial b_residual_restrict_tile64(
    int nf, const double* __restrict__ phi, const double* __restrict__ src,
    const double* __restrict__ f, const OpConst64& c, double* __restrict__ phi_c,
    double* __restrict__ phihat_c, double* __restrict__ rd_c, int x0, int y0, int z0,
    TileShared& S) {
  int ue;
  const bool ok = tile_load_all(nf, phi, x0, y0, z0, S, ue);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = x0 + lane, j0 = y0 + 2 * w, n2 = nf * nf, nc = nf >> 1;
  const bool in = i < nf && j0 < nf;  // nf is even: whole coarse cells
  Partial p;
  partial_init(p);
  double sum = 0.0;
  long long kmax = order_key(-INFINITY), kmin = order_key(INFINITY);
  const long long* q[2];
  TilePlane lo[2], mid[2];
#pragma unroll
  for (int y = 0; y < 2; ++y) {
    q[y] = S.v + kTilePlane + (2 * w + y + 1) * kTileRow + lane + 1;
    lo[y] = tile_plane(q[y] - kTilePlane);
    mid[y] = tile_plane(q[y]);
  }
#pragma unroll 1
  for (int k0 = z0; k0 < z0 + kTileZ && k0 < nf; k0 += 2) {
    double sd = 0.0;
    unsigned long long sphi = 0;
    if (in) {
      auto place = [&](int ch) { return (k0 + (ch >> 1)) * n2 + (j0 + (ch & 1)) * nf + i; };
      double dv[4];
      unsigned rare = 0xf;
      if (ok) {
        rare = 0;
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
          const int y = ch & 1;
          double qd;
          const TilePlane up = tile_plane(q[y] + kTilePlane);
          if (!tile_defect<LIN>(q[y], lo[y], mid[y], up, ue, src[place(ch)], c, dv[ch], qd))
            rare |= 1u << ch;
          sphi += mid[y].c;
          lo[y] = mid[y];
          mid[y] = up;
          q[y] += kTilePlane;
        }
      }
#pragma unroll 1
      for (; rare != 0; rare &= rare - 1) {  // as in tile_defects
        const int r = __ffs((int)rare) - 1;
        bool g;
        const double d = tile_defect_rare<LIN>(phi, nf, i, j0 + (r & 1), k0 + (r >> 1),
                                               src[place(r)], &c, &g);
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) dv[ch] = ch == r ? d : dv[ch];
        p.guards += g ? 1 : 0;
      }
#pragma unroll
      for (int ch = 0; ch < 4; ++ch) {
        const double d = F ? dv[ch] - f[place(ch)] : dv[ch];
        const bool fin = finite_bits(d);
        const long long key = order_key(d);
        kmax = (fin && key > kmax) ? key : kmax;
        kmin = (fin && key < kmin) ? key : kmin;
        p.nonfinite += fin ? 0 : 1;
        sd += d;
      }
    }
    // with a non-finite defect the level has no residual, and its sum no use
    if (p.nonfinite == 0) sum += sd;
    const double sd2 = sd + __shfl_xor_sync(0xffffffffu, sd, 1);
    const unsigned long long sp2 = sphi + __shfl_xor_sync(0xffffffffu, sphi, 1);
    if (in && (lane & 1) == 0) {
      const int cid = (k0 >> 1) * nc * nc + (j0 >> 1) * nc + (i >> 1);
      const int h = (int)(sp2 >> 32);
      double r;
      if (ok && (unsigned)(h ^ (h >> 31)) >= (1u << 24)) {
        r = fix_signed((long long)sp2, FixRef{0, ue - 3, false});
      } else {
        r = 0.0;
#pragma unroll 1
        for (int ch = 0; ch < 8; ++ch)
          r += phi[(k0 + (ch >> 2)) * n2 + (j0 + ((ch >> 1) & 1)) * nf + i + (ch & 1)];
        r *= 0.125;
      }
      phi_c[cid] = r;
      phihat_c[cid] = r;
      rd_c[cid] = sd2 * 0.125;
    }
  }
  p.sum = sum;
  if (kmax >= kmin) {
    p.dmax = from_order_key(kmax);
    p.dmin = from_order_key(kmin);
  }
  return tile_reduce(p, S);
}

// The FAS right-hand side of a tile (cell_fas_rhs64).
template <bool LIN>
__device__ __forceinline__ void b_fas_rhs_tile64(int nc, const double* __restrict__ phi_c,
                                                 const double* __restrict__ src_c,
                                                 double* __restrict__ f_c, const OpConst64& c,
                                                 const LevelScalars* __restrict__ fine_sc,
                                                 LevelScalars* __restrict__ coarse_sc, int x0,
                                                 int y0, int z0, TileShared& S) {
  if ((x0 | y0 | z0) == 0 && threadIdx.x == 0) coarse_sc->lambda = 0.0;
  const double lam = fine_sc->lambda;
  tile_defects<LIN>(
      nc, phi_c, c, x0, y0, z0, S, [&](int id) { return src_c[id]; },
      [&](int id, int, int, int, double L, double, bool) { f_c[id] = L - f_c[id] + lam; });
}

}  // namespace mg
