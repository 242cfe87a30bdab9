// Shared-memory tiles of refinement patches: the ghosted (B+2)^3 block of one
// patch with its neighbours' cells and the Dirichlet values outside the union.
// Used by the patch kernels (mg_patch.cu) and the union's linear coarse-grid
// correction (mg_patch_galerkin.cu).
#pragma once

#include "mg_common.cuh"
#include "mg_tile64.cuh"

namespace mg {

// Load the ghosted tile of patch p at block size B into shared memory.
template <int B>
__device__ __forceinline__ void load_tile(double* __restrict__ tile, int p,
                                          const double* __restrict__ phi,
                                          const double* __restrict__ ghost,
                                          const int* __restrict__ nbr) {
  constexpr int T = B + 2, TC = T * T * T, BC = B * B * B;
  for (int q = threadIdx.x; q < TC; q += blockDim.x) {
    const int i = q % T - 1, j = (q / T) % T - 1, k = q / (T * T) - 1;
    const int ox = i < 0 ? -1 : (i >= B ? 1 : 0);
    const int oy = j < 0 ? -1 : (j >= B ? 1 : 0);
    const int oz = k < 0 ? -1 : (k >= B ? 1 : 0);
    double v;
    if ((ox | oy | oz) == 0) {
      v = phi[(long long)p * BC + i + B * (j + B * k)];
    } else {
      const int nb = nbr[p * 27 + (ox + 1) + 3 * ((oy + 1) + 3 * (oz + 1))];
      if (nb >= 0)
        v = phi[(long long)nb * BC + (i - ox * B) + B * ((j - oy * B) + B * (k - oz * B))];
      else
        v = ghost[(long long)p * TC + q];
    }
    tile[q] = v;
  }
}

template <int B>
__device__ __forceinline__ StencilT<double> gather_tile(const double* tile, int i, int j, int k) {
  constexpr int T = B + 2;
  auto at = [&](int a, int b, int c) { return tile[(a + 1) + T * ((b + 1) + T * (c + 1))]; };
  StencilT<double> s;
  s.sx = at(i + 1, j, k) + at(i - 1, j, k);
  s.sy = at(i, j + 1, k) + at(i, j - 1, k);
  s.sz = at(i, j, k + 1) + at(i, j, k - 1);
  s.cxy = (at(i + 1, j + 1, k) + at(i - 1, j - 1, k)) - (at(i + 1, j - 1, k) + at(i - 1, j + 1, k));
  s.cxz = (at(i + 1, j, k + 1) + at(i - 1, j, k - 1)) - (at(i + 1, j, k - 1) + at(i - 1, j, k + 1));
  s.cyz = (at(i, j + 1, k + 1) + at(i, j - 1, k - 1)) - (at(i, j + 1, k - 1) + at(i, j - 1, k + 1));
  return s;
}

template <int B>
__device__ __forceinline__ double tile_ctr(const double* tile, int i, int j, int k) {
  constexpr int T = B + 2;
  return tile[(i + 1) + T * ((j + 1) + T * (k + 1))];
}

// Where each of the 1000 cells of a ghosted 8^3 block comes from: neighbour slot (13: the
// patch itself) x 512 + place in it, and its colour in the two bits above.
struct PatchSource {
  unsigned short v[1000];
};
constexpr PatchSource patch_source() {
  PatchSource s{};
  for (int q = 0; q < 1000; ++q) {
    const int c[3] = {q % 10 - 1, q / 10 % 10 - 1, q / 100 - 1};
    int slot = 0, at = 0;
    for (int a = 2; a >= 0; --a) {
      const int o = c[a] < 0 ? 0 : (c[a] > 7 ? 2 : 1);
      slot = 3 * slot + o;
      at = 8 * at + (c[a] & 7);
    }
    const int colour = ((c[0] + c[2]) & 1) + 2 * ((c[1] + c[2]) & 1);
    s.v[q] = (unsigned short)(colour << 14 | slot << 9 | at);
  }
  return s;
}
static __device__ const PatchSource k_patch_source = patch_source();

// The ghosted 8^3 block of a patch as integers of one unit (128 threads).
struct PatchTile {
  long long v[1000];
  int nbr[27];
  int em[4];
};

__device__ __forceinline__ double patch_value(const double* __restrict__ phi,
                                              const double* __restrict__ ghost, int p, int q,
                                              unsigned e, const int* nbr) {
  const int slot = (int)(e >> 9) & 31, nb = slot == 13 ? p : nbr[slot];
  return nb >= 0 ? phi[(long long)nb * 512 + (e & 511)] : ghost[(long long)p * 1000 + q];
}

// colour >= 0: without that colour's cells, which the launch is writing.  False (for every
// thread): no unit (tile_exponent).
__device__ __forceinline__ bool patch_load(int p, const double* __restrict__ phi,
                                           const double* __restrict__ ghost,
                                           const int* __restrict__ nbr, int colour, PatchTile& S,
                                           int& ue) {
  if (threadIdx.x < 27) S.nbr[threadIdx.x] = nbr[p * 27 + threadIdx.x];
  __syncthreads();
  long long v[8];
  float fm = 0.f;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int q = threadIdx.x + 128 * r;
    v[r] = 0;
    if (q < 1000) {
      const unsigned e = k_patch_source.v[q];
      if ((int)(e >> 14) != colour)
        v[r] = __double_as_longlong(patch_value(phi, ghost, p, q, e, S.nbr));
    }
    fm = tile_max(fm, v[r]);
  }
  int em = __reduce_max_sync(0xffffffffu, __float_as_int(fm) & 0x7fffffff);
  if ((threadIdx.x & 31) == 0) S.em[threadIdx.x >> 5] = em;
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 4; ++k) em = max(em, S.em[k]);
  if (em < (kFixMinExp << 20) || em >= ((kFixMaxExp + 1) << 20)) {
    long long any = em;
#pragma unroll
    for (int r = 0; r < 8; ++r) any |= v[r] << 1;
    if (__syncthreads_or(any != 0)) return false;
    em = 1023 << 20;
  }
  em &= 0x7ff00000;
  ue = (em >> 20) - 1082;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    const int q = threadIdx.x + 128 * r;
    if (q < 1000) S.v[q] = tile_convert(v[r], em);
  }
  __syncthreads();
  return true;
}

// The sums of the cell at q of the block: face sum, the form N 2^(64 - 2 sh) (0 with LIN)
// and a bound of its terms.  False: the block's unit does not resolve the stencil as FP64
// would (`bound`: kTileSmall or kTileSmallDefect).
template <bool LIN>
__device__ __forceinline__ bool patch_forms(const long long* q, unsigned bound, long long& face,
                                            unsigned long long& N, int& sh, unsigned& tq) {
  typedef unsigned long long u64;
  constexpr int Y = 10, Z = 100;
  auto v = [&](int o) { return (u64)q[o]; };
  const u64 sx = v(1) + v(-1), sy = v(Y) + v(-Y), sz = v(Z) + v(-Z);
  face = (long long)(sx + sy + sz);
  N = 0;
  sh = 0;
  tq = 1;
  if (!LIN) {
    const long long a[3] = {(long long)(sx - sy), (long long)(sx - sz), (long long)(sy - sz)};
    const long long c[3] = {
        (long long)((v(1 + Y) + v(-1 - Y)) - (v(1 - Y) + v(-1 + Y))),
        (long long)((v(1 + Z) + v(-1 - Z)) - (v(1 - Z) + v(-1 + Z))),
        (long long)((v(Y + Z) + v(-Y - Z)) - (v(Y - Z) + v(-Y + Z)))};
    N = fix_quad(a, c, sh, tq);
  }
  if (tq == 0) return false;
  if ((tile_mag(face) | tq) >= 8 * bound) return true;
  return (tile_mag(q[1]) | tile_mag(q[-1]) | tile_mag(q[Y]) | tile_mag(q[-Y]) | tile_mag(q[Z]) |
          tile_mag(q[-Z])) >= bound;
}

// The stencil of the cell at place q of the ghosted block in FP64, from memory.
static __device__ __noinline__ StencilT<double> patch_stencil64(const double* phi,
                                                                const double* ghost, int p, int q,
                                                                const int* nbr) {
  auto at = [&](int o) {
    return patch_value(phi, ghost, p, q + o, k_patch_source.v[q + o], nbr);
  };
  constexpr int Y = 10, Z = 100;
  StencilT<double> s;
  s.sx = at(1) + at(-1);
  s.sy = at(Y) + at(-Y);
  s.sz = at(Z) + at(-Z);
  s.cxy = (at(1 + Y) + at(-1 - Y)) - (at(1 - Y) + at(-1 + Y));
  s.cxz = (at(1 + Z) + at(-1 - Z)) - (at(1 - Z) + at(-1 + Z));
  s.cyz = (at(Y + Z) + at(-Y - Z)) - (at(Y - Z) + at(-Y + Z));
  return s;
}

}  // namespace mg
