// FP64 kernels of the periodic FAS V-cycle (Sec. III.B and III.C of
// arXiv:1303.0008): four-colour Newton-Gauss-Seidel sweep, residual with its
// norms, residual evaluation fused with full-weighting restriction, the coarse
// FAS right-hand side, trilinear prolongation of the correction, the coarsest
// solve in one CTA, density restriction, gauge fix and the force output.
//
// Every kernel works on dense n^3 arrays, x fastest (idx = i + n(j + n k)), with
// periodic wrap.  In FP64 they would be bound by GB300's narrow FP64 pipe (about 35-45
// FP64 operations per cell against 24 bytes of traffic); the colour stages therefore do
// the same arithmetic in integers (mg_fix64.cuh), the large levels in tiles
// (mg_tile64.cuh), and the others favour a low FP64 instruction count.
#include "mg_common.cuh"
#include "mg_internal.h"
#include "mg_bodies64.cuh"
#include "mg_tile64.cuh"

namespace mg {

// ---------------------------------------------------------------------------
// Four-colour Gauss-Seidel: colour c = ((i+k)&1) + 2((j+k)&1).  No face or edge
// neighbour of a cell shares its colour (only the corners do, and they are not
// in the 19-point stencil), so the cells of one colour update independently
// and each update is the exact Newton step of Sec. III.B.
// ---------------------------------------------------------------------------
// A warp takes a block of 8 x 2 x 2 of the colour's cells (x, y, z), a CTA warps / 2 of
// them along x on each of two pairs of planes: a compact block mostly lies in one binade
// of the field, which is the cheapest path of fix_align.  One kernel per mode (by_mode), here
// and below: with all of them in one, the linear and the general form (40 and 32 registers)
// carried the integer form's 80, and its code ran longer by the others' branches (FP64 solves
// of 32^3 2.86 -> 2.73 ms, 64^3 4.60 -> 4.37, 128^3 8.31 -> 8.04).
template <int MODE>
__global__ void __launch_bounds__(256) k_smooth_colour64(int n, double* __restrict__ phi,
                                                         const double* __restrict__ src,
                                                         const double* __restrict__ f,
                                                         const LevelScalars* __restrict__ sc,
                                                         OpConst64 c, int colour) {
  PdlScope pdl_scope;
  __shared__ double s_c;
  if (threadIdx.x == 0) s_c = smooth_scalar64(sc, c);
  __syncthreads();
  const int hn = n >> 1;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int m = ((int)blockIdx.x * (int)(blockDim.x >> 6) + (w >> 1)) * 8 + (lane & 7);
  const int jj = (int)blockIdx.y * 2 + ((lane >> 3) & 1);
  const int k = (int)blockIdx.z * 4 + (w & 1) * 2 + (lane >> 4);
  if (m >= hn || jj >= hn || k >= n) return;
  cell_smooth64_at<MODE>(n, phi, src, f, s_c, c, 2 * m + ((colour ^ k) & 1),
                   2 * jj + (((colour >> 1) ^ k) & 1), k);
}

// The same for levels of many tiles.
template <bool F, bool LIN>
__global__ void __launch_bounds__(256, 4) k_smooth_tile64(int n, double* __restrict__ phi,
                                                          const double* __restrict__ src,
                                                          const double* __restrict__ f,
                                                          const LevelScalars* __restrict__ sc,
                                                          OpConst64 c, int colour) {
  PdlScope pdl_scope;
  __shared__ TileShared S;
  b_smooth_tile64<F, LIN>(n, phi, src, f, sc, c, colour, (int)blockIdx.x * kTileX,
                          (int)blockIdx.y * kTileY, (int)blockIdx.z * kTileZ, S);
}

// d = L^h phi - f with block partial norms.
template <int MODE>
__global__ void __launch_bounds__(256) k_residual64(int n, const double* __restrict__ phi,
                                                    const double* __restrict__ src,
                                                    const double* __restrict__ f,
                                                    double* __restrict__ dout, OpConst64 c,
                                                    Partial* __restrict__ partials) {
  PdlScope pdl_scope;
  const long long cells = (long long)n * n * n;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  Partial p;
  partial_init(p);
  if (t < cells) {
    int i, j, k;
    split3((unsigned)t, n, i, j, k);
    bool g;
    double ctr;
    const double d = fine_defect64<MODE>(n, phi, src, f, c, i, j, k, t, ctr, g);
    if (dout) dout[t] = d;
    partial_add(p, d, g);
  }
  p = block_reduce(p);
  if (threadIdx.x == 0) partials[blockIdx.x] = p;
}

// The same for levels of many tiles, one partial per tile.
template <bool LIN>
__global__ void __launch_bounds__(256, 4) k_residual_tile64(int n, const double* __restrict__ phi,
                                                            const double* __restrict__ src,
                                                            const double* __restrict__ f,
                                                            double* __restrict__ dout,
                                                            OpConst64 c,
                                                            Partial* __restrict__ partials) {
  PdlScope pdl_scope;
  __shared__ TileShared S;
  Partial p;
  partial_init(p);
  tile_defects<LIN>(
      n, phi, c, (int)blockIdx.x * kTileX, (int)blockIdx.y * kTileY, (int)blockIdx.z * kTileZ, S,
      [&](int id) { return src[id]; },
      [&](int id, int, int, int, double d, double, bool g) {
        if (f) d -= f[id];
        if (dout) dout[id] = d;
        partial_add(p, d, g);
      });
  p = tile_reduce(p, S);
  if (threadIdx.x == 0) partials[tile_index()] = p;
}

// Residual of the 8 children of each coarse cell, averaged (full weighting),
// together with R phi; the partial norms cover every fine cell.
template <int MODE>
__global__ void __launch_bounds__(256) k_residual_restrict64(
    int nf, const double* __restrict__ phi, const double* __restrict__ src,
    const double* __restrict__ f, OpConst64 c, double* __restrict__ phi_c,
    double* __restrict__ phihat_c, double* __restrict__ rd_c, Partial* __restrict__ partials) {
  PdlScope pdl_scope;
  b_residual_restrict64<MODE>(nf, phi, src, f, c, phi_c, phihat_c, rd_c, partials, blockIdx.x);
}

// The same for levels of many tiles, one partial per tile.
template <bool F, bool LIN>
__global__ void __launch_bounds__(256, 2) k_residual_restrict_tile64(
    int nf, const double* __restrict__ phi, const double* __restrict__ src,
    const double* __restrict__ f, OpConst64 c, double* __restrict__ phi_c,
    double* __restrict__ phihat_c, double* __restrict__ rd_c, Partial* __restrict__ partials) {
  PdlScope pdl_scope;
  __shared__ TileShared S;
  const Partial p = b_residual_restrict_tile64<F, LIN>(nf, phi, src, f, c, phi_c, phihat_c, rd_c,
                                                  (int)blockIdx.x * kTileX,
                                                  (int)blockIdx.y * kTileY,
                                                  (int)blockIdx.z * kTileZ, S);
  if (threadIdx.x == 0) partials[tile_index()] = p;
}

// The same residual restriction in two launches, for levels whose coarse cells
// fill only a few 256-thread blocks: per fine cell the defect and guard flag
// (blocks of any size), then the walk over each coarse cell's children in the
// order and 256-thread partition of k_residual_restrict64 (the same bits).
template <int MODE>
__global__ void __launch_bounds__(256) k_defect64(int nf, const double* __restrict__ phi,
                                                  const double* __restrict__ src,
                                                  const double* __restrict__ f, OpConst64 c,
                                                  double* __restrict__ dout,
                                                  unsigned char* __restrict__ gout) {
  PdlScope pdl_scope;
  cell_defect64<MODE>(nf, phi, src, f, c, dout, gout, (long long)blockIdx.x * blockDim.x + threadIdx.x);
}

__global__ void __launch_bounds__(256) k_restrict_defects64(
    int nf, const double* __restrict__ phi, const double* __restrict__ din,
    const unsigned char* __restrict__ gin, double* __restrict__ phi_c,
    double* __restrict__ phihat_c, double* __restrict__ rd_c, Partial* __restrict__ partials) {
  PdlScope pdl_scope;
  b_restrict_defects64(nf, phi, din, gin, phi_c, phihat_c, rd_c, partials, blockIdx.x);
}

// The prolongation of a large level by columns (prolong_column).
template <int KZ>
__global__ void __launch_bounds__(256) k_prolong_column64(int nc, const double* __restrict__ phi_c,
                                                          const double* __restrict__ phihat_c,
                                                          double* __restrict__ phi_f) {
  PdlScope pdl_scope;
  prolong_column<double, double2, KZ>(nc, phi_c, phihat_c, phi_f, (int)blockIdx.x,
                                      (int)blockIdx.y, (int)blockIdx.z);
}

// One block: reduce the partials in a fixed order and publish the scalars.
__global__ void __launch_bounds__(1024) k_finalize(const Partial* __restrict__ partials, int nparts,
                                                  double cells, int periodic,
                                                  LevelScalars* __restrict__ sc) {
  PdlScope pdl_scope;
  b_finalize(partials, nparts, cells, periodic, sc, blockIdx.x);
}

// f^H = L^H(R phi) - (R d - lambda^h); lambda^H starts at 0.
template <int MODE>
__global__ void __launch_bounds__(256) k_fas_rhs64(int nc, const double* __restrict__ phi_c,
                                                   const double* __restrict__ src_c,
                                                   double* __restrict__ f_c, OpConst64 c,
                                                   const LevelScalars* __restrict__ fine_sc,
                                                   LevelScalars* __restrict__ coarse_sc) {
  PdlScope pdl_scope;
  b_fas_rhs64<MODE>(nc, phi_c, src_c, f_c, c, fine_sc, coarse_sc, blockIdx.x);
}

// The same for levels of many tiles.
template <bool LIN>
__global__ void __launch_bounds__(256, 4) k_fas_rhs_tile64(int nc, const double* __restrict__ phi_c,
                                                           const double* __restrict__ src_c,
                                                           double* __restrict__ f_c, OpConst64 c,
                                                           const LevelScalars* __restrict__ fine_sc,
                                                           LevelScalars* __restrict__ coarse_sc) {
  PdlScope pdl_scope;
  __shared__ TileShared S;
  b_fas_rhs_tile64<LIN>(nc, phi_c, src_c, f_c, c, fine_sc, coarse_sc, (int)blockIdx.x * kTileX,
                   (int)blockIdx.y * kTileY, (int)blockIdx.z * kTileZ, S);
}

// phi^h += P(phi^H - R phi^h): cell-centred trilinear, per axis 3/4 on the parent
// and 1/4 on the parent's neighbour on the child's side.
__global__ void __launch_bounds__(256) k_prolong_correct64(int nc, const double* __restrict__ phi_c,
                                                           const double* __restrict__ phihat_c,
                                                           double* __restrict__ phi_f) {
  PdlScope pdl_scope;
  b_prolong_correct64(nc, phi_c, phihat_c, phi_f, blockIdx.x);
}

// Coarsest level in one CTA (n^3 <= 4096 cells in shared memory): four-colour
// sweeps until max|d - lambda| has fallen by `drop` or `max_sweeps` sweeps.
__global__ void __launch_bounds__(256) k_coarsest64(int n, double* __restrict__ phi,
                                                    const double* __restrict__ src,
                                                    const double* __restrict__ f, OpConst64 c,
                                                    LevelScalars* __restrict__ sc, int max_sweeps,
                                                    double drop, int check_every) {
  PdlScope pdl_scope;
  b_coarsest64(n, phi, src, f, c, sc, max_sweeps, drop, check_every, blockIdx.x);
}

// coarse = mean of the 8 children.
__global__ void __launch_bounds__(256) k_restrict64(int nc, const double* __restrict__ fine,
                                                    double* __restrict__ coarse) {
  PdlScope pdl_scope;
  const int nf = nc << 1;
  const long long cells = (long long)nc * nc * nc;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= cells) return;
  const int I = (int)(t % nc);
  const int J = (int)((t / nc) % nc);
  const int K = (int)(t / ((long long)nc * nc));
  double s = 0.0;
#pragma unroll
  for (int ch = 0; ch < 8; ++ch)
    s += fine[lidx(2 * I + (ch & 1), 2 * J + ((ch >> 1) & 1), 2 * K + (ch >> 2), nf)];
  coarse[t] = s * 0.125;
}

// src = a * delta + b, optionally held where 1 + c3 kappa delta < 0 (the bound under
// which the root of Eq. two_branch stays real for any field): in the sqrt form
// (b = 1) src >= 0, in the kappa*delta form c3 * src >= -1.  Floored cells are
// counted into *floored.
__global__ void __launch_bounds__(256) k_affine64(long long cells, const double* __restrict__ delta,
                                                  double* __restrict__ out, double a, double b,
                                                  double c3, int floor,
                                                  unsigned long long* __restrict__ floored) {
  PdlScope pdl_scope;
  b_affine64(cells, delta, out, a, b, c3, floor, floored, blockIdx.x);
}

// Partial sums of x (for the gauge fix).
__global__ void __launch_bounds__(256) k_sum_partials(long long cells, const double* __restrict__ x,
                                                      Partial* __restrict__ partials) {
  PdlScope pdl_scope;
  b_sum_partials(cells, x, partials, blockIdx.x);
}

// x -= mean (the mean sits in sc->lambda, computed by k_finalize).
__global__ void __launch_bounds__(256) k_sub_mean(long long cells, double* __restrict__ x,
                                                  const LevelScalars* __restrict__ sc) {
  PdlScope pdl_scope;
  b_sub_mean(cells, x, sc, blockIdx.x);
}

// x -2^k by the exponent, on the integer pipe (its FP64 product where that is not a normal
// number).
static __device__ __noinline__ double scale_rare(double x, int k) { return -scalbn(x, k); }
__device__ __forceinline__ double neg_scale(double x, int k) {
  const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
  if (e == 0 || e + k < 1 || e + k > 2046) return scale_rare(x, k);
  return __hiloint2double((hi + (k << 20)) ^ 0x80000000, __double2loint(x));
}

// g = -(1/2) grad phi, central differences; out is 3 x n^3 (x, y, z).  The factor
// -(1/2) / (2h) = -n/4; log2n: of a power of two n, else -1.  512^3: 2060 -> 791 us with
// the three products taken off the FP64 pipe, which bounded it; the three differences and
// the 4.3 GB moved now take about the same.
__global__ void __launch_bounds__(256) k_force64(int n, int log2n, const double* __restrict__ phi,
                                                 double* __restrict__ out) {
  PdlScope pdl_scope;
  const long long cells = (long long)n * n * n;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= cells) return;
  int i, j, k;
  split3((unsigned)t, n, i, j, k);
  const NbrOff o = nbr_offsets(i, j, k, n);
  const double* c = phi + t;
  const double d[3] = {c[o.xp] - c[o.xm], c[o.yp] - c[o.ym], c[o.zp] - c[o.zm]};
  const double sc = -0.25 * (double)n;
#pragma unroll
  for (int a = 0; a < 3; ++a)
    out[a * cells + t] = log2n >= 0 ? neg_scale(d[a], log2n - 2) : sc * d[a];
}

// ---------------------------------------------------------------------------
// Host launchers
// ---------------------------------------------------------------------------
static inline unsigned blocks_for(long long work, int threads) {
  return (unsigned)((work + threads - 1) / threads);
}

OpConst64 make_op64(int n, double alpha, double kappa, int branch, double w) {
  OpConst64 c{};
  const double h = 1.0 / (double)n;
  c.h2 = h * h;
  c.inv_h2 = (double)n * (double)n;
  c.h2_6 = c.h2 / 6.0;
  c.omega = 1.0;
  const double h4 = c.h2 * c.h2;
  c.c3 = 4.0 * (1.0 - w) * alpha;
  if (alpha == 0.0) {
    c.mode = OP_LINEAR;
    return c;
  }
  const double sigma = (branch == 0) ? 1.0 : ((branch > 0) == (alpha > 0) ? 1.0 : -1.0);
  c.k2 = 2.0 / c.c3;
  c.k2s = sigma * c.k2;
  c.c1 = alpha / (3.0 * h4);
  c.c2 = alpha / (8.0 * h4);
  c.e1 = c.c3 * c.c1;
  c.e2 = c.c3 * c.c2;
  c.e1h = 2.0 * c.e1;
  c.c1h = 2.0 * c.c1;
  c.upd_s = -c.h2 * c.k2s / 6.0;
  // k2 (sigma sqrt(q) - 1) loses about |k2| * eps to cancellation on the physical
  // root; below |alpha| = 1e-4 the conjugate form 2u/(1+sqrt q) is used instead.
  c.mode = (sigma > 0 && fabs(alpha) < 1e-4) ? OP_CONJ : OP_SQRT;
  if (w != 1.0 / 3.0) {
    // Sec. III.B with a general splitting constant: q = src + c3 alpha Sigma_ijk
    c.mode = OP_GENW;
    c.gA = c.c3 * alpha * (1.0 - w) / h4;
    c.gB = -2.0 * c.c3 * alpha * w / h4;
    c.gC = c.c3 * alpha / (8.0 * h4);
    c.gAB = c.gA + c.gB;
  }
  return c;
}

void src_coefficients(const OpConst64& c, double kappa, double* a, double* b) {
  if (c.mode == OP_SQRT || c.mode == OP_GENW) {
    *a = c.c3 * kappa;
    *b = 1.0;
  } else {
    *a = kappa;
    *b = 0.0;
  }
}

thread_local long long tl_launches = 0;

// Threads per block of a per-cell FP64 launch: 256, or 64 where 256-thread
// blocks would not give every SM two blocks.  An SM retires only two FP64
// lane-operations per clock, so on small levels the launch time is set by how
// many SMs the cells reach.  Per-cell results do not depend on the partition.
int tpb_for(long long items) {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0, v = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    sms = v > 0 ? v : 1;
  }
  return (long long)blocks_for(items, 256) < 2LL * sms ? 64 : 256;
}

// 1024 threads (as the batch's) where there are partials for them; the order of the sums is
// the same with fewer.
void launch_finalize(cudaStream_t st, const Partial* partials, int nparts, double cells,
                     int periodic, LevelScalars* sc) {
  launch_k(k_finalize, 1, nparts > 256 ? 1024 : 256, 0, st, partials, nparts, cells, periodic, sc);
  count_launches(1);
}

void launch_smooth64(cudaStream_t st, int n, double* phi, const double* src, const double* f,
                     const LevelScalars* sc, const OpConst64& c, int sweeps, EventPairs* timer) {
  const int hn = n / 2;
  // A splitting constant of its own runs in FP64 with 32 registers, all CTAs at once: wide ones
  // that reach past the row leave some SMs idle warps only (96^3 solves 11.3 against 9.6 ms).
  const unsigned tpb = c.mode == OP_GENW && hn % 32 != 0
                           ? 64u
                           : (unsigned)tpb_for((long long)hn * hn * n);
  const unsigned bx = tpb / 8;  // cells of the colour along x per CTA
  const dim3 grid((hn + bx - 1) / bx, (hn + 1) / 2, (n + 3) / 4);
  const bool tiles = smooth_in_tiles(n, c), lin = c.mode == OP_LINEAR;
  auto tile_kernel = lin ? (f ? k_smooth_tile64<true, true> : k_smooth_tile64<false, true>)
                         : (f ? k_smooth_tile64<true, false> : k_smooth_tile64<false, false>);
  for (int s = 0; s < sweeps; ++s)
    for (int colour = 0; colour < 4; ++colour) {
      // an event between two launches removes their programmatic overlap, so the
      // sampled mode brackets one colour stage per call
      const bool timed = timer && (!timer->first_only || (s == 0 && colour == 0));
      if (timed) timer->begin(st);
      if (tiles)
        launch_k(tile_kernel, tile_grid(n), 256, 0, st, n, phi, src, f, sc, c, colour);
      else
        by_mode(c.mode, [&](auto m) {
          launch_k(k_smooth_colour64<m()>, grid, tpb, 0, st, n, phi, src, f, sc, c, colour);
        });
      if (timed) timer->end(st);
    }
  count_launches(4LL * sweeps);
}

int partials_needed(long long cells) { return (int)blocks_for(cells, 128) + 1; }

void launch_residual64(cudaStream_t st, int n, const double* phi, const double* src,
                       const double* f, double* dout, const OpConst64& c, Partial* partials,
                       LevelScalars* sc, int periodic) {
  const long long cells = (long long)n * n * n;
  const bool tiles = in_tiles(n, c);
  const unsigned nb = tiles ? tile_count(n) : blocks_for(cells, 256);
  if (tiles)
    launch_k(c.mode == OP_LINEAR ? k_residual_tile64<true> : k_residual_tile64<false>,
             tile_grid(n), 256, 0, st, n, phi, src, f, dout, c, partials);
  else
    by_mode(c.mode, [&](auto m) {
      launch_k(k_residual64<m()>, nb, 256, 0, st, n, phi, src, f, dout, c, partials);
    });
  launch_finalize(st, partials, (int)nb, (double)cells, periodic, sc);
  count_launches(1);
}

void launch_residual_restrict64(cudaStream_t st, int nf, const double* phi, const double* src,
                                const double* f, const OpConst64& c, double* phi_c,
                                double* phihat_c, double* rd_c, Partial* partials,
                                LevelScalars* sc, double* def, unsigned char* guard) {
  const long long fcells = (long long)nf * nf * nf;
  const long long ccells = fcells / 8;
  const bool tiles = in_tiles(nf, c);
  const unsigned nb = tiles ? tile_count(nf) : blocks_for(ccells, 256);
  if (tiles) {
    const bool lin = c.mode == OP_LINEAR;
    launch_k(lin ? (f ? k_residual_restrict_tile64<true, true>
                      : k_residual_restrict_tile64<false, true>)
                 : (f ? k_residual_restrict_tile64<true, false>
                      : k_residual_restrict_tile64<false, false>),
             tile_grid(nf), 256, 0, st, nf, phi, src, f, c, phi_c, phihat_c, rd_c, partials);
  } else if (def && guard && fcells <= kTwoStepMaxFine) {
    const int tpb = tpb_for(fcells);
    by_mode(c.mode, [&](auto m) {
      launch_k(k_defect64<m()>, blocks_for(fcells, tpb), tpb, 0, st, nf, phi, src, f, c, def,
               guard);
    });
    launch_k(k_restrict_defects64, nb, 256, 0, st, nf, phi, (const double*)def,
             (const unsigned char*)guard, phi_c, phihat_c, rd_c, partials);
    count_launches(1);
  } else {
    by_mode(c.mode, [&](auto m) {
      launch_k(k_residual_restrict64<m()>, nb, 256, 0, st, nf, phi, src, f, c, phi_c, phihat_c,
               rd_c, partials);
    });
  }
  launch_finalize(st, partials, (int)nb, (double)fcells, 1, sc);
  count_launches(1);
}

void launch_fas_rhs64(cudaStream_t st, int nc, const double* phi_c, const double* src_c,
                      double* f_c, const OpConst64& c, const LevelScalars* fine_sc,
                      LevelScalars* coarse_sc) {
  const long long cells = (long long)nc * nc * nc;
  const int tpb = tpb_for(cells);
  if (in_tiles(nc, c))
    launch_k(c.mode == OP_LINEAR ? k_fas_rhs_tile64<true> : k_fas_rhs_tile64<false>,
             tile_grid(nc), 256, 0, st, nc, phi_c, src_c, f_c, c, fine_sc, coarse_sc);
  else
    by_mode(c.mode, [&](auto m) {
      launch_k(k_fas_rhs64<m()>, blocks_for(cells, tpb), tpb, 0, st, nc, phi_c, src_c, f_c, c,
               fine_sc, coarse_sc);
    });
  count_launches(1);
}

// By columns where prolong_columns says so.  Their loads of pairs need a 16-byte aligned
// field.
void launch_prolong_correct64(cudaStream_t st, int nc, const double* phi_c,
                              const double* phihat_c, double* phi_f) {
  const long long cells = 8LL * nc * nc * nc;
  if (prolong_columns(nc) && reinterpret_cast<uintptr_t>(phi_f) % 16 == 0) {
    const int kz = prolong_depth(nc);
    launch_k(kz == 8 ? k_prolong_column64<8> : k_prolong_column64<4>, prolong_grid(nc, kz), 256, 0,
             st, nc, phi_c, phihat_c, phi_f);
  } else {
    const int tpb = tpb_for(cells);
    launch_k(k_prolong_correct64, blocks_for(cells, tpb), tpb, 0, st, nc, phi_c, phihat_c, phi_f);
  }
  count_launches(1);
}

void launch_coarsest64(cudaStream_t st, int n, double* phi, const double* src, const double* f,
                       const OpConst64& c, LevelScalars* sc, int max_sweeps, double drop) {
  const size_t smem = 3 * sizeof(double) * (size_t)n * n * n;
  static bool attr_set = false;
  if (!attr_set) {
    cudaFuncSetAttribute(k_coarsest64, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         3 * sizeof(double) * 4096);
    attr_set = true;
  }
  launch_k(k_coarsest64, 1, 256, smem, st, n, phi, src, f, c, sc, max_sweeps, drop, 2);
  count_launches(1);
}

void launch_restrict64(cudaStream_t st, int nc, const double* fine, double* coarse) {
  const long long cells = (long long)nc * nc * nc;
  launch_k(k_restrict64, blocks_for(cells, 256), 256, 0, st, nc, fine, coarse);
  count_launches(1);
}

void launch_affine64(cudaStream_t st, long long cells, const double* x, double* out, double a,
                     double b, double c3, int floor, unsigned long long* floored) {
  launch_k(k_affine64, blocks_for(cells, 256 * kAffineCells), 256, 0, st, cells, x, out, a, b, c3,
           floor, floored);
  count_launches(1);
}

void launch_gauge64(cudaStream_t st, long long cells, double* x, Partial* partials,
                    LevelScalars* sc) {
  const unsigned nb = blocks_for(cells, 256 * kSumCells);
  launch_k(k_sum_partials, nb, 256, 0, st, cells, x, partials);
  launch_finalize(st, partials, (int)nb, (double)cells, 1, sc);
  launch_k(k_sub_mean, blocks_for(cells, 256), 256, 0, st, cells, x, sc);
  count_launches(2);
}

// max |x - mean x| into sc->res (sc->lambda = mean x)
void launch_spread64(cudaStream_t st, long long cells, const double* x, Partial* partials,
                     LevelScalars* sc) {
  const unsigned nb = blocks_for(cells, 256 * kSumCells);
  launch_k(k_sum_partials, nb, 256, 0, st, cells, x, partials);
  launch_finalize(st, partials, (int)nb, (double)cells, 1, sc);
  count_launches(1);
}

// out = x + a y
__global__ void __launch_bounds__(256) k_axpy64(long long cells, const double* __restrict__ x,
                                                const double* __restrict__ y, double a,
                                                double* __restrict__ out) {
  PdlScope pdl_scope;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < cells) out[t] = fma(a, y[t], x[t]);
}

void launch_axpy64(cudaStream_t st, long long cells, const double* x, const double* y, double a,
                   double* out) {
  if (cells <= 0) return;
  launch_k(k_axpy64, blocks_for(cells, 256), 256, 0, st, cells, x, y, a, out);
  count_launches(1);
}

void launch_force64(cudaStream_t st, int n, const double* phi, double* out) {
  const long long cells = (long long)n * n * n;
  int log2n = -1;
  if ((n & (n - 1)) == 0)
    for (log2n = 0; (1 << log2n) < n;) ++log2n;
  launch_k(k_force64, blocks_for(cells, 256), 256, 0, st, n, log2n, phi, out);
  count_launches(1);
}

}  // namespace mg
