// Per-thread bodies of the FP64 kernels of mg_fp64.cu.  Each b_* body takes the
// block index as an argument so that the single-grid kernels (blk = blockIdx.x)
// and the batched work-list kernels of mg_batch.cu (blk = block within its item)
// run the same code; the cell_* functions take the item index itself, so that
// the cluster sub-cycle (mg_subcycle.cu) can spread items over its CTAs freely.
#pragma once

#include "mg_common.cuh"

namespace mg {

// The block-wide constant of a colour stage (thread 0 computes it into shared
// memory): -h^2 (lambda - k2)/6 in the sqrt form, -h^2 lambda/6 in the root form,
// lambda itself for OP_GENW.
__device__ __forceinline__ double smooth_scalar64(const LevelScalars* __restrict__ sc,
                                                  const OpConst64& c) {
  return c.mode == OP_GENW ? sc->lambda
                           : -c.h2_6 * (c.mode == OP_SQRT ? sc->lambda - c.k2 : sc->lambda);
}

// phi += omega (v - phi), the relaxed step (omega < 1).
static __device__ __noinline__ void relax64(double* phi, double v, double omega) {
  const double old = *phi;
  *phi = fma(omega, v - old, old);
}

// The update of cell (i,j,k) of a colour stage:
//   phi_new = (Sx + Sy + Sz - h^2 (D + f + lambda)) / 6.
// In the sqrt form, D = k2s sqrt(q) - k2, so phi_new = upd_s sqrt(q) + (Sx+Sy+Sz)/6 -
// h^2 f/6 + C with the block-wide C = -h^2 (lambda - k2)/6 (s_c).
template <int MODE>
__device__ __forceinline__ void cell_smooth64_at(int n, double* __restrict__ phi,
                                                 const double* __restrict__ src,
                                                 const double* __restrict__ f, double s_c,
                                                 const OpConst64& c, int i, int j, int k) {
  const long long id = lidx(i, j, k, n);
  auto nbr = [&] { return nbr_offsets(i, j, k, n); };
  if constexpr (MODE == OP_GENW) {
    const double old = phi[id];
    const double v = genw_newton(gather_at(phi + id, nbr()), old, src[id],
                                 (f ? f[id] : 0.0) + s_c, c);
    phi[id] = not_one(c.omega) ? fma(c.omega, v - old, old) : v;
    return;
  }
  const double sv = src[id];
  const double fv = f ? f[id] : 0.0;
  double face, M;
  double acc = fma(fv, -c.h2_6, s_c);
  if constexpr (MODE == OP_LINEAR) {
    long long b[6];
    gather_bits(phi + id, nbr(), b);
    stencil_forms(phi + id, nbr, b, false, face, M);
    acc = fma(-c.h2_6, sv, acc);
  } else {
    long long b[18];
    gather_bits(phi + id, nbr(), b);
    stencil_forms(phi + id, nbr, b, MODE == OP_CONJ, face, M);
    if constexpr (MODE == OP_SQRT) {
      acc = fma(c.upd_s, sqrt_clamped_fix(fma(c.e1, M, sv)), acc);
    } else {
      double q;
      bool g;
      acc = fma(-c.h2_6, root_of_M<MODE>(M, sv, c, q, g), acc);
    }
  }
  const double v = fma(face, 1.0 / 6.0, acc);
  if (not_one(c.omega))
    relax64(phi + id, v, c.omega);
  else
    phi[id] = v;
}

// One cell of a colour stage: t indexes the colour's n^3/4 cells; t >= n^3/4 does
// nothing.
template <int MODE>
__device__ __forceinline__ void cell_smooth64(int n, double* __restrict__ phi,
                                              const double* __restrict__ src,
                                              const double* __restrict__ f, double s_c,
                                              const OpConst64& c, int colour, long long t) {
  const int hn = n >> 1;
  const long long total = (long long)hn * hn * n;
  if (t >= total) return;
  int m, jj, k;
  split3((unsigned)t, hn, m, jj, k);
  const int i = 2 * m + ((colour ^ k) & 1);
  const int j = 2 * jj + (((colour >> 1) ^ k) & 1);
  cell_smooth64_at<MODE>(n, phi, src, f, s_c, c, i, j, k);
}

template <int MODE>
__device__ __forceinline__ void b_smooth_colour64(int n, double* __restrict__ phi,
                                                         const double* __restrict__ src,
                                                         const double* __restrict__ f,
                                                         const LevelScalars* __restrict__ sc,
                                                         OpConst64 c, int colour,
    long long blk) {
  __shared__ double s_c;
  if (threadIdx.x == 0) s_c = smooth_scalar64(sc, c);
  __syncthreads();
  cell_smooth64<MODE>(n, phi, src, f, s_c, c, colour, (long long)blk * blockDim.x + threadIdx.x);
}

// The defect L(phi) of cell (i,j,k) (linear index id) without a right-hand side, its
// discriminant (1 where the mode has none) and guard flag.
template <int MODE>
__device__ __forceinline__ double cell_defect_fix64(const double* __restrict__ phi, int n, int i,
                                                    int j, int k, long long id, double src,
                                                    const OpConst64& c, double& q, bool& g) {
  auto nbr = [&] { return nbr_offsets(i, j, k, n); };
  if constexpr (MODE == OP_GENW) {
    const StencilT<double> s = gather_at(phi + id, nbr());
    q = 1.0;
    const double D = root_Dc(s, phi[id], src, c, g);
    return fma((s.sx + s.sy + s.sz) - 6.0 * phi[id], c.inv_h2, -D);
  }
  double lap, M;
  if constexpr (MODE == OP_LINEAR) {
    long long b[7];
    gather_bits(phi + id, nbr(), b);
    stencil_forms(phi + id, nbr, b, false, lap, M);
    q = 1.0;
    g = false;
    return fma(lap, c.inv_h2, -src);
  }
  long long b[19];
  gather_bits(phi + id, nbr(), b);
  stencil_forms(phi + id, nbr, b, MODE == OP_CONJ, lap, M);
  return fma(lap, c.inv_h2, -root_of_M<MODE>(M, src, c, q, g));
}

// The defect d = L(phi) - f of fine cell (i,j,k) and its guard flag; ctr returns phi there.
template <int MODE>
__device__ __forceinline__ double fine_defect64(int nf, const double* __restrict__ phi,
                                               const double* __restrict__ src,
                                               const double* __restrict__ f,
                                               const OpConst64& c, int i, int j, int k,
                                               long long id, double& ctr, bool& g) {
  ctr = phi[id];
  double q;
  const double d = cell_defect_fix64<MODE>(phi, nf, i, j, k, id, src[id], c, q, g);
  return f ? d - f[id] : d;
}

template <int MODE>
__device__ __forceinline__ void b_residual_restrict64(
    int nf, const double* __restrict__ phi, const double* __restrict__ src,
    const double* __restrict__ f, OpConst64 c, double* __restrict__ phi_c,
    double* __restrict__ phihat_c, double* __restrict__ rd_c, Partial* __restrict__ partials,
    long long blk) {
  const int nc = nf >> 1;
  const long long ccells = (long long)nc * nc * nc;
  const long long t = (long long)blk * blockDim.x + threadIdx.x;
  Partial p;
  partial_init(p);
  if (t < ccells) {
    int I, J, K;
    split3((unsigned)t, nc, I, J, K);
    // The partial norms of the 8 children.  With every child finite, the sum is sd
    // itself (the same additions in the same order) and the extremes are kept as
    // integer order keys, so that the FP64 pipe, GB300's limit here, does only the
    // two sums per child.  A non-finite child sends the coarse cell through the
    // element-wise partial_add again (same values).
    double sphi = 0.0, sd = 0.0;
    long long kmax = order_key(-INFINITY), kmin = order_key(INFINITY), guards = 0;
    int bad = 0;
#pragma unroll 1
    for (int ch = 0; ch < 8; ++ch) {
      const int i = 2 * I + (ch & 1), j = 2 * J + ((ch >> 1) & 1), k = 2 * K + (ch >> 2);
      const long long id = lidx(i, j, k, nf);
      bool g;
      double ctr;
      const double d = fine_defect64<MODE>(nf, phi, src, f, c, i, j, k, id, ctr, g);
      const bool fin = finite_bits(d);
      const long long key = order_key(d);
      kmax = (fin && key > kmax) ? key : kmax;
      kmin = (fin && key < kmin) ? key : kmin;
      bad += fin ? 0 : 1;
      guards += g ? 1 : 0;
      sphi += ctr;
      sd += d;
    }
    if (bad == 0) {
      p.sum = sd;
      p.dmax = from_order_key(kmax);
      p.dmin = from_order_key(kmin);
      p.guards = guards;
    } else {
#pragma unroll 1
      for (int ch = 0; ch < 8; ++ch) {
        const int i = 2 * I + (ch & 1), j = 2 * J + ((ch >> 1) & 1), k = 2 * K + (ch >> 2);
        bool g;
        double ctr;
        partial_add(p, fine_defect64<MODE>(nf, phi, src, f, c, i, j, k, lidx(i, j, k, nf), ctr, g), g);
      }
    }
    phi_c[t] = sphi * 0.125;
    phihat_c[t] = sphi * 0.125;
    rd_c[t] = sd * 0.125;
  }
  p = block_reduce(p);
  if (threadIdx.x == 0) partials[blk] = p;
}

// The residual restriction in two steps, for launches whose per-coarse-cell
// loop would leave most SMs idle: cell_defect64 stores each fine cell's defect
// and guard flag (t indexes the nf^3 fine cells), then b_restrict_defects64
// walks every coarse cell's 8 children in the order of b_residual_restrict64,
// with its block partition, so both give the same bits.
template <int MODE>
__device__ __forceinline__ void cell_defect64(int nf, const double* __restrict__ phi,
                                              const double* __restrict__ src,
                                              const double* __restrict__ f, const OpConst64& c,
                                              double* __restrict__ dout,
                                              unsigned char* __restrict__ gout, long long t) {
  const long long cells = (long long)nf * nf * nf;
  if (t >= cells) return;
  int i, j, k;
  split3((unsigned)t, nf, i, j, k);
  bool g;
  double ctr;
  dout[t] = fine_defect64<MODE>(nf, phi, src, f, c, i, j, k, t, ctr, g);
  gout[t] = g ? 1 : 0;
}

__device__ __forceinline__ void b_restrict_defects64(
    int nf, const double* __restrict__ phi, const double* __restrict__ din,
    const unsigned char* __restrict__ gin, double* __restrict__ phi_c,
    double* __restrict__ phihat_c, double* __restrict__ rd_c, Partial* __restrict__ partials,
    long long blk) {
  const int nc = nf >> 1;
  const long long ccells = (long long)nc * nc * nc;
  const long long t = (long long)blk * blockDim.x + threadIdx.x;
  Partial p;
  partial_init(p);
  if (t < ccells) {
    int I, J, K;
    split3((unsigned)t, nc, I, J, K);
    double sphi = 0.0, sd = 0.0;
#pragma unroll
    for (int ch = 0; ch < 8; ++ch) {
      const int i = 2 * I + (ch & 1), j = 2 * J + ((ch >> 1) & 1), k = 2 * K + (ch >> 2);
      const long long id = lidx(i, j, k, nf);
      const double d = din[id];
      partial_add(p, d, gin[id] != 0);
      sphi += phi[id];
      sd += d;
    }
    phi_c[t] = sphi * 0.125;
    phihat_c[t] = sphi * 0.125;
    rd_c[t] = sd * 0.125;
  }
  p = block_reduce(p);
  if (threadIdx.x == 0) partials[blk] = p;
}

// The level norms from the per-block partials: the block-wide merge of b_finalize
// (thread 0 holds the result), and the scalars it stores.
__device__ __forceinline__ Partial merge_partials(const Partial* __restrict__ partials,
                                                  int nparts) {
  Partial p;
  partial_init(p);
  for (int b = threadIdx.x; b < nparts; b += blockDim.x) partial_merge(p, partials[b]);
  return block_reduce(p);
}

__device__ __forceinline__ double level_lambda(const Partial& p, double cells, int periodic) {
  return periodic ? p.sum / cells : 0.0;
}

__device__ __forceinline__ void store_scalars(const Partial& p, double lam,
                                              LevelScalars* __restrict__ sc) {
  sc->lambda = lam;
  sc->sum = p.sum;
  sc->dmax = p.dmax;
  sc->dmin = p.dmin;
  sc->res = (p.nonfinite > 0) ? NAN : fmax(p.dmax - lam, lam - p.dmin);
  sc->guards = p.guards;
  sc->nonfinite = p.nonfinite;
}

__device__ __forceinline__ void b_finalize(const Partial* __restrict__ partials, int nparts,
                                                  double cells, int periodic,
                                                  LevelScalars* __restrict__ sc,
    long long blk) {
  const Partial p = merge_partials(partials, nparts);
  if (threadIdx.x == 0) store_scalars(p, level_lambda(p, cells, periodic), sc);
}

// One coarse cell of the FAS right-hand side f_c = L_c(phi_c) - f_c + lambda_f
// (t indexes the nc^3 cells; lam_f is the fine level's lambda; cell 0 also clears
// the coarse lambda).
template <int MODE>
__device__ __forceinline__ void cell_fas_rhs64(int nc, const double* __restrict__ phi_c,
                                               const double* __restrict__ src_c,
                                               double* __restrict__ f_c, const OpConst64& c,
                                               double lam_f, LevelScalars* __restrict__ coarse_sc,
                                               long long t) {
  const long long cells = (long long)nc * nc * nc;
  if (t == 0) coarse_sc->lambda = 0.0;
  if (t >= cells) return;
  int i, j, k;
  split3((unsigned)t, nc, i, j, k);
  double q;
  bool g;
  const double L = cell_defect_fix64<MODE>(phi_c, nc, i, j, k, t, src_c[t], c, q, g);
  f_c[t] = L - f_c[t] + lam_f;
}

template <int MODE>
__device__ __forceinline__ void b_fas_rhs64(int nc, const double* __restrict__ phi_c,
                                                   const double* __restrict__ src_c,
                                                   double* __restrict__ f_c, OpConst64 c,
                                                   const LevelScalars* __restrict__ fine_sc,
                                                   LevelScalars* __restrict__ coarse_sc,
    long long blk) {
  cell_fas_rhs64<MODE>(nc, phi_c, src_c, f_c, c, fine_sc->lambda, coarse_sc,
                 (long long)blk * blockDim.x + threadIdx.x);
}

// One fine cell of the trilinear prolongation of the coarse correction
// phi_c - phihat_c, added to phi_f (t indexes the (2 nc)^3 fine cells): 3 parent + 1
// neighbour along x, y and z in turn, the order of k_prolong_column64 too.
__device__ __forceinline__ void cell_prolong64(int nc, const double* __restrict__ phi_c,
                                               const double* __restrict__ phihat_c,
                                               double* __restrict__ phi_f, long long t) {
  const int nf = nc << 1;
  const long long cells = (long long)nf * nf * nf;
  if (t >= cells) return;
  int i, j, k;
  split3((unsigned)t, nf, i, j, k);
  const int I0 = i >> 1, J0 = j >> 1, K0 = k >> 1;
  const int I1 = (i & 1) ? wrap_up(I0, nc) : wrap_dn(I0, nc);
  const int J1 = (j & 1) ? wrap_up(J0, nc) : wrap_dn(J0, nc);
  const int K1 = (k & 1) ? wrap_up(K0, nc) : wrap_dn(K0, nc);
  auto e = [&](int a, int b, int cc) {
    const long long q = lidx(a, b, cc, nc);
    return phi_c[q] - phihat_c[q];
  };
  auto row = [&](int b, int cc) { return fma(3.0, e(I0, b, cc), e(I1, b, cc)); };
  auto plane = [&](int cc) { return fma(3.0, row(J0, cc), row(J1, cc)); };
  phi_f[t] = fma(fma(3.0, plane(K0), plane(K1)), 1.0 / 64.0, phi_f[t]);
}

__device__ __forceinline__ void b_prolong_correct64(int nc, const double* __restrict__ phi_c,
                                                           const double* __restrict__ phihat_c,
                                                           double* __restrict__ phi_f,
    long long blk) {
  cell_prolong64(nc, phi_c, phihat_c, phi_f, (long long)blk * blockDim.x + threadIdx.x);
}

__device__ __forceinline__ void b_coarsest64(int n, double* __restrict__ phi,
                                                    const double* __restrict__ src,
                                                    const double* __restrict__ f, OpConst64 c,
                                                    LevelScalars* __restrict__ sc, int max_sweeps,
                                                    double drop, int check_every,
    long long blk) {
  extern __shared__ double smem64[];
  __shared__ double s_lam, s_res0, s_res;
  const int cells = n * n * n;
  double* sphi = smem64;
  double* ssrc = smem64 + cells;
  double* sf = smem64 + 2 * cells;
  for (int q = threadIdx.x; q < cells; q += blockDim.x) {
    sphi[q] = phi[q];
    ssrc[q] = src[q];
    sf[q] = f ? f[q] : 0.0;
  }
  if (threadIdx.x == 0) s_lam = sc->lambda;
  __syncthreads();
  double scale = 0.0;
  auto residual = [&](double& res_out) {
    Partial p;
    partial_init(p);
    double mag = 0.0;
    for (int q = threadIdx.x; q < cells; q += blockDim.x) {
      const int i = q % n, j = (q / n) % n, k = q / (n * n);
      const StencilT<double> s = gather_periodic<double>(sphi, i, j, k, n);
      bool g;
      const double D = root_Dc(s, sphi[q], ssrc[q], c, g);
      const double lnb = s.sx + s.sy + s.sz;
      const double lap = lnb - 6.0 * sphi[q];
      partial_add(p, fma(lap, c.inv_h2, -D) - sf[q], g);
      mag = fmax(mag, (fabs(lnb) + 6.0 * fabs(sphi[q])) * c.inv_h2 + fabs(D) + fabs(sf[q]));
    }
    scale = block_max(mag);
    p = block_reduce(p);
    if (threadIdx.x == 0) {
      const double lam = p.sum / (double)cells;
      s_lam = lam;
      s_res = (p.nonfinite > 0) ? NAN : fmax(p.dmax - lam, lam - p.dmin);
      sc->guards = p.guards;
      sc->nonfinite = p.nonfinite;
    }
    __syncthreads();
    res_out = s_res;
  };
  double r;
  residual(r);
  if (threadIdx.x == 0) s_res0 = r;
  __syncthreads();
  const double r0 = s_res0;
  double r_prev = r0;
  const int hn = n >> 1;
  const int per_colour = hn * hn * n;
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    for (int colour = 0; colour < 4; ++colour) {
      for (int t = threadIdx.x; t < per_colour; t += blockDim.x) {
        const int m = t % hn, jj = (t / hn) % hn, k = t / (hn * hn);
        const int i = 2 * m + ((colour ^ k) & 1);
        const int j = 2 * jj + (((colour >> 1) ^ k) & 1);
        const int id = i + n * (j + n * k);
        const StencilT<double> s = gather_periodic<double>(sphi, i, j, k, n);
        double v;
        if (c.mode == OP_GENW) {
          v = genw_newton(s, sphi[id], ssrc[id], sf[id] + s_lam, c);
        } else {
          bool g;
          const double D = root_D(s, ssrc[id], c, g);
          v = fma(-c.h2, D + sf[id] + s_lam, s.sx + s.sy + s.sz) * (1.0 / 6.0);
        }
        sphi[id] = not_one(c.omega) ? fma(c.omega, v - sphi[id], sphi[id]) : v;
      }
      __syncthreads();
    }
    if ((sweep + 1) % check_every == 0 || sweep + 1 == max_sweeps) {
      residual(r);
      if (coarsest_done(r, r0, r_prev, scale, drop)) break;
      r_prev = r;
    }
  }
  for (int q = threadIdx.x; q < cells; q += blockDim.x) phi[q] = sphi[q];
  if (threadIdx.x == 0) {
    sc->lambda = s_lam;
    sc->res = s_res;
  }
}

// Cells per thread of b_affine64.  The floored cells are counted once per block: one
// atomic per warp, all on one counter, took 2.5 of the 3.5 ms of a 512^3 field with most of
// its cells floored (now 1.2 ms in all).
constexpr int kAffineCells = 4;

__device__ __forceinline__ void b_affine64(long long cells, const double* __restrict__ delta,
                                                  double* __restrict__ out, double a, double b,
                                                  double c3, int floor,
                                                  unsigned long long* __restrict__ floored,
    long long blk) {
  int hits = 0;
#pragma unroll
  for (int r = 0; r < kAffineCells; ++r) {
    const long long t = (blk * kAffineCells + r) * blockDim.x + threadIdx.x;
    if (t < cells) {
      double v = fma(a, delta[t], b);
      if (floor) {
        const double lhs = (b != 0.0) ? v : fma(c3, v, 1.0);  // 1 + c3 kappa delta
        if (neg_guard(lhs)) {
          ++hits;
          v = (b != 0.0) ? 0.0 : -1.0 / c3;
        }
      }
      out[t] = v;
    }
  }
  if (floored) {
    __shared__ unsigned total;
    if (threadIdx.x == 0) total = 0;
    __syncthreads();
    const unsigned h = __reduce_add_sync(0xffffffffu, (unsigned)hits);
    if ((threadIdx.x & 31) == 0 && h) atomicAdd(&total, h);
    __syncthreads();
    if (threadIdx.x == 0 && total) atomicAdd(floored, (unsigned long long)total);
  }
}

// Cells per thread of b_sum_partials: with one, the block reduction (about 15 FP64 warp
// instructions) outweighed the addition it follows (512^3: 4676 -> 368 us).
constexpr int kSumCells = 16;

__device__ __forceinline__ void b_sum_partials(long long cells, const double* __restrict__ x,
                                                      Partial* __restrict__ partials,
    long long blk) {
  Partial p;
  partial_init(p);
#pragma unroll 4
  for (int r = 0; r < kSumCells; ++r) {
    const long long t = (blk * kSumCells + r) * blockDim.x + threadIdx.x;
    if (t < cells) partial_add(p, x[t], false);
  }
  p = block_reduce(p);
  if (threadIdx.x == 0) partials[blk] = p;
}

__device__ __forceinline__ void b_sub_mean(long long cells, double* __restrict__ x,
                                                  const LevelScalars* __restrict__ sc,
    long long blk) {
  const long long t = (long long)blk * blockDim.x + threadIdx.x;
  if (t < cells) x[t] -= sc->lambda;
}

}  // namespace mg
