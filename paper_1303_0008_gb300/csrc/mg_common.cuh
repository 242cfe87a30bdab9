// Device-side building blocks shared by the CUDA kernels of libmg.
//
// The discrete operator is the one of Sec. III.B of arXiv:1303.0008 (the L^h
// equation with its Sigma_ijk), written for the operator-splitting constant
// w = 1/3 (Sec. III.A).  With w = 1/3 the non-source part of Sigma,
//     Sigma_d h^4 = [(Sx-Sy)^2 + (Sx-Sz)^2 + (Sy-Sz)^2]/3 + (Cxy^2 + Cxz^2 + Cyz^2)/8,
// (Sx = phi_{i+1} + phi_{i-1}, Cxy the four-point cross difference), does not
// involve the centre value, so the Newton step of Sec. III.B is the exact
// pointwise solve of L^h phi = rhs for the centre cell.
//
// Parameters follow the library convention: alpha is the coefficient of the
// nonlinear term of Eq. code_eqn (the paper's alpha is 1/alpha), kappa the source
// coefficient.  With u = kappa*delta + alpha*Sigma_d and q = 1 + 4(1-w) alpha u,
// the root of Eq. two_branch is D = (sigma sqrt(q) - 1) / (2(1-w) alpha) where
// sigma = +1 picks the physical root of Eq. one_branch.  When q < 0 the square
// root is taken of 0 (the real part of the complex root) and the cell counts as
// guarded.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>
#include <type_traits>

#include "mg_fix64.cuh"

namespace mg {

// How the root D is evaluated.
enum OpMode : int {
  OP_LINEAR = 0,  // alpha == 0: D = kappa*delta
  OP_SQRT = 1,    // D = k2 (sigma sqrt(q) - 1); src = 1 + c3 kappa delta
  OP_CONJ = 2,    // physical root as 2u/(1+sqrt(q)) for small |alpha|; src = kappa delta
  OP_GENW = 3     // splitting w != 1/3: Sigma involves the centre value (full Newton step)
};

// run(mode) with the mode as a type: the kernels that go cell by cell are compiled for one
// mode each, without the others' code and registers.
template <typename Run>
__host__ __device__ __forceinline__ void by_mode(int mode, Run run) {
  switch (mode) {
    case OP_LINEAR: run(std::integral_constant<int, OP_LINEAR>{}); break;
    case OP_SQRT: run(std::integral_constant<int, OP_SQRT>{}); break;
    case OP_CONJ: run(std::integral_constant<int, OP_CONJ>{}); break;
    default: run(std::integral_constant<int, OP_GENW>{});
  }
}

// Per-level constants of the FP64 operator.
struct OpConst64 {
  double h2;      // h^2
  double inv_h2;  // 1/h^2
  double e1, e2;  // OP_SQRT: q = src + e1*A + e2*B
  double c1, c2;  // OP_CONJ: u = src + c1*A + c2*B
  double c3;      // 4(1-w) alpha
  double k2s;     // sigma * k2, k2 = 2/c3
  double k2;
  double e1h, c1h;  // 2*e1, 2*c1: the same terms written with A/2
  double h2_6;      // h^2/6
  double upd_s;     // -h^2 k2s / 6: the smoother's coefficient of sqrt(q)
  double omega;     // relaxation of the pointwise Newton step (1 = the plain step)
  // OP_GENW: q = src + gA (Dxx^2 + Dyy^2 + Dzz^2) + gB (Dxx Dyy + Dxx Dzz + Dyy Dzz)
  //            + gC (Cxy^2 + Cxz^2 + Cyz^2), the D's including the centre value;
  //          gAB = gA + gB, so dq/dphi_centre = -4 gAB (Sx + Sy + Sz - 6 phi)
  double gA, gB, gC, gAB;
  int mode;
};

// Per-level constants of the FP32 correction operator (mixed precision).
struct OpConst32 {
  float h2, inv_h2;
  float g1, g2;   // alpha/(3h^4), alpha/(8h^4): Delta u = g1*dA + g2*dB
  float c3;       // 4(1-w) alpha
  float k2;       // 2/c3 (0 when alpha == 0)
  float sigma;    // +1 physical root, -1 the other one
  float sigma2;   // 2 sigma
  float sk2;      // sigma k2
  int linear;     // alpha == 0
};

// Scalars that a residual evaluation leaves for one level.
struct LevelScalars {
  double lambda;     // compatibility constant mean(d) (periodic), 0 (Dirichlet)
  double res;        // max |d - lambda|
  double sum;        // sum of d
  double dmax, dmin;
  long long guards;  // cells with q < 0
  long long nonfinite;
  unsigned long long floored;  // cells whose source was held at the real-root bound
};

// Programmatic dependent launch.  Kernels launched with launch_k() may start
// while the grid before them in the stream is still finishing; each such kernel
// opens a PdlScope first, which waits until that grid has completed and its
// writes are visible (griddepcontrol.wait), and on exit lets the next grid
// begin launching (griddepcontrol.launch_dependents).  What overlaps is launch
// latency and the scheduling of CTAs, never a kernel's memory accesses.
struct PdlScope {
  __device__ __forceinline__ PdlScope() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
  __device__ __forceinline__ ~PdlScope() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  }
};

// Split a cell index t (< 2^31; grids have n <= 1024) into (t % d, (t / d) % d,
// t / d^2) with 32-bit arithmetic; shifts and masks when d is a power of two.
__device__ __forceinline__ void split3(unsigned t, int d, int& i, int& j, int& k) {
  const unsigned ud = (unsigned)d;
  if ((ud & (ud - 1u)) == 0u) {
    const int s = __ffs(d) - 1;
    const unsigned r = t >> s;
    i = (int)(t & (ud - 1u));
    j = (int)(r & (ud - 1u));
    k = (int)(r >> s);
  } else {
    const unsigned r = t / ud, r2 = r / ud;
    i = (int)(t - r * ud);
    j = (int)(r - r2 * ud);
    k = (int)r2;
  }
}

__device__ __forceinline__ int wrap_up(int i, int n) { return (i + 1 == n) ? 0 : i + 1; }
__device__ __forceinline__ int wrap_dn(int i, int n) { return (i == 0) ? n - 1 : i - 1; }

__device__ __forceinline__ long long lidx(int i, int j, int k, int n) {
  return (long long)i + (long long)n * ((long long)j + (long long)n * (long long)k);
}

// Cells per thread of the outer FP64 residual with its FP32 hand-off.
constexpr int kHandoffCells = 4;


// The 18 stencil neighbours of one cell in the form the operator uses: face pair
// sums and cross differences (without the 1/4).
template <typename T>
struct StencilT {
  T sx, sy, sz, cxy, cxz, cyz;
};

// Offsets from cell (i,j,k) to its six face neighbours in a periodic n^3 array,
// x fastest, with the wrap folded in (n <= 1024, so every offset fits in 32 bits).
struct NbrOff {
  int xp, xm, yp, ym, zp, zm;
};

__device__ __forceinline__ NbrOff nbr_offsets(int i, int j, int k, int n) {
  const int n2 = n * n, n3 = n2 * n;
  NbrOff o;
  o.xp = (i + 1 == n) ? 1 - n : 1;
  o.xm = (i == 0) ? n - 1 : -1;
  o.yp = (j + 1 == n) ? n - n2 : n;
  o.ym = (j == 0) ? n2 - n : -n;
  o.zp = (k + 1 == n) ? n2 - n3 : n2;
  o.zm = (k == 0) ? n3 - n2 : -n2;
  return o;
}

// Face sums and cross differences around the cell at c (a pointer to it).
template <typename T>
__device__ __forceinline__ StencilT<T> gather_at(const T* __restrict__ c, const NbrOff& o) {
  StencilT<T> s;
  s.sx = c[o.xp] + c[o.xm];
  s.sy = c[o.yp] + c[o.ym];
  s.sz = c[o.zp] + c[o.zm];
  s.cxy = (c[o.xp + o.yp] + c[o.xm + o.ym]) - (c[o.xp + o.ym] + c[o.xm + o.yp]);
  s.cxz = (c[o.xp + o.zp] + c[o.xm + o.zm]) - (c[o.xp + o.zm] + c[o.xm + o.zp]);
  s.cyz = (c[o.yp + o.zp] + c[o.ym + o.zm]) - (c[o.yp + o.zm] + c[o.ym + o.zp]);
  return s;
}

// Gather the face sums and cross differences of cell (i,j,k) of a periodic n^3
// array.
template <typename T>
__device__ __forceinline__ StencilT<T> gather_periodic(const T* __restrict__ p, int i, int j,
                                                       int k, int n) {
  return gather_at(p + lidx(i, j, k, n), nbr_offsets(i, j, k, n));
}

// A/2 with A = (Sx-Sy)^2 + (Sx-Sz)^2 + (Sy-Sz)^2 = 2[a1(a1-a2) + a2^2], a1 = Sx-Sy,
// a2 = Sx-Sz (the form is positive definite, so no cancellation).
__device__ __forceinline__ double half_A(const StencilT<double>& s) {
  const double a1 = s.sx - s.sy, a2 = s.sx - s.sz;
  return fma(a1, a1 - a2, a2 * a2);
}

// sqrt(q) for q >= 0 as q * rsqrt(q) (rsqrt is within 1 ulp); 0 stays 0 and a NaN
// stays NaN.
__device__ __forceinline__ double sqrt_nonneg(double q) {
  return (q == 0.0) ? 0.0 : q * rsqrt(q);
}

// sqrt_nonneg(q < 0 ? 0 : q) with both tests on the bit pattern (integer ALU
// instructions instead of FP64 compares, which share GB300's narrow FP64 pipe).
// As a signed 64-bit integer, +0 is 0 and the negative non-NaN doubles (-0 to
// -inf) are exactly the values <= the pattern of -inf; negative NaNs lie above it
// and, like every other input, take q * rsqrt(q).  Same result for every q.
__device__ __forceinline__ double sqrt_clamped(double q) {
  const long long b = __double_as_longlong(q);
  return (b == 0 || b <= (long long)0xFFF0000000000000ULL) ? 0.0 : q * rsqrt(q);
}

// q < 0 on the bit pattern: the negative non-NaN doubles other than -0.
__device__ __forceinline__ bool neg_guard(double q) {
  const long long b = __double_as_longlong(q);
  return b <= (long long)0xFFF0000000000000ULL && b != (long long)0x8000000000000000ULL;
}

// x != 1.0 on the bit pattern (for the relaxation factor, validated in (0, 1]).
__device__ __forceinline__ bool not_one(double x) {
  return __double_as_longlong(x) != 0x3FF0000000000000LL;
}

// An integer key of a double whose order is the numeric order (-0 below +0): the
// bit pattern with the magnitude bits flipped for negative values.  The map is
// its own inverse.
__device__ __forceinline__ long long order_key(double d) {
  const long long b = __double_as_longlong(d);
  return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFLL);
}
__device__ __forceinline__ double from_order_key(long long k) {
  return __longlong_as_double(k ^ ((k >> 63) & 0x7FFFFFFFFFFFFFFFLL));
}

// isfinite(d) on the bit pattern: the exponent field is not all ones.
__device__ __forceinline__ bool finite_bits(double d) {
  return ((__double_as_longlong(d) >> 52) & 0x7ff) != 0x7ff;
}

// D (the root of Eq. two_branch) from the stencil and the per-cell source term.
// `guard` is set when the discriminant is negative.
__device__ __forceinline__ double root_D(const StencilT<double>& s, double src,
                                         const OpConst64& c, bool& guard) {
  if (c.mode == OP_LINEAR) {
    guard = false;
    return src;
  }
  const double A2 = half_A(s);
  const double B = fma(s.cxy, s.cxy, fma(s.cxz, s.cxz, s.cyz * s.cyz));
  if (c.mode == OP_SQRT) {
    const double q = fma(c.e1h, A2, fma(c.e2, B, src));
    guard = neg_guard(q);
    return fma(c.k2s, sqrt_clamped(q), -c.k2);
  }
  const double u = fma(c.c1h, A2, fma(c.c2, B, src));
  const double q = fma(c.c3, u, 1.0);
  guard = q < 0.0;
  if (guard) return -c.k2;
  return (2.0 * u) / (1.0 + sqrt(q));
}

// The 18 neighbours of a cell (with NV = 6 those across its faces alone; with NV = 7 and 19
// the cell itself too) as bit patterns, in the order x, y, z face pairs, the xy, xz, yz cells
// as (++, --, +-, -+), the centre.
template <int NV>
__device__ __forceinline__ void gather_bits(const double* __restrict__ c, const NbrOff& o,
                                            long long (&b)[NV]) {
  const int off[18] = {o.xp,        o.xm,        o.yp,        o.ym,        o.zp,        o.zm,
                       o.xp + o.yp, o.xm + o.ym, o.xp + o.ym, o.xm + o.yp, o.xp + o.zp,
                       o.xm + o.zm, o.xp + o.zm, o.xm + o.zp, o.yp + o.zp, o.ym + o.zm,
                       o.yp + o.zm, o.ym + o.zp};
#pragma unroll
  for (int k = 0; k < NV; ++k)
    b[k] = __double_as_longlong(c[(NV & 1) && k == NV - 1 ? 0 : off[k]]);
}

// stencil_forms of the cell at c in FP64, for values that fix_align refuses.  Not
// inlined, as the other rare paths here: kept out of the way of the code that runs.
static __device__ __noinline__ void stencil_forms_fp64(const double* c, NbrOff o, int nv,
                                                       double* face, double* M) {
  const StencilT<double> s = gather_at(c, o);
  const double sum = s.sx + s.sy + s.sz;
  const double B = fma(s.cxy, s.cxy, fma(s.cxz, s.cxz, s.cyz * s.cyz));
  *face = (nv & 1) ? sum - 6.0 * *c : sum;
  *M = fma(0.375, B, 2.0 * half_A(s));
}

// What the operator needs of the stencil at `at` (b: its gather_bits, used up; nbr()
// its offsets):
//   face = Sx + Sy + Sz, with the centre (NV = 7, 19) Sx + Sy + Sz - 6 phi;
//   M = A + (3/8) B of Sigma_d h^4 = A/3 + B/8 (0 with NV = 6, 7: the linear form).
// near: of fix_align.
template <int NV, typename Nbr>
__device__ __forceinline__ void stencil_forms(const double* at, Nbr nbr, long long (&b)[NV],
                                              bool near, double& face, double& M) {
  FixRef r;
  M = 0.0;
  if (!fix_align(b, r, near)) {
    double fs, ms;
    stencil_forms_fp64(at, nbr(), NV, &fs, &ms);
    face = fs;
    if (NV >= 18) M = ms;
    return;
  }
  unsigned long long u[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) u[k] = (unsigned long long)b[k];
  const unsigned long long sx = u[0] + u[1], sy = u[2] + u[3], sz = u[4] + u[5];
  const unsigned long long sub = (NV & 1) ? 6 * u[NV - 1] : (unsigned long long)r.off6;
  face = fix_signed((long long)(sx + sy + sz - sub), r);
  if constexpr (NV >= 18) {
    const long long a[3] = {(long long)(sx - sy), (long long)(sx - sz), (long long)(sy - sz)};
    const long long c[3] = {(long long)((u[6] + u[7]) - (u[8] + u[9])),
                            (long long)((u[10] + u[11]) - (u[12] + u[13])),
                            (long long)((u[14] + u[15]) - (u[16] + u[17]))};
    int sh;
    unsigned top;
    const unsigned long long N = fix_quad(a, c, sh, top);
    M = fix_double(N, 64 - 2 * sh + 2 * r.ue);
  }
}

// sqrt_clamped with the square root of a normal q on the integer pipe.
static __device__ __noinline__ double sqrt_clamped_rare(double q) { return sqrt_clamped(q); }

__device__ __forceinline__ double sqrt_clamped_fix(double q) {
  return fix_normal(q) ? sqrt_fix_normal(q) : sqrt_clamped_rare(q);
}

// The root D of Eq. two_branch from M (stencil_forms) and the source term; q is the
// discriminant (1 in the linear mode) and guard whether it is negative.
template <int MODE>
__device__ __forceinline__ double root_of_M(double M, double src, const OpConst64& c, double& q,
                                            bool& guard) {
  q = 1.0;
  guard = false;
  if (MODE == OP_LINEAR) return src;
  if (MODE == OP_SQRT) {
    q = fma(c.e1, M, src);
    guard = neg_guard(q);
    return fma(c.k2s, sqrt_clamped_fix(q), -c.k2);
  }
  const double u = fma(c.c1, M, src);
  q = fma(c.c3, u, 1.0);
  guard = q < 0.0;
  if (guard) return -c.k2;
  return (2.0 * u) / (1.0 + sqrt(q));
}

// Discriminant of a cell for a general splitting constant w (Sec. III.B,
// Sigma_ijk with every second difference taken through the centre value).
__device__ __forceinline__ double genw_q(const StencilT<double>& s, double ctr, double src,
                                         const OpConst64& c) {
  const double dxx = fma(-2.0, ctr, s.sx), dyy = fma(-2.0, ctr, s.sy), dzz = fma(-2.0, ctr, s.sz);
  const double sq = fma(dxx, dxx, fma(dyy, dyy, dzz * dzz));
  const double cr = fma(dxx, dyy, fma(dxx, dzz, dyy * dzz));
  const double cc = fma(s.cxy, s.cxy, fma(s.cxz, s.cxz, s.cyz * s.cyz));
  return fma(c.gA, sq, fma(c.gB, cr, fma(c.gC, cc, src)));
}

// D of any mode; ctr (the cell's own value) enters only for OP_GENW.
__device__ __forceinline__ double root_Dc(const StencilT<double>& s, double ctr, double src,
                                          const OpConst64& c, bool& guard) {
  if (c.mode != OP_GENW) return root_D(s, src, c, guard);
  const double q = genw_q(s, ctr, src, c);
  guard = neg_guard(q);
  return fma(c.k2s, sqrt_clamped(q), -c.k2);
}

// Newton step of one cell for OP_GENW: phi - L/(dL/dphi) with
// L = (Sx + Sy + Sz - 6 phi)/h^2 - D - rhs and dL/dphi = -6/h^2 - dD/dphi, where
// dD/dphi = -2 k2s gAB (Sx + Sy + Sz - 6 phi) / sqrt(q) (taken as 0 for q <= 1e-12).
__device__ __forceinline__ double genw_newton(const StencilT<double>& s, double ctr, double src,
                                              double rhs, const OpConst64& c) {
  const double q = genw_q(s, ctr, src, c);
  const double sq = sqrt_nonneg(q < 0.0 ? 0.0 : q);
  const double D = fma(c.k2s, sq, -c.k2);
  const double lap6 = fma(-6.0, ctr, s.sx + s.sy + s.sz);
  const double L = fma(lap6, c.inv_h2, -D) - rhs;
  const double dD = q > 1e-12 ? -2.0 * c.k2s * c.gAB * lap6 / sq : 0.0;
  const double J = fma(-6.0, c.inv_h2, -dD);
  return ctr - L / J;
}

// Deterministic block reduction of (sum, max, min, guards, nonfinite).
struct Partial {
  double sum, dmax, dmin;
  long long guards, nonfinite;
};

__device__ __forceinline__ void partial_init(Partial& p) {
  p.sum = 0.0;
  p.dmax = -INFINITY;
  p.dmin = INFINITY;
  p.guards = 0;
  p.nonfinite = 0;
}

// The extremes compare integer order keys (order_key) rather than FP64 values:
// the FP64 pipe is the limit of the kernels that call this per cell.
__device__ __forceinline__ void partial_add(Partial& p, double d, bool guard) {
  if (finite_bits(d)) {
    p.sum += d;
    const long long k = order_key(d);
    if (k > order_key(p.dmax)) p.dmax = d;
    if (k < order_key(p.dmin)) p.dmin = d;
  } else {
    p.nonfinite += 1;
  }
  p.guards += guard ? 1 : 0;
}

__device__ __forceinline__ void partial_merge(Partial& a, const Partial& b) {
  a.sum += b.sum;
  if (order_key(b.dmax) > order_key(a.dmax)) a.dmax = b.dmax;
  if (order_key(b.dmin) < order_key(a.dmin)) a.dmin = b.dmin;
  a.guards += b.guards;
  a.nonfinite += b.nonfinite;
}

__device__ __forceinline__ Partial warp_reduce(Partial p) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    Partial q;
    q.sum = __shfl_down_sync(0xffffffffu, p.sum, o);
    q.dmax = __shfl_down_sync(0xffffffffu, p.dmax, o);
    q.dmin = __shfl_down_sync(0xffffffffu, p.dmin, o);
    q.guards = __shfl_down_sync(0xffffffffu, p.guards, o);
    q.nonfinite = __shfl_down_sync(0xffffffffu, p.nonfinite, o);
    partial_merge(p, q);
  }
  return p;
}

// Reduce over the block; thread 0 returns the block's value.  blockDim.x must
// be a multiple of 32 and at most 1024.
__device__ __forceinline__ Partial block_reduce(Partial p) {
  __shared__ Partial sh[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  p = warp_reduce(p);
  if (lane == 0) sh[wid] = p;
  __syncthreads();
  const int nw = (blockDim.x + 31) >> 5;
  if (wid == 0) {
    Partial q;
    if (lane < nw) q = sh[lane];
    else partial_init(q);
    q = warp_reduce(q);
    p = q;
  }
  __syncthreads();
  return p;
}

// Maximum over the block; every thread returns it.
__device__ __forceinline__ double block_max(double v) {
  __shared__ double shm[32];
  __shared__ double result;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
  if (lane == 0) shm[wid] = v;
  __syncthreads();
  if (wid == 0) {
    const int nw = (blockDim.x + 31) >> 5;
    double w = lane < nw ? shm[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) w = fmax(w, __shfl_down_sync(0xffffffffu, w, o));
    if (lane == 0) result = w;
  }
  __syncthreads();
  return result;
}

// Stopping rule of the one-CTA coarsest solves: the residual fell by `drop`, or
// it reached the rounding level of the operator's terms (`scale` is the largest
// term), or it stopped falling.
__device__ __forceinline__ bool coarsest_done(double r, double r0, double r_prev, double scale,
                                              double drop) {
  if (!(r > drop * r0)) return true;
  if (r <= 64.0 * 1.1102230246251565e-16 * scale) return true;
  return r >= 0.95 * r_prev;
}

// From nc = 48 on (fine side 96, where columns of four cells reach most SMs) the
// prolongation runs by columns; they are eight cells deep once that leaves four CTAs per SM.
__host__ __device__ inline bool prolong_columns(int nc) { return nc >= 48; }
__host__ __device__ inline dim3 prolong_grid(int nc, int kz) {
  return dim3((unsigned)(nc + 31) / 32, (unsigned)(nc + 7) / 8, (unsigned)(nc + kz - 1) / kz);
}
__host__ __device__ inline int prolong_depth(int nc) {
  const dim3 g = prolong_grid(nc, 8);
  return (long long)g.x * g.y * g.z >= 608 ? 8 : 4;
}

// Trilinear prolongation of the coarse correction coarse - hat into a field, by columns: a
// thread takes KZ coarse cells above one
// another and their 8 KZ children, the CTA 32 x 8 columns.  A coarse plane's corrections
// are formed once in shared memory, interpolated along x and y once (10 multiply-adds per
// coarse cell) and used for the planes of children above and below: 3.7 FP64 instructions
// per fine cell instead of 11 (19 with the corrections formed by each of their readers).
// At 300^3 the kernel takes 223 instead of 873 us; in the FP64 solve of 512^3
// the finest one 1.0 instead of 2.4 ms.  The FP64 pipe still bounds it.
// The FP32 cycle's was bound by its eight loads per fine cell: all of a 512^3 mixed solve
// 16.0 -> 4.0 ms, of the 64-solve batch 9.3 -> 3.4 ms.
template <typename T, typename T2, int KZ>
__device__ __forceinline__ void prolong_column(int nc, const T* __restrict__ coarse,
                                               const T* __restrict__ hat, T* __restrict__ field,
                                               int bx, int by, int bz) {
  constexpr int W = 34, H = 10;
  __shared__ T e[2][W * H];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int I0 = bx * 32, J0 = by * 8, K0 = bz * KZ;
  auto wrap = [nc](int v) { return v < 0 ? v + nc : (v >= nc ? v - nc : v); };
  int at[2];  // this thread's cells of a plane of the CTA's tile
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int q = threadIdx.x + 256 * r, y = q / W;
    at[r] = wrap(J0 - 1 + y) * nc + wrap(I0 - 1 + q - W * y);
  }
  auto load = [&](int K, T* t) {
    const long long p = (long long)wrap(K) * nc * nc;
    t[threadIdx.x] = coarse[p + at[0]] - hat[p + at[0]];
    if (threadIdx.x < W * H - 256)
      t[threadIdx.x + 256] = coarse[p + at[1]] - hat[p + at[1]];
  };
  // (y side, x side) of the column's cell in a plane: towards -y or +y, -x or +x
  auto interpolate = [&](const T* t, T (&b)[4]) {
    T a[3][2];
#pragma unroll
    for (int y = 0; y < 3; ++y) {
      const T* r = t + (w + y) * W + lane + 1;
      a[y][0] = fma(T(3), r[0], r[-1]);
      a[y][1] = fma(T(3), r[0], r[1]);
    }
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      b[x] = fma(T(3), a[1][x], a[0][x]);
      b[2 + x] = fma(T(3), a[1][x], a[2][x]);
    }
  };
  T lo[4], mid[4], up[4];
  load(K0 - 1, e[0]);
  load(K0, e[1]);
  __syncthreads();
  interpolate(e[0], lo);
  interpolate(e[1], mid);
  __syncthreads();
  const int I = I0 + lane, J = J0 + w, nf = 2 * nc;
  const bool in = I < nc && J < nc;
#pragma unroll 1
  for (int s = 0; s < KZ && K0 + s < nc; ++s) {
    const int K = K0 + s;
    T* t = e[s & 1];
    load(K + 1, t);
    T2 v[4];
    T2* f = reinterpret_cast<T2*>(field + lidx(2 * I, 2 * J, 2 * K, nf));
    const long long row = nf / 2, plane = (long long)nf * nf / 2;  // in pairs
    if (in) {
      v[0] = f[0];
      v[1] = f[row];
      v[2] = f[plane];
      v[3] = f[plane + row];
    }
    __syncthreads();
    interpolate(t, up);
    if (in) {
#pragma unroll
      for (int y = 0; y < 2; ++y) {
        v[y].x = fma(fma(T(3), mid[2 * y], lo[2 * y]), T(1) / T(64), v[y].x);
        v[y].y = fma(fma(T(3), mid[2 * y + 1], lo[2 * y + 1]), T(1) / T(64), v[y].y);
        v[2 + y].x = fma(fma(T(3), mid[2 * y], up[2 * y]), T(1) / T(64), v[2 + y].x);
        v[2 + y].y = fma(fma(T(3), mid[2 * y + 1], up[2 * y + 1]), T(1) / T(64), v[2 + y].y);
      }
      f[0] = v[0];
      f[row] = v[1];
      f[plane] = v[2];
      f[plane + row] = v[3];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      lo[q] = mid[q];
      mid[q] = up[q];
    }
  }
}

}  // namespace mg
