// Dense (Sigma^T Sigma)^+ by Newton-Schulz refinement on the tensor cores.
//
// With M = Sigma^T Sigma + 1 1^T / n, the identity of Sec. 3.2 gives
// (Sigma^T Sigma)^+ = M^{-1} - 1 1^T / n.  The start X0 ~ M^{-1} is one symmetric multigrid
// V(1,1) cycle applied to the projected identity (a convergent V-cycle B has the eigenvalues of
// M B in (0, 2), so the spectral radius of I - M X0 is below 1), or a loose multigrid-PCG solve;
// then
//     R_k = I - M X_k   (FP64, formed exactly along rows: (X M)_ij = sum_k X_ik M_kj, M sparse),
//     X_{k+1} = X_k + X_k R_k   (dense product, split-BF16 tensor-core GEMM, FP64 update; X_k R_k
//                                is symmetric, so only its upper tiles are computed)
// converges quadratically: the relative error e_k of X_k obeys e_{k+1} <= e_k^2 + c e_k with
// c ~ 2^-16 the accuracy of one split product.  A V-cycle start leaves the smallest eigenvalue a
// of M X0 near 0.02, where plain steps only double it; so after one plain step (which puts the
// spectrum in (0, 1]) the lower end a is estimated by a few power steps on I - M X and the next
// steps are scaled (X <- alpha X (2 I - alpha M X), alpha = 2 / (1 + a)), which roughly
// quadruples a per step until it nears 1; plain quadratic steps finish.  X_k stays exactly
// symmetric (the update mirrors the upper tiles; the residual below is formed along rows, as
// R^T, which needs it); a plain iteration that stops contracting ends early so that the caller
// can fall back to a PCG solve.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "rfcmp_internal.h"

namespace rfcmp {

namespace {

// Rt[i][j] = delta_ij - alpha (X M)[i][j] with M = L + 1 1^T / n (L symmetric CSR; without
// rowsum, M = L), written as BF16 hi/lo planes; rowsum[i] = sum_j X[i][j] is precomputed.  Also
// tracks max |Rt|.  The FP64 sums bound this kernel (GB300's FP64 pipe runs at a small
// fraction of the FP32 rate), so everything else stays off that pipe: the maximum is taken on
// the FP32 value and reduced per CTA before its single atomic.  A CTA sweeps part of one row i,
// whose gathers X[i][col] the CTA's L1 keeps.
constexpr int NSR_THREADS = 256;
constexpr int NSR_SPLIT = 8;  // CTAs per row
__global__ void __launch_bounds__(NSR_THREADS)
ns_residual_kernel(const double* __restrict__ X, long long ldx, int n, const int32_t* __restrict__ ptr,
                   const int32_t* __restrict__ col, const double* __restrict__ val,
                   const double* __restrict__ rowsum, double alpha, __nv_bfloat16* __restrict__ hi,
                   __nv_bfloat16* __restrict__ lo, long long ldp, unsigned long long* __restrict__ maxbits) {
  RF_COUNT_LAUNCH();
  const int i = blockIdx.y;
  const double* xr = X + (size_t)i * ldx;
  const double rs = rowsum ? rowsum[i] / n : 0.0;  // the 1 1^T / n term of the projected case
  float mx = 0.f;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
    double a = rs;
    for (int q = ptr[j]; q < ptr[j + 1]; ++q) a += xr[col[q]] * val[q];  // (X L)_ij, L symmetric
    const double r = (i == j ? 1.0 : 0.0) - alpha * a;
    const float rf = (float)r;
    const __nv_bfloat16 h = __float2bfloat16_rn(rf);
    hi[(size_t)i * ldp + j] = h;
    lo[(size_t)i * ldp + j] = __float2bfloat16_rn(rf - __bfloat162float(h));
    mx = fmaxf(mx, fabsf(rf));
  }
  for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
  __shared__ float wmax[NSR_THREADS / 32];
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    float m = 0.f;
    for (int w = 0; w < NSR_THREADS / 32; ++w) m = fmaxf(m, wmax[w]);
    atomicMax(maxbits, (unsigned long long)__double_as_longlong((double)m));
  }
}

// ---- the same residual for the graph Laplacian (the projected case), in fixed point ----
// L has the cell's neighbour count on its diagonal and -1 per neighbour (at most three), so a row of X M
// is a sum of X entries: X is taken as integers of 2^(e - 60) (|X| < 2^(e - 1), e from the largest
// diagonal entry, which bounds a positive definite matrix), the row is staged in shared memory, and the
// sums and 1 / alpha - (X M)_ij are exact 64-bit integers.  An entry of at least 2^-6 of the largest diagonal's power
// of two converts exactly; a smaller one is rounded at 2^-59 of that power and so keeps fewer than FP64's 53 bits,
// with an absolute error below that of an FP64 sum beside a diagonal entry.  The row's sum for the 1 1^T / n term and
// the BF16 split of X, which the product after this reads, come out of the same pass (they took a pass over X each).
// Bound: the conversions and the integer sums (at 5120 cells the FP64 pipe, which converts 64-bit integers, 60 % busy,
// the integer pipe 52 %) beside DRAM, 16 bytes an entry (8 read, 4 + 4 written; 26 %); the FP64 form was bound by the
// FP64 pipe alone (90 %).  8000 cells on GB300: 0.87 ms for the three passes, 0.36 ms in this one.
// Rows longer than LAP_MAX do not fit shared memory and take the kernels around this one.
constexpr int LAP_MAX = 28900;
constexpr int FIX_BITS = 60;

// x 2^(60 - e) rounded to an integer, |x| < 2^(e - 1): the mantissa with its leading bit at bit 60, shifted
// right by the distance of x's exponent from the range's and one more; larger values and non-finite ones saturate
__device__ __forceinline__ long long to_fixed(double x, int e) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const int ex = (int)((h >> 20) & 2047u), sh = e + 1022 - ex;  // >= 1 in range
  uint32_t mh = (h & 0xfffffu) | 0x100000u, ml = l;
  mh = __funnelshift_l(ml, mh, 8);
  ml <<= 8;
  if (sh > 62) mh = ml = 0;  // below the range's last bit (zeros and subnormals among them)
  if (sh < 1) mh = 1u << 28, ml = 0;
  const int s1 = min(max(sh, 0), 62);  // one place short: the last is rounded off
  if (s1 >= 32) ml = mh, mh = 0;
  ml = __funnelshift_r(ml, mh, s1 & 31);
  mh >>= s1 & 31;
  unsigned long long v = (((unsigned long long)mh << 32 | ml) + 1ull) >> 1;
  if (sh < 1) v = 1ull << (FIX_BITS - 1);
  return (int)h < 0 ? -(long long)v : (long long)v;
}
// x rounded to FP32 from its bits (halves away from zero), zero below FP32's normal range
__device__ __forceinline__ float to_float(double x) {
  const uint32_t h = (uint32_t)__double2hiint(x), l = (uint32_t)__double2loint(x);
  const uint32_t m = __funnelshift_l(l, h & 0x7fffffffu, 3) + 0x40000000u;  // exponent rebased by 896 (mod 2^9)
  const uint32_t f = m + ((l >> 28) & 1u);
  const uint32_t ex = h & 0x7ff00000u;
  return ex < 0x38100000u ? 0.f : __uint_as_float((ex >= 0x47f00000u ? 0x7f800000u : f) | (h & 0x80000000u));
}
__device__ __forceinline__ uint32_t bf16_pair(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}
// BF16 hi and lo planes of (a, b), at words p of the rows
__device__ __forceinline__ void store_split(float a, float b, uint32_t* hi, uint32_t* lo, int p) {
  const uint32_t h = bf16_pair(a, b);
  hi[p] = h;
  lo[p] = bf16_pair(a - __uint_as_float(h << 16), b - __uint_as_float(h & 0xffff0000u));
}

// largest diagonal entry of X, by its bits (out zeroed before)
__global__ void diag_max_kernel(const double* __restrict__ X, long long ldx, int n, unsigned long long* __restrict__ out) {
  RF_COUNT_LAUNCH();
  unsigned long long m = 0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    m = max(m, (unsigned long long)__double_as_longlong(fabs(X[(size_t)i * ldx + i])));
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

// CTA per row i: Rt[i][j] = delta_ij - alpha (X M)[i][j] and X's split, as BF16 hi/lo planes; max |Rt|.
// nb: per two cells, each one's three neighbours (n where there is none) and its diagonal entry, 16 bits
// each (an index list of int4 per cell took as much of the L1 as the rest of the kernel).
__global__ void __launch_bounds__(1024, 1)
ns_residual_lap_kernel(const double* __restrict__ X, long long ldx, int n, const uint4* __restrict__ nb,
                       const unsigned long long* __restrict__ diag, double alpha, uint32_t* __restrict__ rhi,
                       uint32_t* __restrict__ rlo, uint32_t* __restrict__ xhi, uint32_t* __restrict__ xlo,
                       long long ldp, unsigned long long* __restrict__ maxbits) {
  RF_COUNT_LAUNCH();
  extern __shared__ __align__(16) long long row[];  // n + 1 entries, the last zero (n + 2 for an even n)
  __shared__ long long red[2][32];
  __shared__ long long mean;
  __shared__ float wmax[32];
  const int i = blockIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int e = max(ilogb(__longlong_as_double((long long)*diag)), -2) + 2;
  const float xs = __int_as_float((127 + e - FIX_BITS) << 23);  // 2^(e - 60); e <= 62 below any use of it
  const size_t o = (size_t)i * (ldp / 2);
  const int words = (n + 1) / 2;
  long long sh = 0, sl = 0;  // the row's sum is sh 2^32 + sl, exactly
  constexpr int B = 2;
  const double2* xr = reinterpret_cast<const double2*>(X + (size_t)i * ldx);
  for (int p0 = threadIdx.x; p0 < words; p0 += B * blockDim.x) {
    double2 x[B];
#pragma unroll
    for (int u = 0; u < B; ++u) {
      const int p = p0 + u * blockDim.x;
      x[u] = p < words ? xr[p] : make_double2(0.0, 0.0);
    }
#pragma unroll
    for (int u = 0; u < B; ++u) {
      const int p = p0 + u * blockDim.x, j = 2 * p;
      if (p >= words) break;
      if (j + 1 >= n) x[u].y = 0.0;  // the padding of an odd row
      const long long a = to_fixed(x[u].x, e), b = to_fixed(x[u].y, e);
      *reinterpret_cast<longlong2*>(row + j) = make_longlong2(a, b);  // of an odd row: also its zero entry
      sh += (a >> 32) + (b >> 32);
      sl += (long long)(a & 0xffffffffll) + (long long)(b & 0xffffffffll);
      store_split(to_float(x[u].x), to_float(x[u].y), xhi + o, xlo + o, p);
    }
  }
  for (int k = 16; k > 0; k >>= 1) {
    sh += __shfl_xor_sync(0xffffffffu, sh, k);
    sl += __shfl_xor_sync(0xffffffffu, sl, k);
  }
  if (lane == 0) {
    red[0][w] = sh;
    red[1][w] = sl;
  }
  if (threadIdx.x == 0) row[n] = 0;
  __syncthreads();
  if (threadIdx.x == 0) {
    sh = sl = 0;
    for (int k = 0; k < nw; ++k) {
      sh += red[0][k];
      sl += red[1][k];
    }
    mean = __double2ll_rn(((double)sh * 4294967296.0 + (double)sl) / n);
  }
  __syncthreads();
  const long long mu = mean, one = __double2ll_rn(ldexp(1.0 / alpha, FIX_BITS - e));
  const float rs = (float)alpha * xs;
  float mx = 0.f;
  for (int p0 = threadIdx.x; p0 < words; p0 += B * blockDim.x) {
    uint4 q[B];  // neighbours and diagonal of two cells, 16 bits each
#pragma unroll
    for (int u = 0; u < B; ++u) q[u] = nb[min(p0 + u * (int)blockDim.x, words - 1)];
#pragma unroll
    for (int u = 0; u < B; ++u) {
      const int p = p0 + u * blockDim.x;
      if (p >= words) break;
      const longlong2 own = *reinterpret_cast<const longlong2*>(row + 2 * p);
      float r[2];
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        const int j = 2 * p + z;
        const uint32_t c0 = z ? q[u].z : q[u].x, c1 = z ? q[u].w : q[u].y;
        const long long a = (long long)(c1 >> 16) * (z ? own.y : own.x) - row[c0 & 0xffffu] - row[c0 >> 16] -
                            row[c1 & 0xffffu] + mu;
        r[z] = j < n ? rs * __ll2float_rn((i == j ? one : 0ll) - a) : 0.f;
        mx = fmaxf(mx, fabsf(r[z]));
      }
      store_split(r[0], r[1], rhi + o, rlo + o, p);
    }
  }
  for (int k = 16; k > 0; k >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, k));
  if (lane == 0) wmax[w] = mx;
  __syncthreads();
  if (threadIdx.x == 0) {
    float m = 0.f;
    for (int k = 0; k < nw; ++k) m = fmaxf(m, wmax[k]);
    atomicMax(maxbits, (unsigned long long)__double_as_longlong((double)m));
  }
}

__global__ void row_sum_kernel(const double* __restrict__ X, long long ldx, int n, double* __restrict__ out) {
  RF_COUNT_LAUNCH();
  const int i = blockIdx.x;
  double s = 0.0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) s += X[(size_t)i * ldx + j];
  __shared__ double red[32];
  for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    out[i] = t;
  }
}

// out = X - shift of an exactly symmetric X, split into FP32 hi + lo planes (row stride ld): block (bx, by), by <= bx,
// reads tile (by, bx) and writes its planes there and, transposed, to tile (bx, by).
// Bound: the FP64 pipe (conversions and subtractions of an entry on or above the diagonal); 8000 rows: 0.30 ms where a pass over
// all of X and X^T took 0.71 ms.
constexpr int TT = 32;
__global__ void store_planes_kernel(const double* __restrict__ X, long long ldx, int n, double shift,
                                    float* __restrict__ hi, float* __restrict__ lo, long long ld) {
  RF_COUNT_LAUNCH();
  __shared__ float th[TT][TT + 1], tl[TT][TT + 1];
  const int bx = blockIdx.x, by = blockIdx.y;
  if (by > bx) return;
  const int r0 = by * TT, c0 = bx * TT;
  for (int r = threadIdx.y; r < TT; r += blockDim.y) {
    const int i = r0 + r, j = c0 + threadIdx.x;
    if (i >= n || j >= n) continue;
    const double v = X[(size_t)i * ldx + j] - shift;
    const float h = (float)v, l = (float)(v - (double)h);
    hi[(size_t)i * ld + j] = h;
    lo[(size_t)i * ld + j] = l;
    th[r][threadIdx.x] = h;
    tl[r][threadIdx.x] = l;
  }
  if (bx == by) return;
  __syncthreads();
  for (int r = threadIdx.y; r < TT; r += blockDim.y) {
    const int i = c0 + r, j = r0 + threadIdx.x;
    if (i >= n || j >= n) continue;
    hi[(size_t)i * ld + j] = th[threadIdx.x][r];
    lo[(size_t)i * ld + j] = tl[threadIdx.x][r];
  }
}

// X <- (X + X^T) / 2 in place: block (bx, by), by <= bx, averages tile (by, bx) with the
// transpose of tile (bx, by) and writes both
__global__ void symmetrize_inplace_kernel(double* __restrict__ X, long long ldx, int n) {
  RF_COUNT_LAUNCH();
  __shared__ double a[TT][TT + 1], b[TT][TT + 1];
  const int bx = blockIdx.x, by = blockIdx.y;
  if (by > bx) return;
  const int r0 = by * TT, c0 = bx * TT;  // tile a = X[r0.., c0..], tile b = X[c0.., r0..]
  for (int r = threadIdx.y; r < TT; r += blockDim.y) {
    const int i = r0 + r, j = c0 + threadIdx.x;
    a[r][threadIdx.x] = (i < n && j < n) ? X[(size_t)i * ldx + j] : 0.0;
    const int i2 = c0 + r, j2 = r0 + threadIdx.x;
    b[r][threadIdx.x] = (i2 < n && j2 < n) ? X[(size_t)i2 * ldx + j2] : 0.0;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < TT; r += blockDim.y) {
    const int i = r0 + r, j = c0 + threadIdx.x;
    const double v = 0.5 * (a[r][threadIdx.x] + b[threadIdx.x][r]);
    if (i < n && j < n) X[(size_t)i * ldx + j] = v;
    const int i2 = c0 + r, j2 = r0 + threadIdx.x;
    const double w = 0.5 * (b[r][threadIdx.x] + a[threadIdx.x][r]);
    if (i2 < n && j2 < n) X[(size_t)i2 * ldx + j2] = w;
  }
}

// hi + lo <- (M + M^T) / 2 of M = hi + lo in place, tiles paired as above: a factor whose columns were solved one
// by one is symmetric only to the solver's tolerance, and the streaming products read its upper triangle
__global__ void symmetrize_planes_kernel(float* __restrict__ hi, float* __restrict__ lo, long long ld, int n) {
  RF_COUNT_LAUNCH();
  __shared__ double a[TT][TT + 1], b[TT][TT + 1];
  const int bx = blockIdx.x, by = blockIdx.y;
  if (by > bx) return;
  const int r0 = by * TT, c0 = bx * TT;
  auto get = [&](int i, int j) {
    const size_t at = (size_t)i * ld + j;
    return i < n && j < n ? (double)hi[at] + (double)lo[at] : 0.0;
  };
  auto put = [&](int i, int j, double v) {
    if (i >= n || j >= n) return;
    const float h = (float)v;
    hi[(size_t)i * ld + j] = h;
    lo[(size_t)i * ld + j] = (float)(v - (double)h);
  };
  for (int r = threadIdx.y; r < TT; r += blockDim.y) {
    a[r][threadIdx.x] = get(r0 + r, c0 + threadIdx.x);
    b[r][threadIdx.x] = get(c0 + r, r0 + threadIdx.x);
  }
  __syncthreads();
  for (int r = threadIdx.y; r < TT; r += blockDim.y) {
    put(r0 + r, c0 + threadIdx.x, 0.5 * (a[r][threadIdx.x] + b[threadIdx.x][r]));
    put(c0 + r, r0 + threadIdx.x, 0.5 * (b[r][threadIdx.x] + a[threadIdx.x][r]));
  }
}

// ---------------------------------------------------------------- one V-cycle as a matrix
// A V(1,1) cycle with Jacobi smoothing is M_l = S M_{l+1} S^T + 2 w D^{-1} - w^2 D^{-1} A D^{-1} with the sparse
// S = (I - w D^{-1} A) P (three to five entries a row) and M_L the coarsest inverse, so the dense cycle is built
// from the coarsest level up and every level touches only its own n_l x n_l entries.
//
// Bound: the FP64 pipe (about 4.5 fused operations an entry on and above the diagonal, as many for the n_l x
// n_{l+1} products) and the 8 n^2 bytes written.  A CTA takes RB rows: it forms their rows of S M_{l+1} in shared
// memory, then each thread a column j >= i of S M_{l+1} S^T; the mirrored entries go out as runs of RB.  Applying
// the cycle to the n columns of I - J (six n x n arrays, each smoothing and transfer a pass over them, a division
// per row and column pair) took 5.3 ms of 8000 cells; the factor's build went from 32 to 27 ms.
constexpr int LIFT_THREADS = 512;
constexpr int LIFT_SMEM = 220 * 1024;
struct LiftLevel {
  const int32_t *sp, *sc, *ap, *ac;
  const double *sv, *av, *diag;
  double omega;
  int n, nc;
};

// shift (or null): 1 / n^2 of the sum of the n values behind it, then those values, the row sums of M
template <int RB>
__global__ void __launch_bounds__(LIFT_THREADS)
mg_lift_kernel(LiftLevel L, const double* __restrict__ Mc, long long ldc, const double* __restrict__ shift,
               double* __restrict__ M, long long ld) {
  RF_COUNT_LAUNCH();
  extern __shared__ __align__(32) double u[];  // [nc][RB]
  const int n = L.n, i0 = blockIdx.x * RB;
  for (int K = threadIdx.x; K < L.nc; K += LIFT_THREADS)
#pragma unroll
    for (int r = 0; r < RB; ++r) {
      double a = 0.0;
      if (i0 + r < n)
        for (int q = L.sp[i0 + r]; q < L.sp[i0 + r + 1]; ++q) a = fma(L.sv[q], Mc[(size_t)L.sc[q] * ldc + K], a);
      u[(size_t)K * RB + r] = a;
    }
  __syncthreads();
  const double inv = shift ? -1.0 / n : 0.0;
  double base[RB];
#pragma unroll
  for (int r = 0; r < RB; ++r)
    base[r] = shift && i0 + r < n ? fma(shift[1 + i0 + r], inv, fma(shift[0], inv * inv, -inv)) : 0.0;
  for (int j = i0 + threadIdx.x; j < n; j += LIFT_THREADS) {
    double a[RB];
    const double sj = shift ? shift[1 + j] : 0.0;
#pragma unroll
    for (int r = 0; r < RB; ++r) a[r] = fma(sj, inv, base[r]);
    for (int q = L.sp[j]; q < L.sp[j + 1]; ++q) {
      const double v = L.sv[q];
      const double* w = u + (size_t)L.sc[q] * RB;
      if constexpr (RB == 4) {
        const double2 w0 = *reinterpret_cast<const double2*>(w), w1 = *reinterpret_cast<const double2*>(w + 2);
        a[0] = fma(v, w0.x, a[0]);
        a[1] = fma(v, w0.y, a[1]);
        a[2] = fma(v, w1.x, a[2]);
        a[3] = fma(v, w1.y, a[3]);
      } else {
#pragma unroll
        for (int r = 0; r < RB; ++r) a[r] = fma(v, w[r], a[r]);
      }
    }
    for (int q = L.ap[j]; q < L.ap[j + 1]; ++q) {
      const int r = L.ac[q] - i0;
      if (r < 0 || r >= RB) continue;
      const double fj = L.omega / L.diag[j];
      double t = -fj * (L.omega / L.diag[i0 + r]) * L.av[q];
      if (i0 + r == j) t += 2.0 * fj;
#pragma unroll
      for (int e = 0; e < RB; ++e)
        if (e == r) a[e] += t;
    }
#pragma unroll
    for (int r = 0; r < RB; ++r)
      if (i0 + r <= j) M[(size_t)(i0 + r) * ld + j] = a[r];
    double* m = M + (size_t)j * ld + i0;
    if (RB > 1 && j >= i0 + RB) {
#pragma unroll
      for (int r = 0; r + 1 < RB; r += 2) *reinterpret_cast<double2*>(m + r) = make_double2(a[r], a[r + (RB > 1)]);
    } else {
#pragma unroll
      for (int r = 0; r < RB; ++r)
        if (i0 + r < j) m[r] = a[r];
    }
  }
}

// z = M y, one warp a row
__global__ void mg_rows_kernel(const double* __restrict__ M, long long ld, int n, const double* __restrict__ y,
                               double* __restrict__ z) {
  RF_COUNT_LAUNCH();
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (i >= n) return;
  double a = 0.0;
  for (int j = lane; j < n; j += 32) a = fma(M[(size_t)i * ld + j], y[j], a);
  for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
  if (lane == 0) z[i] = a;
}

// row sums of M_l, shift[1 + i] = (S z)_i + 2 f_i - f_i sum_j A_ij f_j with f = w / D; shift[0] += each
__global__ void mg_row_sum_kernel(LiftLevel L, const double* __restrict__ z, double* __restrict__ shift) {
  RF_COUNT_LAUNCH();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double a = 0.0;
  if (i < L.n) {
    for (int q = L.sp[i]; q < L.sp[i + 1]; ++q) a = fma(L.sv[q], z[L.sc[q]], a);
    double b = 0.0;
    for (int q = L.ap[i]; q < L.ap[i + 1]; ++q) b = fma(L.av[q], L.omega / L.diag[L.ac[q]], b);
    const double f = L.omega / L.diag[i];
    a += f * (2.0 - b);
    shift[1 + i] = a;
  }
  for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
  if ((threadIdx.x & 31) == 0) atomicAdd(shift, a);
}

template <int RB>
cudaError_t lift(const LiftLevel& L, const double* Mc, long long ldc, const double* shift, double* M, long long ld,
                 cudaStream_t s) {
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, [] {
    attr = cudaFuncSetAttribute(mg_lift_kernel<RB>, cudaFuncAttributeMaxDynamicSharedMemorySize, LIFT_SMEM);
  });
  if (attr != cudaSuccess) return attr;
  mg_lift_kernel<RB><<<(L.n + RB - 1) / RB, LIFT_THREADS, sizeof(double) * RB * (size_t)L.nc, s>>>(L, Mc, ldc, shift, M, ld);
  return cudaGetLastError();
}

// X <- alpha (X + D) for an exactly symmetric X and a symmetric D of which only the 128 x 128 tiles on or above the
// diagonal were computed: block (bx, by), by <= bx, updates tile (by, bx) of X and writes it there and, transposed,
// to tile (bx, by); a diagonal tile adds (D + D^T) / 2, so X stays exactly symmetric.  !SCALED: alpha = 1 (a plain
// step), one FP64 operation fewer per entry.
// Bound: HBM (X read once on and above the diagonal, D, X written).  8000 rows: 0.18 ms plain and 0.19 scaled; reading
// both triangles and updating each entry of both, 0.30 and 0.42 ms, FP64 pipe.
template <bool SCALED>
__global__ void ns_update_sym_kernel(double* __restrict__ X, long long ldx, const float* __restrict__ D, long long ldd,
                                     int n, double alpha) {
  RF_COUNT_LAUNCH();
  __shared__ double t[TT][TT + 1];
  const int bx = blockIdx.x, by = blockIdx.y;
  if (by > bx) return;
  const int r0 = by * TT, c0 = bx * TT, c = threadIdx.x;
  if (bx == by) {
    for (int r = threadIdx.y; r < TT; r += blockDim.y)
      t[r][c] = r0 + r < n && c0 + c < n ? (double)D[(size_t)(r0 + r) * ldd + c0 + c] : 0.0;
    __syncthreads();
    for (int r = threadIdx.y; r < TT; r += blockDim.y) {
      if (r0 + r >= n || c0 + c >= n) continue;
      double* x = X + (size_t)(r0 + r) * ldx + c0 + c;
      const double v = *x + 0.5 * (t[r][c] + t[c][r]);
      *x = SCALED ? alpha * v : v;
    }
    return;
  }
  for (int r = threadIdx.y; r < TT; r += blockDim.y) {
    const int i = r0 + r, j = c0 + c;
    if (i >= n || j >= n) continue;
    double* x = X + (size_t)i * ldx + j;
    double v = *x + (double)D[(size_t)i * ldd + j];
    if (SCALED) v *= alpha;
    *x = v;
    t[r][c] = v;
  }
  __syncthreads();
  for (int r = threadIdx.y; r < TT; r += blockDim.y) {
    const int i = c0 + r, j = r0 + c;
    if (i < n && j < n) X[(size_t)i * ldx + j] = t[c][r];
  }
}

// u = X v (dense FP64, one warp per row); sum += sum_i u_i
__global__ void dmatvec_kernel(const double* __restrict__ X, long long ldx, int n, const double* __restrict__ v,
                               double* __restrict__ u, double* __restrict__ sum) {
  RF_COUNT_LAUNCH();
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (warp >= n) return;
  const double* xr = X + (size_t)warp * ldx;
  double a = 0.0;
  for (int j = lane; j < n; j += 32) a = fma(xr[j], v[j], a);
  for (int off = 16; off > 0; off >>= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
  if (lane == 0) {
    u[warp] = a;
    atomicAdd(sum, a);
  }
}

// w = v - (L u + (sum / n) 1 if project); norm2 += |w|^2
__global__ void resid_vec_kernel(const int32_t* __restrict__ ptr, const int32_t* __restrict__ col,
                                 const double* __restrict__ val, int n, int project, const double* __restrict__ v,
                                 const double* __restrict__ u, const double* __restrict__ sum,
                                 double* __restrict__ w, double* __restrict__ norm2) {
  RF_COUNT_LAUNCH();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double d = 0.0;
  if (i < n) {
    double a = project ? *sum / n : 0.0;
    for (int q = ptr[i]; q < ptr[i + 1]; ++q) a += val[q] * u[col[q]];
    const double r = v[i] - a;
    w[i] = r;
    d = r * r;
  }
  for (int off = 16; off > 0; off >>= 1) d += __shfl_xor_sync(0xffffffffu, d, off);
  if ((threadIdx.x & 31) == 0) atomicAdd(norm2, d);
}

__global__ void scale_vec_kernel(int n, double c, const double* __restrict__ w, double* __restrict__ v) {
  RF_COUNT_LAUNCH();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) v[i] = c * w[i];
}

// X = c D^{-1} (D the diagonal of the CSR matrix), the rest of X zero
__global__ void jacobi_start_kernel(const int32_t* __restrict__ ptr, const int32_t* __restrict__ col,
                                    const double* __restrict__ val, int n, double c, double* __restrict__ X,
                                    long long ldx) {
  RF_COUNT_LAUNCH();
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double d = 0.0;
    for (int q = ptr[i]; q < ptr[i + 1]; ++q)
      if (col[q] == i) d = val[q];
    X[(size_t)i * ldx + i] = d > 0.0 ? c / d : 0.0;
  }
}

}  // namespace

cudaError_t jacobi_start(const int32_t* ptr, const int32_t* col, const double* val, int n, double c, double* X,
                         long long ldx, cudaStream_t s) {
  cudaError_t err = cudaMemsetAsync(X, 0, sizeof(double) * (size_t)n * ldx, s);
  if (err != cudaSuccess) return err;
  jacobi_start_kernel<<<(n + 255) / 256, 256, 0, s>>>(ptr, col, val, n, c, X, ldx);
  return cudaGetLastError();
}

cudaError_t newton_schulz_pseudo_inverse(const int32_t* ptr, const int32_t* col, const double* val, const uint4* lap,
                                         int n, bool project, bool symmetric, double* X, long long ldx, int max_steps, double tol, float* Xhi,
                                         float* Xlo, int* steps_done, double* final_residual, cudaStream_t s) {
  // X holds an approximation of M^{-1} on entry (row-major, stride ldx): M = L + 1 1^T / n with
  // project (the result is M^{-1} - 1 1^T / n = L^+), M = L without
  const long long ldp = ldx;  // plane stride (elements); ldx is a multiple of 64
  std::vector<void*> own;
  auto fail = [&](cudaError_t e) {
    for (void* p : own) dev_free(p);
    return e;
  };
  cudaError_t err;
  __nv_bfloat16 *xh, *xl, *rh, *rl;
  float* D;
  double* rowsum;
  unsigned long long* maxbits;  // max |R| and, for the fixed-point residual, the largest diagonal entry of X
  int* gerr;
  const bool fixed = project && lap && n <= LAP_MAX;
  const size_t lap_smem = ((size_t)n + 2) * sizeof(long long);
  if (fixed) {
    static std::once_flag once;
    static cudaError_t attr = cudaSuccess;
    std::call_once(once, [] {
      attr = cudaFuncSetAttribute(ns_residual_lap_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (LAP_MAX + 2) * (int)sizeof(long long));
    });
    if (attr != cudaSuccess) return attr;
  }
  const size_t plane = (size_t)n * ldp;
  for (__nv_bfloat16** p : {&xh, &xl, &rh, &rl}) {
    if ((err = dev_malloc(p, plane * sizeof(__nv_bfloat16))) != cudaSuccess) return fail(err);
    own.push_back(*p);
  }
  if ((err = dev_malloc(&D, plane * sizeof(float))) != cudaSuccess) return fail(err);
  own.push_back(D);
  if ((err = dev_malloc(&rowsum, n * sizeof(double))) != cudaSuccess) return fail(err);
  own.push_back(rowsum);
  if ((err = dev_malloc(&maxbits, 2 * sizeof(unsigned long long))) != cudaSuccess) return fail(err);
  own.push_back(maxbits);
  if ((err = dev_malloc(&gerr, sizeof(int))) != cudaSuccess) return fail(err);
  own.push_back(gerr);
  if ((err = cudaMemsetAsync(gerr, 0, sizeof(int), s)) != cudaSuccess) return fail(err);
  SplitOperand A, B;
  A.hi = xh;
  A.lo = xl;
  A.rows = n;
  A.ld = ldp;
  B.hi = rh;
  B.lo = rl;
  B.rows = n;
  B.ld = ldp;
  // vectors of the spectral-radius estimate: v, u, w (n each) and two scalars
  double* pv;
  if ((err = dev_malloc(&pv, (3 * (size_t)n + 2) * sizeof(double))) != cudaSuccess) return fail(err);
  own.push_back(pv);
  double *pu = pv + n, *pw = pv + 2 * (size_t)n, *psc = pv + 3 * (size_t)n;
  // rho(I - M X) by a few power steps on I - M X (matrix-free: one dense FP64 product with X and
  // one sparse product with M per step).  Any bound a in (0, 1) keeps the scaled steps
  // convergent.
  auto estimate_rho = [&](double& rho) -> cudaError_t {
    std::vector<double> h(n);
    for (int i = 0; i < n; ++i) h[i] = 1.0 + 0.5 * std::sin(0.7 * i) + 0.25 * std::cos(1.3 * i + 0.4);
    double nrm = 0.0;
    for (double x : h) nrm += x * x;
    for (double& x : h) x /= std::sqrt(nrm);
    cudaError_t e;
    if ((e = cudaMemcpyAsync(pv, h.data(), n * sizeof(double), cudaMemcpyHostToDevice, s)) != cudaSuccess) return e;
    rho = 0.0;
    for (int it = 0; it < 12; ++it) {
      if ((e = cudaMemsetAsync(psc, 0, 2 * sizeof(double), s)) != cudaSuccess) return e;
      dmatvec_kernel<<<(n * 32 + 255) / 256, 256, 0, s>>>(X, ldx, n, pv, pu, psc);
      resid_vec_kernel<<<(n + 255) / 256, 256, 0, s>>>(ptr, col, val, n, project ? 1 : 0, pv, pu, psc, pw, psc + 1);
      double nw2 = 0.0;
      if ((e = cudaMemcpyAsync(&nw2, psc + 1, sizeof(double), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
      if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
      rho = std::sqrt(nw2);
      if (!(rho > 0.0)) break;
      scale_vec_kernel<<<(n + 255) / 256, 256, 0, s>>>(n, 1.0 / rho, pw, pv);
    }
    return cudaGetLastError();
  };
  double res = 1.0, prev = 1.0;
  bool prev_plain = false;
  double alpha = 1.0, a = -1.0;  // scaling of the next step; lower bound on the spectrum of M X
  int k = 0;
  const dim3 sgrid((n + TT - 1) / TT, (n + TT - 1) / TT), sblock(TT, 8);
  // the residual below is formed along rows as I - X M, which is R^T only for symmetric X
  if (!symmetric) symmetrize_inplace_kernel<<<sgrid, sblock, 0, s>>>(X, ldx, n);
  for (;; ++k) {
    if (project && !fixed) row_sum_kernel<<<n, 256, 0, s>>>(X, ldx, n, rowsum);
    if ((err = cudaMemsetAsync(maxbits, 0, 2 * sizeof(unsigned long long), s)) != cudaSuccess) return fail(err);
    if (fixed) {
      ProfScope prof("factor_ns_residual", 16.0 * (double)n * n, 0.0, s);
      diag_max_kernel<<<std::min((n + 255) / 256, 64), 256, 0, s>>>(X, ldx, n, maxbits + 1);
      // two or more rows share an SM up to 14000 cells; a longer row gets twice the threads
      ns_residual_lap_kernel<<<n, n <= 14000 ? 512 : 1024, lap_smem, s>>>(
          X, ldx, n, lap, maxbits + 1, alpha, reinterpret_cast<uint32_t*>(rh), reinterpret_cast<uint32_t*>(rl),
          reinterpret_cast<uint32_t*>(xh), reinterpret_cast<uint32_t*>(xl), ldp, maxbits);
    } else {
      ProfScope prof("factor_ns_residual", 12.0 * (double)n * n, 0.0, s);
      dim3 grid(std::min((n + NSR_THREADS - 1) / NSR_THREADS, NSR_SPLIT), n);
      ns_residual_kernel<<<grid, NSR_THREADS, 0, s>>>(X, ldx, n, ptr, col, val, project ? rowsum : nullptr, alpha, rh, rl,
                                              ldp, maxbits);
    }
    unsigned long long hb = 0;
    if ((err = cudaMemcpyAsync(&hb, maxbits, sizeof(hb), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return fail(err);
    if ((err = cudaStreamSynchronize(s)) != cudaSuccess) return fail(err);
    const bool plain = alpha == 1.0;
    if (plain) {  // the residual of the current iterate: stop and contraction checks
      std::memcpy(&res, &hb, sizeof(res));
      if (!(res > tol)) break;
      if (prev_plain && k >= 2 && !(res < 0.9 * prev)) break;  // not contracting: the caller falls back
      prev = res;
    }
    prev_plain = plain;
    if (k >= max_steps) break;
    if (!fixed && (err = split_bf16_f64(X, ldx, n, n, xh, xl, ldp, s)) != cudaSuccess) return fail(err);
    // D = X R' with B = R'^T stored row-major, R' = I - alpha M X; X R' is symmetric, so only the
    // tiles on and above the diagonal are computed; then X <- alpha (X + D)
    if ((err = gemm_bf16x3(&A, &B, nullptr, 1, n, n, n, D, ldp, false, gerr, s, 0, true)) != cudaSuccess)
      return fail(err);
    {
      ProfScope prof("factor_ns_update", 12.0 * (double)n * n, 0.0, s);
      if (alpha == 1.0) ns_update_sym_kernel<false><<<sgrid, sblock, 0, s>>>(X, ldx, D, ldp, n, alpha);
      else ns_update_sym_kernel<true><<<sgrid, sblock, 0, s>>>(X, ldx, D, ldp, n, alpha);
    }
    if ((err = cudaGetLastError()) != cudaSuccess) return fail(err);
    // scaling of the next step (scaled Newton-Schulz): with the spectrum of M X in [a, 1], the
    // step X <- alpha X (2 I - alpha M X), alpha = 2 / (1 + a), maps it into [a', 1] with
    // a' = alpha a (2 - alpha a), which grows about four-fold per step while a is small
    if (k == 0) {  // after one plain step the spectrum lies in (0, 1]: estimate its lower end
      double rho = 1.0;
      if ((err = estimate_rho(rho)) != cudaSuccess) return fail(err);
      // the power steps approach rho from below, so 1 - rho can overstate the true lower end;
      // an overstated bound ends the scaled steps too early, an understated one only costs a
      // fraction of a step (the bound roughly quadruples per step), so take half of it
      a = 0.5 * (1.0 - rho);
    } else if (!plain) {
      a = alpha * a * (2.0 - alpha * a);
    }
    alpha = (a > 1e-6 && a < 0.95) ? 2.0 / (1.0 + a) : 1.0;
  }
  int herr = 0;
  if ((err = cudaMemcpyAsync(&herr, gerr, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess) return fail(err);
  {
    dim3 grid((n + TT - 1) / TT, (n + TT - 1) / TT), block(TT, 8);
    store_planes_kernel<<<grid, block, 0, s>>>(X, ldx, n, project ? 1.0 / n : 0.0, Xhi, Xlo, ldx);
  }
  if ((err = cudaStreamSynchronize(s)) != cudaSuccess) return fail(err);
  if (herr) return fail(cudaErrorLaunchTimeout);
  *steps_done = k;
  *final_residual = res;
  return fail(cudaSuccess);
}

cudaError_t multigrid_inverse(const AmgHierarchy& H, int n, double* X, long long ld, bool* done, cudaStream_t s,
                              int rows) {
  *done = false;
  if (H.levels.empty() || rows < 1) return cudaSuccess;
  for (const AmgLevelHost& h : H.levels)
    if (sizeof(double) * (size_t)h.nc > (size_t)LIFT_SMEM) return cudaSuccess;
  *done = true;
  ProfScope prof("factor_mg_vcycle", 8.0 * (double)n * n, 0.0, s);
  // the hierarchy in one buffer
  std::vector<char> buf;
  auto put = [&](const void* p, size_t bytes) {
    const size_t at = (buf.size() + 15) / 16 * 16;
    buf.resize(at + bytes);
    std::memcpy(buf.data() + at, p, bytes);
    return at;
  };
  auto ints = [&](const std::vector<int32_t>& v) { return put(v.data(), v.size() * sizeof(int32_t)); };
  auto dbls = [&](const std::vector<double>& v) { return put(v.data(), v.size() * sizeof(double)); };
  struct At {
    size_t sp, sc, sv, ap, ac, av, diag;
  };
  std::vector<At> at;
  for (const AmgLevelHost& h : H.levels)
    at.push_back({ints(h.S_ptr), ints(h.S_col), dbls(h.S_val), ints(h.A_ptr), ints(h.A_col), dbls(h.A_val), dbls(h.diag)});
  const size_t at_inv = dbls(H.coarse_inv), at_y = dbls(H.levels[0].S_colsum);
  std::vector<void*> own;
  cudaError_t err = cudaSuccess;
  auto fail = [&](cudaError_t e) {
    for (void* p : own) dev_free(p);
    return e;
  };
  auto get = [&](auto** p, size_t bytes) {
    err = dev_malloc(p, bytes);
    if (err == cudaSuccess) own.push_back(*p);
    return err == cudaSuccess;
  };
  char* d = nullptr;
  double *z = nullptr, *shift = nullptr;
  if (!get(&d, buf.size()) || !get(&z, sizeof(double) * (size_t)H.levels[0].nc) ||
      !get(&shift, sizeof(double) * ((size_t)n + 1)))
    return fail(err);
  if ((err = cudaMemcpyAsync(d, buf.data(), buf.size(), cudaMemcpyHostToDevice, s)) != cudaSuccess) return fail(err);
  if ((err = cudaMemsetAsync(shift, 0, sizeof(double), s)) != cudaSuccess) return fail(err);
  const double* Mc = reinterpret_cast<const double*>(d + at_inv);
  long long ldc = H.coarse_n;
  for (int l = (int)H.levels.size() - 1; l >= 0; --l) {
    const AmgLevelHost& h = H.levels[l];
    const At& a = at[l];
    auto I = [&](size_t o) { return reinterpret_cast<const int32_t*>(d + o); };
    auto D = [&](size_t o) { return reinterpret_cast<const double*>(d + o); };
    const LiftLevel L{I(a.sp), I(a.sc), I(a.ap), I(a.ac), D(a.sv), D(a.av), D(a.diag), h.omega, h.n, h.nc};
    double* M = X;
    long long ldm = ld;
    if (l > 0) {
      ldm = (h.n + 1) / 2 * 2;
      if (!get(&M, sizeof(double) * (size_t)h.n * ldm)) return fail(err);
    } else {
      mg_rows_kernel<<<(h.nc + 7) / 8, 256, 0, s>>>(Mc, ldc, h.nc, D(at_y), z);
      mg_row_sum_kernel<<<(n + 127) / 128, 128, 0, s>>>(L, z, shift);
    }
    const double* sh = l == 0 ? shift : nullptr;
    // four rows share the entries of S (and write whole sectors of the mirrored rows) where they fit
    const size_t row = sizeof(double) * (size_t)h.nc;
    err = rows >= 4 && 4 * row <= (size_t)LIFT_SMEM   ? lift<4>(L, Mc, ldc, sh, M, ldm, s)
          : rows >= 2 && 2 * row <= (size_t)LIFT_SMEM ? lift<2>(L, Mc, ldc, sh, M, ldm, s)
                                                      : lift<1>(L, Mc, ldc, sh, M, ldm, s);
    if (err != cudaSuccess) return fail(err);
    Mc = M;
    ldc = ldm;
  }
  // pageable host memory: the copy has been staged; the frees follow the queued work
  return fail(cudaSuccess);
}

cudaError_t symmetrize_planes(float* hi, float* lo, int n, int ld, cudaStream_t s) {
  const dim3 grid((n + TT - 1) / TT, (n + TT - 1) / TT), block(TT, 8);
  symmetrize_planes_kernel<<<grid, block, 0, s>>>(hi, lo, ld, n);
  return cudaGetLastError();
}

RF_LAUNCH_READER(launches_factor)

}  // namespace rfcmp
