// Exact-digit GEMM: float-float accurate multi-column products on the tensor cores.
//
// The refinement residual r = b - A i and the right-hand side b need products about 40 bits
// accurate, where the split-BF16 GEMM gives 16 and a float-float GEMV costs some 40 FP32
// instructions per complex multiply-add.  Here every row of an operand (a row of the matrix, or
// a column of the right-hand-side block) is scaled by a power of two 2^e that puts its entries
// in [-1/2, 1/2] and written as S = 6 signed 8-bit digits
//
//     v = 2^e sum_{s<S} d_s 256^-(s+1),   d_s integer, |d_s| <= 128,
//
// every digit exact in BF16.  A product of two digits is an integer of magnitude at most 2^14,
// so the level sums P_L = sum_{s+t=L} D_s E_t^T over a K-block of KB = 128 columns stay below
// 6 * 128 * 2^14 < 2^24 and the FP32 tensor-memory accumulators hold them exactly, whatever
// the order of the additions.  After every K-block the epilogue warps fold the level sums into
// two 64-bit integer accumulators per output, H += P_0 2^16 + P_1 2^8 + P_2 and
// G += P_3 2^16 + P_4 2^8 + P_5, and at the end
//     D = 2^(eA_i + eB_j) 2^-56 (2^24 H + G)
// is rounded once to FP64.  Digit pairs of level S and beyond are dropped together with the
// digits past S: per term a truncation of about 2^-48 of the row scale times the column scale,
// the only error of the product.
//
// Kernel layout: one CTA per 128 x 32 output tile, 320 threads.  Warp 0 lane 0 issues the TMA
// loads of a 3-stage ring (each stage: the S digit planes of A, 128 x 32, and the S of B, 32 x 32,
// BF16 with the 64-byte swizzle; the B planes lie back to back, so B_0..B_t read as one operand
// of 32 (t + 1) rows).  Warp 1 lane 0 issues, per 16-wide K step, one MMA per A plane s against
// B_0..B_{S-1-s}: its N = 32 (S - s) output columns land on the accumulators of levels s..S-1,
// which sit side by side in tensor memory (level L at column 32 L), so S MMAs cover all S(S+1)/2
// digit pairs and every A plane is read from shared memory once per K step.  Two sets of level
// accumulators alternate between K-blocks; warps 2..9 fold a finished K-block (two warps per
// 32-lane quadrant of tensor memory, 16 columns each) while the next one accumulates, and write D.  Every wait
// is bounded; on timeout the kernel records an error code, frees its tensor memory and returns.
//
// Up to XI_COLS columns D is the pair of integers (H, G) itself, scaled and combined by the kernel
// after it.  The integer sums are exact, so the K range of a tile can be split over CTAs that add
// theirs with 64-bit atomics (any order, the same bits): a matrix of few row tiles still fills the
// chip.  16 columns on GB300: a factor of 5120 cells (40 tiles, split 3) 136 -> 66 us, V (80 tiles,
// split 5) 160 -> 121 us, T_A of 7680 functions (120 tiles) unchanged at 237 us, where the digit
// planes take 209 us to leave HBM.
#include <cuda.h>
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstring>
#include <mutex>

#include "rfcmp_internal.h"
#include "tc_common.cuh"

namespace rfcmp {

namespace {

using namespace tc;

constexpr int XS = EXACT_DIGITS;  // digits per value
static_assert(XS == 6, "the integer fold below is written for 6 digits");
constexpr int XBN = 32;           // output columns per CTA
constexpr int XBK = 32;           // K per ring step (64-byte rows)
constexpr int XKB = 128;          // K-block between integer folds
constexpr int XSTAGES = 3;
constexpr int XSPK = XKB / XBK;   // ring steps per K-block
constexpr int XTILE_A = BM * XBK * 2;
constexpr int XTILE_B = XBN * XBK * 2;
constexpr int XSTAGE = XS * (XTILE_A + XTILE_B);
constexpr int XSMEM = XSTAGES * XSTAGE + 1024 + 256;
constexpr int XBUF = XS * XBN;  // tensor-memory columns of one set of level accumulators
constexpr uint32_t XTMEM_COLS = 2 * XBUF <= 128 ? 128 : (2 * XBUF <= 256 ? 256 : 512);
static_assert(2 * XBUF <= 512, "level accumulators exceed tensor memory");
static_assert(XS * XBN <= 256, "one MMA spans the accumulators of all levels");
static_assert((long long)XS * (128LL * 128LL) * XKB < (1LL << 24), "K-block level sums must stay exact in FP32");
static_assert(XSMEM <= 227 * 1024, "shared memory");
static_assert(XKB % XBK == 0 && XTILE_B % 512 == 0 && XTILE_A % 1024 == 0, "tile geometry");

struct ExactMaps {
  CUtensorMap a[XS];
  CUtensorMap b[XS];
};

constexpr int XTHREADS = 320;  // producer warp, MMA warp, 8 epilogue warps
static_assert(XBN == 32, "two epilogue warps of 16 columns per tensor-memory quadrant");

constexpr int NOT_FINITE = INT_MIN;  // exponent of a column with an infinity or a NaN: its products are NaN
__device__ __forceinline__ double quiet_nan() { return __longlong_as_double(0x7ff8000000000000ll); }

__global__ void __launch_bounds__(XTHREADS, 1)
exact_gemm_kernel(const __grid_constant__ ExactMaps maps, int M, int N, int K, const int* __restrict__ ea,
                  const int* __restrict__ eb, double* __restrict__ D, longlong2* __restrict__ DI, long long ldd,
                  int* __restrict__ err) {
  RF_COUNT_LAUNCH();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + XSTAGES * XSTAGE);
  uint64_t* empty = full + XSTAGES;
  uint64_t* acc_full = empty + XSTAGES;  // [2]
  uint64_t* acc_empty = acc_full + 2;    // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n0 = blockIdx.x * XBN, m0 = blockIdx.y * BM;  // N tiles fastest: CTAs sharing A run together
  const int all_steps = (K + XBK - 1) / XBK, all_kb = (all_steps + XSPK - 1) / XSPK;
  // this CTA's K-blocks [kb0, kb1)
  const int kb0 = (int)((long long)all_kb * blockIdx.z / gridDim.z);
  const int kb1 = (int)((long long)all_kb * (blockIdx.z + 1) / gridDim.z);
  const int step0 = kb0 * XSPK, ksteps = min(kb1 * XSPK, all_steps) - step0, nkb = kb1 - kb0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < XSTAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 8);  // one arrival per epilogue warp
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(XTMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0) {
    if (lane == 0) {
      for (int it = 0; it < ksteps; ++it) {
        const int s = it % XSTAGES, round = it / XSTAGES;
        if (round > 0 && !mbar_wait(&empty[s], (round - 1) & 1)) {
          atomicExch(err, 11);
          break;
        }
        uint8_t* st = smem + s * XSTAGE;
        const int kx = (step0 + it) * XBK;
        mbar_expect_tx(&full[s], XSTAGE);
#pragma unroll
        for (int p = 0; p < XS; ++p) tma_load_2d(st + p * XTILE_A, &maps.a[p], &full[s], kx, m0);
#pragma unroll
        for (int p = 0; p < XS; ++p) tma_load_2d(st + XS * XTILE_A + p * XTILE_B, &maps.b[p], &full[s], kx, n0);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      for (int it = 0; it < ksteps; ++it) {
        const int s = it % XSTAGES, round = it / XSTAGES;
        const int kb = it / XSPK, buf = kb & 1;
        const bool first = (it % XSPK) == 0;
        // this buffer's level sums of K-block kb - 2 must have been folded
        if (first && kb >= 2 && !mbar_wait(&acc_empty[buf], ((kb >> 1) - 1) & 1)) {
          atomicExch(err, 12);
          break;
        }
        if (!mbar_wait(&full[s], round & 1)) {
          atomicExch(err, 13);
          break;
        }
        tc_fence_after();
        const uint32_t a0 = smem_u32(smem + s * XSTAGE), b0 = a0 + XS * XTILE_A;
        const uint32_t t0 = tmem + (uint32_t)(buf * XBUF);
#pragma unroll
        for (int kk = 0; kk < XBK / 16; ++kk) {
          const uint32_t off = kk * 32;  // 16 BF16 along K inside the 64-byte swizzled row
          const uint64_t bd = sw64_desc(b0 + off);
#pragma unroll
          for (int sa = 0; sa < XS; ++sa)
            mma_bf16(t0 + (uint32_t)(sa * XBN), sw64_desc(a0 + sa * XTILE_A + off), bd,
                     idesc_bf16(BM, (XS - sa) * XBN, false), (first && kk == 0 && sa == 0) ? 0u : 1u);
        }
        mma_commit(&empty[s]);
        if ((it % XSPK) == XSPK - 1 || it == ksteps - 1) mma_commit(&acc_full[buf]);
      }
    }
  } else {
    // epilogue warps 2..9: warp w reads tensor-memory lanes 32 (w % 4) .. 32 (w % 4) + 31 and
    // folds output columns 16 h .. 16 h + 15, h = (w - 2) / 4
    const int q = warp & 3, h = ((warp - 2) >> 2) * 16;
    const int row = m0 + 32 * q + lane;
    long long H[16], G[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) H[j] = G[j] = 0;
    bool ok = true;
    for (int kb = 0; kb < nkb; ++kb) {
      const int buf = kb & 1;
      ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[buf], (kb >> 1) & 1));
      if (!ok) {
        if (lane == 0) atomicExch(err, 14);
        break;
      }
      tc_fence_after();
      const uint32_t base = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * XBUF + h);
      uint32_t r[XS][16];
#pragma unroll
      for (int L = 0; L < XS; ++L) tmem_ld16_async(base + (uint32_t)(L * XBN), r[L]);
      tmem_wait_ld();
#pragma unroll
      for (int L = 0; L < XS; ++L)  // no use of a loaded register may move before the wait
#pragma unroll
        for (int j = 0; j < 16; ++j) asm volatile("" : "+r"(r[L][j]));
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[buf]);  // the buffer may take the next K-block
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        long long p[XS];
#pragma unroll
        for (int L = 0; L < XS; ++L) p[L] = (long long)__float2int_rn(__uint_as_float(r[L][j]));
        H[j] += p[0] * 65536LL + p[1] * 256LL + p[2];
        G[j] += p[3] * 65536LL + p[4] * 256LL + p[5];
      }
    }
    if (ok && row < M && DI) {
      longlong2* dst = DI + (size_t)row * ldd;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int col = n0 + h + j;
        if (col >= N) continue;
        if (gridDim.z == 1) {
          dst[col] = make_longlong2(H[j], G[j]);
        } else {
          atomicAdd(reinterpret_cast<unsigned long long*>(&dst[col].x), (unsigned long long)H[j]);
          atomicAdd(reinterpret_cast<unsigned long long*>(&dst[col].y), (unsigned long long)G[j]);
        }
      }
    } else if (ok && row < M) {
      const int er = ea[row];
      double* dst = D + (size_t)row * ldd;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const int col = n0 + h + j;
        if (col < N) {
          const int x = eb[col], e = er + (x == NOT_FINITE ? 0 : x);
          dst[col] = x == NOT_FINITE ? quiet_nan() : ldexp((double)H[j], e - 32) + ldexp((double)G[j], e - 56);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(XTMEM_COLS) : "memory");
}

// ---- digit planes ----
// The 48 bits v 2^48, v = x 2^-e, |v| < 1/2, are rounded once and cut into bytes with integer
// operations, 128 added to each so that the bytes are the digits plus 128 (GB300's FP64 pipe runs at
// 1/64 of the integer rate; in FP64 the digits of 16 columns of 7680 took 48 us, and now 7).
constexpr unsigned long long DIGIT_BIAS = 0x808080808080ull;

// m 2^-s rounded to an integer
__device__ __forceinline__ unsigned long long shift_round(unsigned long long m, int s) {
  if (s <= 0) return m << -s;
  return s > 62 ? 0ull : (m + (1ull << (s - 1))) >> s;
}
// x 2^(b - e) rounded, for |x| < 2^(e - 1) and b <= 60
__device__ __forceinline__ long long fixed_f64(double x, int e, int b) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((u >> 52) & 2047);
  const unsigned long long m = (u & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0ull);
  const long long v = (long long)shift_round(m, 1075 - b + e - max(ex, 1));
  return (u >> 63) ? -v : v;
}
__device__ __forceinline__ long long fixed_f32(float x, int e, int b) {
  const uint32_t u = __float_as_uint(x);
  const int ex = (int)((u >> 23) & 255);
  const unsigned long long m = (u & 0x7fffffu) | (ex ? 1u << 23 : 0u);
  const long long v = (long long)shift_round(m, 150 - b + e - max(ex, 1));
  return (u >> 31) ? -v : v;
}

// rows of an operand: mag() is the size of an entry by its bits, fixed() its 48 bits under 2^e
struct SrcC64Stacked {  // rows 0..n-1: Re of the complex64 matrix rows, rows n..2n-1: Im
  const float2* M;
  long long ld;
  int n;
  __device__ float at(int r, int k) const { return r < n ? M[(size_t)r * ld + k].x : M[(size_t)(r - n) * ld + k].y; }
  __device__ uint32_t mag(int r, int k) const { return __float_as_uint(at(r, k)) & 0x7fffffffu; }
  __device__ long long fixed(int r, int k, int e) const { return fixed_f32(at(r, k), e, 48); }
};
struct SrcF32Pair {  // hi + lo FP32 planes of an FP64-accurate real matrix (hi the sum rounded to FP32)
  const float* hi;
  const float* lo;
  long long ld;
  __device__ uint32_t mag(int r, int k) const { return __float_as_uint(hi[(size_t)r * ld + k]) & 0x7fffffffu; }
  __device__ long long fixed(int r, int k, int e) const {
    const size_t o = (size_t)r * ld + k;
    return (fixed_f32(hi[o], e, 60) + fixed_f32(lo[o], e, 60) + 2048) >> 12;
  }
};

constexpr int DT = 256;

// the digits of two consecutive k into XS planes (32-bit words p of a row)
__device__ __forceinline__ void store_digits(long long u, long long v, uint32_t* __restrict__ o, size_t plane) {
  const unsigned long long wu = (unsigned long long)u + DIGIT_BIAS, wv = (unsigned long long)v + DIGIT_BIAS;
#pragma unroll
  for (int s = 0; s < XS; ++s) {
    const int sh = 40 - 8 * s;
    const uint32_t mask = s ? 255u : 511u;  // the leading digit runs to 128
    const __nv_bfloat162 d = __floats2bfloat162_rn((float)((int)((uint32_t)(wu >> sh) & mask) - 128),
                                                   (float)((int)((uint32_t)(wv >> sh) & mask) - 128));
    o[s * plane] = *reinterpret_cast<const uint32_t*>(&d);
  }
}

// One CTA per row of a matrix: the row's power-of-two scale 2^e (|v| 2^-e < 1/2) and its XS base-256
// digits, written to XS planes (zeros in the padding).
template <class Src>
__global__ void __launch_bounds__(DT) digits_kernel(Src src, int K, long long ldp, uint32_t* __restrict__ planes,
                                                    long long plane_stride, int* __restrict__ e_out) {
  RF_COUNT_LAUNCH();
  const int r = blockIdx.x;
  uint32_t m = 0;
  for (int k = threadIdx.x; k < K; k += DT) m = max(m, src.mag(r, k));
  m = __reduce_max_sync(0xffffffffu, m);
  __shared__ uint32_t red[DT / 32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < DT / 32; ++w) m = max(m, red[w]);
  const int e = m ? ilogbf(__uint_as_float(m)) + 2 : 0;  // |v| < 2^(e - 1)
  if (threadIdx.x == 0) e_out[r] = e;
  const size_t plane = (size_t)plane_stride / 2;
  for (int p = threadIdx.x; p < (int)(ldp / 2); p += DT) {
    const int k = 2 * p;
    store_digits(k < K ? src.fixed(r, k, e) : 0, k + 1 < K ? src.fixed(r, k + 1, e) : 0,
                 planes + (size_t)r * (ldp / 2) + p, plane);
  }
}

// Re and Im of one column of X per cluster of CTAs: each takes a slice of K, the column maxima
// meet through distributed shared memory, then every slice writes its digits.  Rows 0..nr-1 of the
// planes are Re of the columns, rows nr..2nr-1 Im.  Up to XCL CTAs of at least XCL_PAIRS
// pairs of entries: a cluster of 8 costs a body of 120 functions 7 us a product more (64 columns, 57 and 64 us).
constexpr int XCL = 8;
constexpr int XCL_PAIRS = 64;
__global__ void __launch_bounds__(DT)
x_digits_kernel(const double2* __restrict__ X, int n, int nr, long long ldp, uint32_t* __restrict__ planes,
                int* __restrict__ e_out) {
  RF_COUNT_LAUNCH();
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ unsigned long long mx[2];
  const int r = blockIdx.y, rank = (int)cl.block_rank(), team = (int)cl.num_blocks();
  const double2* x = X + (size_t)r * n;
  const int pairs = (int)(ldp / 2), p0 = (int)((long long)pairs * rank / team), p1 = (int)((long long)pairs * (rank + 1) / team);
  if (threadIdx.x < 2) mx[threadIdx.x] = 0;
  __syncthreads();
  unsigned long long a = 0, b = 0;
  for (int k = 2 * p0 + threadIdx.x; k < min(2 * p1, n); k += DT) {
    const double2 v = x[k];
    a = max(a, (unsigned long long)__double_as_longlong(v.x) & 0x7fffffffffffffffull);
    b = max(b, (unsigned long long)__double_as_longlong(v.y) & 0x7fffffffffffffffull);
  }
  for (int o = 16; o > 0; o >>= 1) {
    a = max(a, __shfl_xor_sync(0xffffffffu, a, o));
    b = max(b, __shfl_xor_sync(0xffffffffu, b, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&mx[0], a);
    atomicMax(&mx[1], b);
  }
  cl.sync();
  int e[2];
#pragma unroll
  for (int z = 0; z < 2; ++z) {
    unsigned long long m = 0;
    for (int c = 0; c < team; ++c) m = max(m, *cl.map_shared_rank(&mx[z], c));
    e[z] = m == 0 ? 0 : (m >> 52) == 2047 ? NOT_FINITE : ilogb(__longlong_as_double((long long)m)) + 2;
    if (rank == 0 && threadIdx.x == 0) e_out[z * nr + r] = e[z];
  }
  cl.sync();  // the other CTAs have read this one's maxima
  const size_t plane = (size_t)nr * ldp;  // 32-bit words of one digit plane (2 nr rows of ldp / 2)
  for (int p = p0 + threadIdx.x; p < p1; p += DT) {
    const double2 zero = make_double2(0.0, 0.0);
    const double2 u = 2 * p < n ? x[2 * p] : zero, v = 2 * p + 1 < n ? x[2 * p + 1] : zero;
#pragma unroll
    for (int z = 0; z < 2; ++z) {
      const bool fin = e[z] != NOT_FINITE;
      store_digits(fin ? fixed_f64(z ? u.y : u.x, e[z], 48) : 0, fin ? fixed_f64(z ? v.y : v.x, e[z], 48) : 0,
                   planes + ((size_t)z * nr + r) * (ldp / 2) + p, plane);
    }
  }
}

// Y[:, r] = scale * op(T) X[:, r] (+ Y) from the integer sums of [Tr; Ti] [Xr Xi] or (real) P [Xr Xi],
// at most XI_COLS columns: a CTA reads R rows of D along their columns and writes Y along its rows.
// The FP64 pipe takes 8 us for 32 rows of 32 columns, so small matrices take 8 rows a CTA (COMBINE_SMALL).
constexpr int XI_COLS = 32;
constexpr int COMBINE_SMALL = 32 * 152;
template <int R>
__global__ void __launch_bounds__(DT)
combine_int_kernel(const longlong2* __restrict__ D, const int* __restrict__ ea, const int* __restrict__ eb, int n,
                   int nr, int conj, int real, double2 scale, int accumulate, double2* __restrict__ Y) {
  RF_COUNT_LAUNCH();
  __shared__ double2 t[XI_COLS][R + 1];
  const int i0 = blockIdx.x * R;
  auto value = [&](int row, int col) {
    const longlong2 d = D[(size_t)row * (2 * nr) + col];
    const int x = eb[col];
    if (x == NOT_FINITE) return quiet_nan();
    const int e = ea[row] + x;
    return ldexp((double)d.x, e - 32) + ldexp((double)d.y, e - 56);
  };
  const double sg = conj ? -1.0 : 1.0;
  for (int q = threadIdx.x; q < R * nr; q += DT) {
    const int i = i0 + q / nr, r = q % nr;
    if (i >= n) break;
    double2 v = make_double2(value(i, r), value(i, nr + r));
    if (!real) {
      v.x -= sg * value(n + i, nr + r);
      v.y += sg * value(n + i, r);
    }
    t[r][i - i0] = make_double2(scale.x * v.x - scale.y * v.y, scale.x * v.y + scale.y * v.x);
  }
  __syncthreads();
  for (int q = threadIdx.x; q < R * nr; q += DT) {
    const int r = q / R, i = i0 + q % R;
    if (i >= n) continue;
    double2 o = t[r][q % R];
    double2* y = Y + (size_t)r * n + i;
    if (accumulate) {
      o.x += y->x;
      o.y += y->y;
    }
    *y = o;
  }
}

// Y[:, r] = scale * op(T) X[:, r] (+ Y) from D = [Tr; Ti] [Xr Xi] (FP64, 2n x 2nr) or, with real,
// D = P [Xr Xi] (n x 2nr); the same tiled combination as the split-BF16 path.
constexpr int CT = 32;
__global__ void combine_f64_kernel(const double* __restrict__ D, long long ldd, int n, int nr, int conj, int real,
                                   double2 scale, int accumulate, double2* __restrict__ Y) {
  RF_COUNT_LAUNCH();
  __shared__ double2 t[CT][CT + 1];
  const int i0 = blockIdx.x * CT, r0 = blockIdx.y * CT;
  const double sg = conj ? -1.0 : 1.0;
  for (int ii = threadIdx.y; ii < CT; ii += blockDim.y) {
    const int i = i0 + ii, r = r0 + threadIdx.x;
    double2 v = make_double2(0.0, 0.0);
    if (i < n && r < nr) {
      const double* top = D + (size_t)i * ldd;
      if (real) {
        v.x = top[r];
        v.y = top[nr + r];
      } else {
        const double* bot = D + (size_t)(n + i) * ldd;
        v.x = top[r] - sg * bot[nr + r];
        v.y = top[nr + r] + sg * bot[r];
      }
    }
    t[ii][threadIdx.x] = v;
  }
  __syncthreads();
  for (int rr = threadIdx.y; rr < CT; rr += blockDim.y) {
    const int r = r0 + rr, i = i0 + threadIdx.x;
    if (i >= n || r >= nr) continue;
    const double2 v = t[threadIdx.x][rr];
    double2 o = make_double2(scale.x * v.x - scale.y * v.y, scale.x * v.y + scale.y * v.x);
    if (accumulate) {
      const double2 p = Y[(size_t)r * n + i];
      o.x += p.x;
      o.y += p.y;
    }
    Y[(size_t)r * n + i] = o;
  }
}

// K split of a launch of `tiles` tiles of nkb K-blocks: the least of (waves of the chip) x (K-blocks of
// a CTA + about two for its start and its integer sums); the smaller split where two are within 3 %
int exact_split(long long tiles, int nkb, int sms) {
  int best = 1;
  double cost = 1e300;
  for (int sp = 1; sp <= 16 && sp <= nkb; ++sp) {
    const double waves = (double)((tiles * sp + sms - 1) / sms);
    const double c = waves * ((nkb + sp - 1) / sp + (sp > 1 ? 2.5 : 1.5));
    if (c < 0.97 * cost) {
      cost = c;
      best = sp;
    }
  }
  return best;
}

// D = A B^T: FP64 values, or with DI the unscaled integer sums
cudaError_t exact_gemm(const ExactOperand& A, const ExactOperand& B, int M, int N, int K, double* D, longlong2* DI,
                       long long ldd, int* err, cudaStream_t s) {
  if (M <= 0 || N <= 0 || K <= 0 || A.rows < M || B.rows < N) return cudaErrorInvalidValue;
  ExactMaps maps;
  std::memset(&maps, 0, sizeof(maps));
  for (int p = 0; p < XS; ++p)
    if (!make_map(&maps.a[p], A.d + p * A.plane_stride, M, K, A.ldp, BM, XBK) ||
        !make_map(&maps.b[p], B.d + p * B.plane_stride, N, K, B.ldp, XBN, XBK))
      return cudaErrorInvalidValue;
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  static int sms = 0;
  std::call_once(once, [] {
    attr = cudaFuncSetAttribute(exact_gemm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, XSMEM);
    int dev = 0;
    if (attr == cudaSuccess) attr = cudaGetDevice(&dev);
    if (attr == cudaSuccess) attr = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  });
  if (attr != cudaSuccess) return attr;
  const int tn = (N + XBN - 1) / XBN, tm = (M + BM - 1) / BM, nkb = (K + XKB - 1) / XKB;
  const int split = DI ? exact_split((long long)tn * tm, nkb, std::max(sms, 1)) : 1;
  if (split > 1) {
    const cudaError_t e = cudaMemsetAsync(DI, 0, sizeof(longlong2) * (size_t)M * ldd, s);
    if (e != cudaSuccess) return e;
  }
  ProfScope prof("gemm_exact", 0.0, 2.0 * (XS * (XS + 1) / 2) * (double)M * N * K, s);
  exact_gemm_kernel<<<dim3(tn, tm, split), XTHREADS, XSMEM, s>>>(maps, M, N, K, A.e, B.e, D, DI, ldd, err);
  return cudaGetLastError();
}

// Y = scale * op(T) X (+ Y) (complex T as 2n stacked rows, or real)
cudaError_t exact_product(const ExactOperand& T, int n, const double2* X, double2* Y, int nr, bool conj, bool real,
                          double2 scale, bool accumulate, MrhsScratch& w, cudaStream_t s) {
  const int rows = real ? n : 2 * n;
  if (nr > w.cap_cols || n > w.cap_n || T.ldp > w.cap_ld || !w.xd || T.rows < rows) return cudaErrorInvalidValue;
  ExactOperand B;
  B.d = w.xd;
  B.e = w.xe;
  B.rows = 2 * nr;
  B.ldp = T.ldp;
  B.plane_stride = (long long)2 * nr * T.ldp;
  int team = 1;
  while (team < XCL && 2LL * team * XCL_PAIRS <= B.ldp / 2) team *= 2;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = (unsigned)team;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)team, (unsigned)nr);
  cfg.blockDim = dim3(DT);
  cfg.stream = s;
  cfg.attrs = &attr;
  cfg.numAttrs = team > 1 ? 1 : 0;
  cudaError_t e = cudaLaunchKernelEx(&cfg, x_digits_kernel, X, n, nr, (long long)B.ldp, reinterpret_cast<uint32_t*>(B.d), B.e);
  if (e != cudaSuccess) return e;
  const bool ints = nr <= XI_COLS;
  longlong2* DI = ints ? reinterpret_cast<longlong2*>(w.D64) : nullptr;
  if ((e = exact_gemm(T, B, rows, 2 * nr, n, w.D64, DI, 2 * nr, w.err, s)) != cudaSuccess) return e;
  if (ints) {
    auto combine = [&](auto kernel, int R) {
      kernel<<<(n + R - 1) / R, DT, 0, s>>>(DI, T.e, B.e, n, nr, conj ? 1 : 0, real ? 1 : 0, scale, accumulate ? 1 : 0, Y);
    };
    if (n < COMBINE_SMALL) combine(combine_int_kernel<8>, 8);
    else combine(combine_int_kernel<32>, 32);
  } else {
    const dim3 g((n + CT - 1) / CT, (nr + CT - 1) / CT), b(CT, 8);
    combine_f64_kernel<<<g, b, 0, s>>>(w.D64, 2 * nr, n, nr, conj ? 1 : 0, real ? 1 : 0, scale, accumulate ? 1 : 0, Y);
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t exact_digits_c64(const float2* M, int n, long long ld, const ExactOperand& out, cudaStream_t s) {
  if (out.rows < 2 * n || out.ldp < ld) return cudaErrorInvalidValue;
  SrcC64Stacked src{M, ld, n};
  digits_kernel<<<2 * n, DT, 0, s>>>(src, n, out.ldp, reinterpret_cast<uint32_t*>(out.d), out.plane_stride, out.e);
  return cudaGetLastError();
}

cudaError_t exact_digits_f32pair(const float* hi, const float* lo, int n, long long ld, const ExactOperand& out,
                                 cudaStream_t s) {
  if (out.rows < n || out.ldp < ld) return cudaErrorInvalidValue;
  SrcF32Pair src{hi, lo, ld};
  digits_kernel<<<n, DT, 0, s>>>(src, n, out.ldp, reinterpret_cast<uint32_t*>(out.d), out.plane_stride, out.e);
  return cudaGetLastError();
}

cudaError_t exact_cplx_gemm(const ExactOperand& T, int n, const double2* X, double2* Y, int nr, bool conj,
                            double2 scale, bool accumulate, MrhsScratch& w, cudaStream_t s) {
  return exact_product(T, n, X, Y, nr, conj, false, scale, accumulate, w, s);
}

cudaError_t exact_real_gemm(const ExactOperand& P, int n, const double2* X, double2* Y, int nr, double scale,
                            bool accumulate, MrhsScratch& w, cudaStream_t s) {
  return exact_product(P, n, X, Y, nr, false, true, make_double2(scale, 0.0), accumulate, w, s);
}

size_t exact_result_doubles(int cols) { return (size_t)std::max(4 * cols, 8 * std::min(cols, XI_COLS)); }

RF_LAUNCH_READER(launches_exact)

}  // namespace rfcmp
