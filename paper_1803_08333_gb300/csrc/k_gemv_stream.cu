// Streaming GEMV: y = op(M) x for one or two columns with the matrix moved by the bulk-copy
// engine.
//
// The operator products of a single-right-hand-side solve are HBM bound: each application
// streams T_A, V and the factors once.  A register-pipelined GEMV keeps only as many bytes in
// flight as its unrolled loads allow; here one producer thread per CTA issues cp.async.bulk
// copies of whole row segments together with the matching part of x into a shared-memory ring, so that
// 128 to 192 KB of matrix per SM are in flight whatever the consumers do; consumers release a stage through an
// mbarrier.  Three kernels:
//   * gemv_sym_kernel (FP32 mode, symmetric M: T_A, V and the factors): reads only the tiles on
//     and above the diagonal and forms both the row and the mirrored column product.  A stage is 8 rows x 512
//     complex64 or 1024 FP32 values (32 KB) and x of the segment; one CTA with four stages, or two CTAs with two or
//     three where the registers allow twice the warps;
//   * gemv_sym_ff_kernel (float-float, symmetric M): the accurate products, from 32 KB tiles of 8 rows of complex
//     values or 4 rows of hi and lo ones, three stages, two CTAs (FfStage);
//   * gemv_stream_ff_kernel (float-float, one column of a complex64 M): one consumer warp per row of a stage of 8
//     rows x 704 values (44 KB) and x hi and lo, two stages, two CTAs (FF_ROW, FF_NST).
// Work units are dealt to persistent CTAs in contiguous ranges of equal size; partial sums meet
// in FP64 atomics.  Every wait is bounded and records an error code on timeout.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "rfcmp_internal.h"
#include "tc_common.cuh"

namespace rfcmp {

namespace {

using tc::mbar_arrive;
using tc::mbar_expect_tx;
using tc::mbar_init;
using tc::mbar_wait;
using tc::smem_u32;

constexpr int SROWS = 8;                 // rows per stage (one consumer warp each)
constexpr int SBYTES_ROW = 4096;         // bytes per row segment
constexpr int SSTAGES = 4;
constexpr int SMAT = SROWS * SBYTES_ROW;    // 32 KB of matrix per stage
constexpr int STHREADS = (SROWS + 1) * 32;  // consumers + producer warp

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// Pairs of FP32 values in one 64-bit register: the packed operations round each half as the scalar ones do and take
// half the issue slots (measured: 128 scalar or 64 packed operations a clock and SM).
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pk(float x, float y) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ f32x2 pk(float2 v) { return pk(v.x, v.y); }
__device__ __forceinline__ float2 unpk(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 neg2(f32x2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { return fma2(b, 0xbf800000bf800000ull, a); }  // a - 1 b
// i z (CONJ: -i z) of z = (re, im)
template <bool CONJ>
__device__ __forceinline__ f32x2 times_i(f32x2 z) {
  const float2 v = unpk(z);
  return CONJ ? pk(v.y, -v.x) : pk(-v.y, v.x);
}
// (s, e): s = a + b rounded, e the rest
__device__ __forceinline__ f32x2 two_sum2(f32x2 a, f32x2 b, f32x2& e) {
  const f32x2 s = add2(a, b), bb = sub2(s, a);
  e = add2(sub2(a, sub2(s, bb)), sub2(b, bb));
  return s;
}

// stage and phase of a ring of N stages, advanced one unit at a time (64-bit divisions of the unit number
// by the ring's size and by the units of a row cost a fifth of a unit's work)
template <int N>
struct Ring {
  int s = 0;
  uint32_t parity = 0;
  __device__ __forceinline__ void next() {
    if (++s == N) {
      s = 0;
      parity ^= 1u;
    }
  }
};

// One product of a launch, and which of two a CTA works on: CTAs 0 .. split - 1 the first.
struct GemvJob {
  const void* M;
  const float2 *xh, *xl;
  double2* out;
  double scale;
  long long units;
  int ld, n;
};

// ---------------------------------------------------------------- symmetric matrices
// For a symmetric M (T_A, V and the factors all are) only the tiles that reach the diagonal or
// lie above it are read: a tile of 8 rows I x one segment J contributes y_I += M_IJ x_J (row part,
// entries j >= i) and y_J += M_IJ^T x_I (column part, entries j > i), so half the matrix bytes
// leave HBM.  Units run column-major over the upper triangle: segment c holds the row blocks
// 0 .. min(RB, P (c + 1)) - 1 (P = segment width / 8 rows), so the column part stays in registers
// across the row blocks of a segment and reaches y once per segment.
//
// Both parts come from one read of the tile: consumer thread t owns float4 column slot t of the
// segment (256 slots = the 8 consumer warps x 32 lanes) in all 8 rows.  For each row it adds
// M_ij x_j into that row's partial (x_j of its slot held in registers) and M_ij x_i into its
// column sums (x_i a shared-memory broadcast).  The 8 x NR complex row partials of a warp are
// reduce-scattered across its lanes (each exchange halves the values a lane holds), the 8 warps'
// results meet in shared memory, and one warp per unit (rotating) adds them and issues the FP64
// atomics of the row part.
struct SymGeom {
  long long RB, P, S, cstar, base;  // row blocks, row blocks per segment step, segments, off() knee
  __host__ __device__ long long nrb(long long c) const { return c < cstar ? P * (c + 1) : RB; }
  // units before segment c
  __host__ __device__ long long off(long long c) const {
    return c <= cstar ? P * c * (c + 1) / 2 : base + (c - cstar) * RB;
  }
};

__host__ __device__ inline SymGeom sym_geom(int n, int ld, int seg, int rows = SROWS) {
  SymGeom g;
  g.RB = (n + rows - 1) / rows;
  g.P = seg / rows;
  g.S = (ld + seg - 1) / seg;
  g.cstar = g.RB / g.P;  // segments c < cstar hold P (c + 1) <= RB row blocks
  g.base = g.P * g.cstar * (g.cstar + 1) / 2;
  return g;
}

// Reduce-scatter of V = 16 or 32 per-lane values over the warp: on return v[0] of lane l is the
// warp sum of value l * V / 32 (for V = 16 lanes l and l ^ 1 hold the same sum).
template <int V>
__device__ __forceinline__ void warp_reduce_scatter(float (&v)[V], int lane) {
#pragma unroll
  for (int step = 0; step < 5; ++step) {
    const int off = 16 >> step;
    const int h = V >> (step + 1);  // values kept after this exchange (0: plain reduction)
    if (h == 0) {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
    } else {
      const bool upper = (lane & off) != 0;
#pragma unroll
      for (int k = 0; k < h; ++k) {
        const float send = upper ? v[k] : v[k + h];
        const float keep = upper ? v[k + h] : v[k];
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, off);
      }
    }
  }
}

// Stage layout of the symmetric kernel: the 8 row segments, the x segments of its NR columns,
// x of the 8 rows, and the consumer warps' row partials, rounded to 128 bytes.  With two CTAs
// per SM a CTA takes three stages where both rings fit the SM's 228 KB of shared memory
// (1 KB per CTA reserved by the system): the one-column complex product (37.5 KB stages);
// the others take two.
template <int NR, bool REAL, int NCTA>
struct SymStage {
  static constexpr int SEG = SBYTES_ROW / (REAL ? 4 : 8);
  static constexpr int XB = NR * SEG * 8;  // x segments of the stage (complex FP32)
  static constexpr int BYTES = ((SMAT + XB + NR * 64 + 8 * (SROWS * NR * 2) * 4) + 127) / 128 * 128;
  static constexpr int NST = NCTA == 1 ? SSTAGES : ((2 * (3 * BYTES + 256 + 1024) <= 233472) ? 3 : 2);
  static constexpr int SMEM = NST * BYTES + 256;  // + alignment slack and the mbarriers
  static_assert(SMEM <= 232448, "dynamic shared memory of one CTA");
  static_assert(NCTA * (SMEM + 1024) <= 233472, "the SM holds NCTA such CTAs");
  static_assert(BYTES % 128 == 0 && (SMAT + XB) % 16 == 0, "bulk-copy destinations stay 16-byte aligned");
};

// The 8 rows of one tile for column slot qc (entries j .. j + EPQ - 1): row partials v gain
// M_ij x_j (j >= i), column partials t gain M_ij x_i (j > i).  DIAG: the tile reaches the
// diagonal and the entries outside those ranges are dropped.
template <int NR, bool REAL, bool CONJ, bool DIAG, int XB, int EPQ = (REAL ? 4 : 2)>
__device__ __forceinline__ void sym_tile(const uint8_t* st, int qc, int row0, int n, int j, const float2 (&xj)[NR][EPQ],
                                         float (&v)[SROWS * NR * 2], float (&t)[NR][EPQ][2]) {
  const float2* sxi = reinterpret_cast<const float2*>(st + SMAT + XB);
#pragma unroll
  for (int rr = 0; rr < SROWS; ++rr) {
    const int row = row0 + rr;
    const float4 m = row < n ? reinterpret_cast<const float4*>(st + rr * SBYTES_ROW)[qc] : make_float4(0.f, 0.f, 0.f, 0.f);
    float er[EPQ], ei[EPQ];  // entries as (re, im)
    if constexpr (REAL) {
      er[0] = m.x, er[1] = m.y, er[2] = m.z, er[3] = m.w;
#pragma unroll
      for (int e = 0; e < EPQ; ++e) ei[e] = 0.f;
    } else {
      er[0] = m.x, ei[0] = CONJ ? -m.y : m.y;
      er[1] = m.z, ei[1] = CONJ ? -m.w : m.w;
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const float2 xi = sxi[r * SROWS + rr];
      float pre = v[(rr * NR + r) * 2], pim = v[(rr * NR + r) * 2 + 1];
#pragma unroll
      for (int e = 0; e < EPQ; ++e) {
        float ar = er[e], ai = ei[e], br = er[e], bi = ei[e];
        if constexpr (DIAG) {
          if (j + e < row) ar = ai = 0.f;
          if (j + e <= row) br = bi = 0.f;
        }
        if constexpr (REAL) {
          pre = fmaf(ar, xj[r][e].x, pre);
          pim = fmaf(ar, xj[r][e].y, pim);
          t[r][e][0] = fmaf(br, xi.x, t[r][e][0]);
          t[r][e][1] = fmaf(br, xi.y, t[r][e][1]);
        } else {
          pre = fmaf(ar, xj[r][e].x, fmaf(-ai, xj[r][e].y, pre));
          pim = fmaf(ar, xj[r][e].y, fmaf(ai, xj[r][e].x, pim));
          t[r][e][0] = fmaf(br, xi.x, fmaf(-bi, xi.y, t[r][e][0]));
          t[r][e][1] = fmaf(br, xi.y, fmaf(bi, xi.x, t[r][e][1]));
        }
      }
      v[(rr * NR + r) * 2] = pre;
      v[(rr * NR + r) * 2 + 1] = pim;
    }
  }
}

template <int NR, bool REAL, bool CONJ, int NCTA>
__global__ void __launch_bounds__(STHREADS, NCTA)
gemv_sym_kernel(const __grid_constant__ GemvJob J0, const __grid_constant__ GemvJob J1, int split,
                int* __restrict__ err) {
  RF_COUNT_LAUNCH();
  const bool other = (int)blockIdx.x >= split;
  const GemvJob& J = other ? J1 : J0;
  const int bid = other ? blockIdx.x - split : blockIdx.x, ctas = other ? gridDim.x - split : split;
  const void* __restrict__ Mv = J.M;
  const float2* __restrict__ xh = J.xh;
  double2* __restrict__ out = J.out;
  const double scale = J.scale;
  const long long units = J.units;
  const int ld = J.ld, n = J.n;
  constexpr int NST = SymStage<NR, REAL, NCTA>::NST;
  constexpr int STG = SymStage<NR, REAL, NCTA>::BYTES;
  constexpr int XB = SymStage<NR, REAL, NCTA>::XB;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + NST * STG);
  uint64_t* empty = full + NST;
  uint64_t* rfull = empty + NST;  // the 8 warps' row partials of a stage are in shared memory
  constexpr int ESZ = REAL ? 4 : 8;
  constexpr int SEG = SBYTES_ROW / ESZ;
  constexpr int EPQ = 16 / ESZ;       // matrix entries per float4
  constexpr int V = SROWS * NR * 2;   // row partials per lane: 8 rows x NR columns x (re, im)
  static_assert(SBYTES_ROW / 16 == SROWS * 32, "one float4 column slot per consumer thread");
  static_assert(V == 16 || V == 32, "reduce-scatter of 16 or 32 values");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const SymGeom G = sym_geom(n, ld, SEG);
  const long long u0 = units * bid / ctas, u1 = units * (bid + 1) / ctas;
  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], SROWS);
      mbar_init(&rfull[s], SROWS);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (u0 >= u1) return;
  // segment and row block of unit u0 (binary search on off())
  int c0 = 0;
  {
    long long lo = 0, hi = G.S - 1;
    while (lo < hi) {
      const long long mid = (lo + hi + 1) / 2;
      if (G.off(mid) <= u0) lo = mid;
      else hi = mid - 1;
    }
    c0 = (int)lo;
  }
  const int rb0 = (int)(u0 - G.off(c0)), cnt = (int)(u1 - u0);
  const char* M = reinterpret_cast<const char*>(Mv);

  if (warp == SROWS) {
    if (lane == 0) {
      int c = c0, rb = rb0, nrb = (int)G.nrb(c);
      Ring<NST> q;
      for (int i = 0; i < cnt; ++i, q.next()) {
        const int s = q.s;
        if (i >= NST && !mbar_wait(&empty[s], q.parity ^ 1u)) {
          atomicExch(err, 24);
          break;
        }
        const int cb = c * SEG, row0 = rb * SROWS, rows = min(SROWS, n - row0);
        const int cols = min(SEG, ld - cb);
        const uint32_t bytes = (uint32_t)cols * ESZ, xbytes = (uint32_t)cols * 8;
        mbar_expect_tx(&full[s], bytes * rows + (xbytes + 64) * NR);
        uint8_t* st = smem + s * STG;
        for (int r = 0; r < rows; ++r)
          bulk_load(st + r * SBYTES_ROW, M + ((size_t)(row0 + r) * ld + cb) * ESZ, bytes, &full[s]);
        for (int r = 0; r < NR; ++r) {
          bulk_load(st + SMAT + r * (XB / NR), xh + (size_t)r * ld + cb, xbytes, &full[s]);
          bulk_load(st + SMAT + XB + r * 64, xh + (size_t)r * ld + row0, 64, &full[s]);  // x of the 8 rows
        }
        if (++rb == nrb) {
          nrb = (int)G.nrb(++c);
          rb = 0;
        }
      }
      for (int i = max(0, cnt - NST); i < cnt; ++i)
        if (!mbar_wait(&full[i % NST], (uint32_t)((i / NST) & 1))) atomicExch(err, 25);
    }
    return;
  }

  // column sums of slot qc (EPQ entries, NR columns) in compensated FP32
  float ca[NR][EPQ][2], cc[NR][EPQ][2];
#pragma unroll
  for (int r = 0; r < NR; ++r)
#pragma unroll
    for (int e = 0; e < EPQ; ++e) ca[r][e][0] = ca[r][e][1] = cc[r][e][0] = cc[r][e][1] = 0.f;
  const int qc = 32 * warp + lane;
  auto flush_cols = [&](int c) {
    const int j0 = c * SEG + EPQ * qc;
#pragma unroll
    for (int r = 0; r < NR; ++r)
#pragma unroll
      for (int e = 0; e < EPQ; ++e) {
        if (j0 + e < n) {
          double* o = reinterpret_cast<double*>(out + (size_t)r * n + j0 + e);
          atomicAdd(o, scale * ((double)ca[r][e][0] + (double)cc[r][e][0]));
          atomicAdd(o + 1, scale * ((double)ca[r][e][1] + (double)cc[r][e][1]));
        }
        ca[r][e][0] = ca[r][e][1] = cc[r][e][0] = cc[r][e][1] = 0.f;
      }
  };
  int c = c0, rb = rb0, nrb = (int)G.nrb(c);
  Ring<NST> q;
  bool ok = true;
  for (int i = 0; i < cnt; ++i, q.next()) {
    const int s = q.s;
    const uint32_t parity = q.parity;
    ok = __all_sync(0xffffffffu, mbar_wait(&full[s], parity));
    if (!ok) {
      if (lane == 0) atomicExch(err, 26);
      break;
    }
    const int cb = c * SEG, row0 = rb * SROWS;
    const bool diag = row0 + SROWS > cb;  // the segment reaches the diagonal of this row block
    uint8_t* st = smem + s * STG;
    const int nq = min(SEG, ld - cb) * ESZ / 16;
    float v[V];  // row partials, index (rr * NR + r) * 2 + (re, im)
#pragma unroll
    for (int k = 0; k < V; ++k) v[k] = 0.f;
    if (qc < nq) {
      // x_j of the slot, NR columns
      float2 xj[NR][EPQ];
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const float4* xr = reinterpret_cast<const float4*>(st + SMAT + r * (XB / NR));
#pragma unroll
        for (int h = 0; h < EPQ / 2; ++h) {
          const float4 x4 = xr[(EPQ / 2) * qc + h];
          xj[r][2 * h] = make_float2(x4.x, x4.y);
          xj[r][2 * h + 1] = make_float2(x4.z, x4.w);
        }
      }
      const int j = cb + EPQ * qc;
      float t[NR][EPQ][2];
#pragma unroll
      for (int r = 0; r < NR; ++r)
#pragma unroll
        for (int e = 0; e < EPQ; ++e) t[r][e][0] = t[r][e][1] = 0.f;
      if (diag) sym_tile<NR, REAL, CONJ, true, XB>(st, qc, row0, n, j, xj, v, t);
      else sym_tile<NR, REAL, CONJ, false, XB>(st, qc, row0, n, j, xj, v, t);
#pragma unroll
      for (int r = 0; r < NR; ++r)
#pragma unroll
        for (int e = 0; e < EPQ; ++e)
#pragma unroll
          for (int z = 0; z < 2; ++z) {  // two-sum into the running column sums
            const float a = ca[r][e][z], b = t[r][e][z], tt = a + b, bb = tt - a;
            cc[r][e][z] += (a - (tt - bb)) + (b - bb);
            ca[r][e][z] = tt;
          }
    }
    // row part: reduce-scatter over the warp, then the 8 warps meet in shared memory
    warp_reduce_scatter<V>(v, lane);
    float* red = reinterpret_cast<float*>(st + SMAT + XB + NR * 64);  // [SROWS warps][V]
    if (V == 32 || (lane & 1) == 0) red[warp * V + lane * V / 32] = v[0];
    __syncwarp();
    if (lane == 0) mbar_arrive(&rfull[s]);
    if (warp == i % SROWS) {
      const bool got = __all_sync(0xffffffffu, mbar_wait(&rfull[s], parity));
      if (!got) {
        if (lane == 0) atomicExch(err, 27);
        ok = false;
        break;
      }
      if (lane < V) {
        float sum = 0.f;
#pragma unroll
        for (int w2 = 0; w2 < SROWS; ++w2) sum += red[w2 * V + lane];
        const int rr = lane / (2 * NR), r = (lane / 2) % NR, z = lane & 1;
        const int row = row0 + rr;
        if (row < n) atomicAdd(reinterpret_cast<double*>(out + (size_t)r * n + row) + z, scale * (double)sum);
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s]);
    if (++rb == nrb) {
      flush_cols(c);
      nrb = (int)G.nrb(++c);
      rb = 0;
    }
  }
  if (ok && rb > 0) flush_cols(c);
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}

// ---------------------------------------------------------------- float-float, one column
// The accurate products (right-hand side, refinement residuals) of a complex64 matrix in the
// streaming layout: x is split into FP32 hi + lo, every product m * x_hi is exact as (p, e) by an
// FMA residual, p enters a float-float (hi, lo) accumulator by an error-free two-sum and
// e + m * x_lo its low word (about 1e-14 of sum |terms|).
// Bound: the FP32 pipe, 22 packed operations an entry (its real and its imaginary part times both parts of x).
// Two CTAs per SM, two stages of 55 KB each (8 rows x 704 entries and x hi and lo of the segment), the longest
// segments that fit: N = 30720 in 1.46 ms; segments of 512 entries 1.54, three CTAs and 448 or 256 entries 1.61 and
// 1.78; with scalar operations (twice the issue slots) and 512 entries 1.64.
constexpr int FF_NCTA = 2;
constexpr int FF_NST = 2;
constexpr int FF_ROW = 5632;                    // bytes of a row segment
constexpr int FF_MAT = SROWS * FF_ROW;
constexpr int FF_STAGE = FF_MAT + 2 * FF_ROW;   // the matrix, x hi, x lo
static_assert(FF_NCTA * (FF_NST * FF_STAGE + 256 + 1024) <= 233472, "the SM holds FF_NCTA float-float CTAs");

__device__ __forceinline__ void ff_acc(float& hi, float& lo, float a, float bh, float bl) {
  const float p = a * bh;
  const float e = fmaf(a, bh, -p);
  const float c = fmaf(a, bl, e);
  const float s = hi + p;
  const float bb = s - hi;
  lo += ((hi - (s - bb)) + (p - bb)) + c;
  hi = s;
}
// both halves: hi + lo += a b with b = bh + bl
__device__ __forceinline__ void ff_acc(f32x2& hi, f32x2& lo, f32x2 a, f32x2 bh, f32x2 bl) {
  const f32x2 p = mul2(a, bh), c = fma2(a, bl, fma2(a, bh, neg2(p)));
  f32x2 rest;
  hi = two_sum2(hi, p, rest);
  lo = add2(lo, add2(rest, c));
}
template <bool CONJ>
__global__ void __launch_bounds__(STHREADS, FF_NCTA)
gemv_stream_ff_kernel(const __grid_constant__ GemvJob J0, const __grid_constant__ GemvJob J1, int split,
                      int* __restrict__ err) {
  RF_COUNT_LAUNCH();
  const bool other = (int)blockIdx.x >= split;
  const GemvJob& J = other ? J1 : J0;
  const int bid = other ? blockIdx.x - split : blockIdx.x, ctas = other ? gridDim.x - split : split;
  const float2* __restrict__ M = static_cast<const float2*>(J.M);
  const float2 *__restrict__ xh = J.xh, *__restrict__ xl = J.xl;
  double2* __restrict__ out = J.out;
  const double scale = J.scale;
  const long long units = J.units;
  const int ld = J.ld, n = J.n;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + FF_NST * FF_STAGE);
  uint64_t* empty = full + FF_NST;
  constexpr int SEG = FF_ROW / 8;  // complex entries per row segment
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int upr = (ld + SEG - 1) / SEG;
  const long long u0 = units * bid / ctas, u1 = units * (bid + 1) / ctas;
  const int cnt = (int)(u1 - u0), rb0 = (int)(u0 / upr), cc0 = (int)(u0 % upr);
  if (threadIdx.x == 0) {
    for (int s = 0; s < FF_NST; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], SROWS);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();

  if (warp == SROWS) {
    if (lane == 0) {
      int rb = rb0, cc = cc0;
      Ring<FF_NST> q;
      for (int i = 0; i < cnt; ++i, q.next()) {
        const int s = q.s;
        if (i >= FF_NST && !mbar_wait(&empty[s], q.parity ^ 1u)) {
          atomicExch(err, 31);
          break;
        }
        const int cb = cc * SEG;
        const int row0 = rb * SROWS, rows = min(SROWS, n - row0);
        const int cols = min(SEG, ld - cb);
        const uint32_t bytes = (uint32_t)cols * 8;
        mbar_expect_tx(&full[s], bytes * rows + 2 * bytes);
        uint8_t* st = smem + s * FF_STAGE;
        for (int r = 0; r < rows; ++r)
          bulk_load(st + r * FF_ROW, M + (size_t)(row0 + r) * ld + cb, bytes, &full[s]);
        bulk_load(st + FF_MAT, xh + cb, bytes, &full[s]);
        bulk_load(st + FF_MAT + FF_ROW, xl + cb, bytes, &full[s]);
        if (++cc == upr) {
          cc = 0;
          ++rb;
        }
      }
      for (int i = max(0, cnt - FF_NST); i < cnt; ++i)
        if (!mbar_wait(&full[i % FF_NST], (uint32_t)((i / FF_NST) & 1))) atomicExch(err, 33);
    }
    return;
  }

  // float-float sums of row `warp`: Re M x and Im M x, their real and imaginary parts paired
  f32x2 rh = 0ull, rl = 0ull, ih = 0ull, il = 0ull;
  auto flush = [&](int rb) {
    const int row = rb * SROWS + warp;
    f32x2 rest;
    const float2 h = unpk(two_sum2(rh, times_i<CONJ>(ih), rest));
    const float2 l = unpk(add2(add2(rl, times_i<CONJ>(il)), rest));
    const double re = warp_sum_d((double)h.x + (double)l.x), im = warp_sum_d((double)h.y + (double)l.y);
    rh = rl = ih = il = 0ull;
    if (lane == 0 && row < n) {
      double* o = reinterpret_cast<double*>(out + row);
      atomicAdd(o, scale * re);
      atomicAdd(o + 1, scale * im);
    }
  };
  int rb = rb0, cc = cc0;
  Ring<FF_NST> r;
  bool ok = true;
  for (int i = 0; i < cnt && ok; ++i, r.next()) {
    const int s = r.s, cb = cc * SEG;
    ok = __all_sync(0xffffffffu, mbar_wait(&full[s], r.parity));
    if (!ok) {
      if (lane == 0) atomicExch(err, 32);
      break;
    }
    const int row = rb * SROWS + warp;
    if (row < n) {
      const uint8_t* st = smem + s * FF_STAGE;
      const float4* sxh = reinterpret_cast<const float4*>(st + FF_MAT);
      const float4* sxl = reinterpret_cast<const float4*>(st + FF_MAT + FF_ROW);
      const float4* srow = reinterpret_cast<const float4*>(st + warp * FF_ROW);
      const int nq = min(SEG, ld - cb) / 2;  // two complex entries per float4
#pragma unroll 4
      for (int q = lane; q < nq; q += 32) {
        const float4 m = srow[q], x4 = sxh[q], l4 = sxl[q];
        const f32x2 h0 = pk(x4.x, x4.y), h1 = pk(x4.z, x4.w), l0 = pk(l4.x, l4.y), l1 = pk(l4.z, l4.w);
        ff_acc(rh, rl, pk(m.x, m.x), h0, l0);
        ff_acc(ih, il, pk(m.y, m.y), h0, l0);
        ff_acc(rh, rl, pk(m.z, m.z), h1, l1);
        ff_acc(ih, il, pk(m.w, m.w), h1, l1);
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s]);
    if (++cc == upr) {
      flush(rb++);
      cc = 0;
    }
  }
  if (ok && cc > 0) flush(rb);
}

// ---------------------------------------------------------------- float-float, symmetric matrices
// The accurate products (right-hand side, refinement residuals) in the symmetric streaming layout: x is
// split into FP32 hi + lo, every product m x_hi is exact as (p, e) by an FMA residual, p enters a
// float-float (hi, lo) accumulator by an error-free two-sum and e + m x_lo its low word.  A factor's
// entries are hi + lo themselves: lo x_hi joins the low word.
//
// Bound: the FP32 pipe, 11 operations per real product (12 of a factor), n^2 products of a column; the
// tiles above the diagonal alone leave HBM half of what a full pass reads, so that it stays out of the
// way.  One column per CTA (grid.y): a second column would only share bytes.  A stage is 32 KB: 8 rows of
// complex entries or 4 rows of hi and lo; a thread keeps x of its column slot in registers over a segment.
// Row sums start afresh every tile and meet as float-float pairs over the warp (a reduce-scatter), then
// over the warps, then in FP64; the column sums are merged every 64 products (FF_MERGE or FF_FLUSH tiles) and go to
// FP64 every FF_FLUSH tiles.  Neither chain is longer than a row-wise pass's, nor is the rounding of their
// low words larger.
// Two complex columns at N = 30720: 3.66 ms where a row-wise kernel over plain loads took 4.93; a factor of
// 20480 rows: 0.53 ms for one column (0.64), 1.02 for two (1.55); small matrices, two columns of 480 rows:
// 11 us (27).
constexpr int FF_FLUSH = 16;
constexpr int FF_MERGE = 4;

__device__ __forceinline__ void ff_first(float& hi, float& lo, float a, float bh, float bl) {
  hi = a * bh;
  lo = fmaf(a, bl, fmaf(a, bh, -hi));
}
__device__ __forceinline__ void ff_add(float& hi, float& lo, float h2, float l2) {
  const float s = hi + h2, bb = s - hi;
  lo += ((hi - (s - bb)) + (h2 - bb)) + l2;
  hi = s;
}

// warp_reduce_scatter for float-float pairs
template <int V>
__device__ __forceinline__ void warp_reduce_scatter_ff(float (&h)[V], float (&l)[V], int lane) {
#pragma unroll
  for (int step = 0; step < 5; ++step) {
    const int off = 16 >> step, c = V >> (step + 1);
    if (c == 0) {
      const float h2 = __shfl_xor_sync(0xffffffffu, h[0], off), l2 = __shfl_xor_sync(0xffffffffu, l[0], off);
      ff_add(h[0], l[0], h2, l2);
    } else {
      const bool up = (lane & off) != 0;
#pragma unroll
      for (int k = 0; k < c; ++k) {
        const float h2 = __shfl_xor_sync(0xffffffffu, up ? h[k] : h[k + c], off);
        const float l2 = __shfl_xor_sync(0xffffffffu, up ? l[k] : l[k + c], off);
        float kh = up ? h[k + c] : h[k], kl = up ? l[k + c] : l[k];
        ff_add(kh, kl, h2, l2);
        h[k] = kh;
        l[k] = kl;
      }
    }
  }
}

template <bool REAL>
struct FfStage {
  static constexpr int ROWS = REAL ? 4 : 8;
  static constexpr int SEG = SBYTES_ROW / (REAL ? 4 : 8);
  static constexpr int XI = SMAT;              // x of the rows: hi, then lo (8 ROWS bytes each)
  static constexpr int RED = SMAT + 16 * ROWS; // row sums of the warps
  static constexpr int V = 2 * ROWS;           // values of a tile's row part
  static constexpr int BYTES = (RED + SROWS * V * 8 + 127) / 128 * 128;
  static constexpr int NST = 3;
  static constexpr int SMEM = NST * BYTES + 256;
  static_assert(2 * (SMEM + 1024) <= 233472, "the SM holds two such CTAs");
};

// the rows of one tile for column slot qc (entries j .. j + EPQ - 1): row sums (h, l) gain M_ij x_j (j >= i),
// column sums (ch, cl) gain M_ij x_i (j > i).  DIAG: the tile reaches the diagonal.
template <bool REAL, bool CONJ, bool DIAG, int EPQ = (REAL ? 4 : 2)>
__device__ __forceinline__ void ff_tile(const uint8_t* st, int qc, int row0, int n, int j, const float2 (&xh)[EPQ],
                                        const float2 (&xl)[EPQ], float (&h)[FfStage<REAL>::V],
                                        float (&l)[FfStage<REAL>::V], float (&ch)[EPQ][2], float (&cl)[EPQ][2]) {
  using S = FfStage<REAL>;
  const float2* sxh = reinterpret_cast<const float2*>(st + S::XI);
  const float2* sxl = sxh + S::ROWS;
#pragma unroll
  for (int rr = 0; rr < S::ROWS; ++rr) {
    const int row = row0 + rr;
    const bool in = row < n;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 m = in ? reinterpret_cast<const float4*>(st + rr * SBYTES_ROW)[qc] : zero;
    const float2 ih = sxh[rr], il = sxl[rr];
    float &rh = h[2 * rr], &rl = l[2 * rr], &jh = h[2 * rr + 1], &jl = l[2 * rr + 1];
    if constexpr (REAL) {
      const float4 w = in ? reinterpret_cast<const float4*>(st + SMAT / 2 + rr * SBYTES_ROW)[qc] : zero;
      const float mh[4] = {m.x, m.y, m.z, m.w}, ml[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const bool a = !DIAG || j + e >= row, b = !DIAG || j + e > row;
        const float ah = a ? mh[e] : 0.f, al = a ? ml[e] : 0.f, bh = b ? mh[e] : 0.f, bl = b ? ml[e] : 0.f;
        if (e == 0) {
          ff_first(rh, rl, ah, xh[e].x, xl[e].x);
          ff_first(jh, jl, ah, xh[e].y, xl[e].y);
        } else {
          ff_acc(rh, rl, ah, xh[e].x, xl[e].x);
          ff_acc(jh, jl, ah, xh[e].y, xl[e].y);
        }
        rl = fmaf(al, xh[e].x, rl);
        jl = fmaf(al, xh[e].y, jl);
        ff_acc(ch[e][0], cl[e][0], bh, ih.x, il.x);
        ff_acc(ch[e][1], cl[e][1], bh, ih.y, il.y);
        cl[e][0] = fmaf(bl, ih.x, cl[e][0]);
        cl[e][1] = fmaf(bl, ih.y, cl[e][1]);
      }
    } else {
      const float mr[2] = {m.x, m.z}, mi[2] = {CONJ ? -m.y : m.y, CONJ ? -m.w : m.w};
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const bool a = !DIAG || j + e >= row, b = !DIAG || j + e > row;
        const float ar = a ? mr[e] : 0.f, ai = a ? mi[e] : 0.f, br = b ? mr[e] : 0.f, bi = b ? mi[e] : 0.f;
        if (e == 0) {
          ff_first(rh, rl, ar, xh[e].x, xl[e].x);
          ff_first(jh, jl, ar, xh[e].y, xl[e].y);
        } else {
          ff_acc(rh, rl, ar, xh[e].x, xl[e].x);
          ff_acc(jh, jl, ar, xh[e].y, xl[e].y);
        }
        ff_acc(rh, rl, -ai, xh[e].y, xl[e].y);
        ff_acc(jh, jl, ai, xh[e].x, xl[e].x);
        ff_acc(ch[e][0], cl[e][0], br, ih.x, il.x);
        ff_acc(ch[e][1], cl[e][1], br, ih.y, il.y);
        ff_acc(ch[e][0], cl[e][0], -bi, ih.y, il.y);
        ff_acc(ch[e][1], cl[e][1], bi, ih.x, il.x);
      }
    }
  }
}

template <bool REAL, bool CONJ>
__global__ void __launch_bounds__(STHREADS, 2)
gemv_sym_ff_kernel(const char* __restrict__ M, const char* __restrict__ Mlo, int ld, int n,
                   const float2* __restrict__ xh_all, const float2* __restrict__ xl_all, double2* __restrict__ out_all,
                   double scale, long long units, int* __restrict__ err) {
  RF_COUNT_LAUNCH();
  using S = FfStage<REAL>;
  constexpr int NST = S::NST, SEG = S::SEG, ROWS = S::ROWS, V = S::V, ESZ = REAL ? 4 : 8, EPQ = 16 / ESZ;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 127) & ~uintptr_t(127));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + NST * S::BYTES);
  uint64_t* empty = full + NST;
  uint64_t* rfull = empty + NST;  // the 8 warps' row sums of a stage are in shared memory
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float2 *xh = xh_all + (size_t)blockIdx.y * ld, *xl = xl_all + (size_t)blockIdx.y * ld;
  double2* out = out_all + (size_t)blockIdx.y * n;
  const SymGeom G = sym_geom(n, ld, SEG, ROWS);
  const long long u0 = units * blockIdx.x / gridDim.x, u1 = units * (blockIdx.x + 1) / gridDim.x;
  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], SROWS);
      mbar_init(&rfull[s], SROWS);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (u0 >= u1) return;
  // segment and row block of unit u0 (binary search on off())
  int c0 = 0;
  {
    long long lo = 0, hi = G.S - 1;
    while (lo < hi) {
      const long long mid = (lo + hi + 1) / 2;
      if (G.off(mid) <= u0) lo = mid;
      else hi = mid - 1;
    }
    c0 = (int)lo;
  }
  const int rb0 = (int)(u0 - G.off(c0)), cnt = (int)(u1 - u0);

  if (warp == SROWS) {
    if (lane == 0) {
      int c = c0, rb = rb0, nrb = (int)G.nrb(c);
      Ring<NST> q;
      for (int i = 0; i < cnt; ++i, q.next()) {
        const int s = q.s;
        if (i >= NST && !mbar_wait(&empty[s], q.parity ^ 1u)) {
          atomicExch(err, 31);
          break;
        }
        const int cb = c * SEG, row0 = rb * ROWS, rows = min(ROWS, n - row0);
        const uint32_t bytes = (uint32_t)min(SEG, ld - cb) * ESZ;
        mbar_expect_tx(&full[s], bytes * rows * (REAL ? 2 : 1) + 16 * ROWS);
        uint8_t* st = smem + s * S::BYTES;
        for (int r = 0; r < rows; ++r) {
          const size_t o = ((size_t)(row0 + r) * ld + cb) * ESZ;
          bulk_load(st + r * SBYTES_ROW, M + o, bytes, &full[s]);
          if (REAL) bulk_load(st + SMAT / 2 + r * SBYTES_ROW, Mlo + o, bytes, &full[s]);
        }
        bulk_load(st + S::XI, xh + row0, 8 * ROWS, &full[s]);
        bulk_load(st + S::XI + 8 * ROWS, xl + row0, 8 * ROWS, &full[s]);
        if (++rb == nrb) {
          nrb = (int)G.nrb(++c);
          rb = 0;
        }
      }
      for (int i = max(0, cnt - NST); i < cnt; ++i)
        if (!mbar_wait(&full[i % NST], (uint32_t)((i / NST) & 1))) atomicExch(err, 33);
    }
    return;
  }

  const int qc = 32 * warp + lane;
  float2 xjh[EPQ], xjl[EPQ];
  float ch[EPQ][2], cl[EPQ][2];
  float dh[REAL ? 1 : EPQ][2], dl[REAL ? 1 : EPQ][2];  // complex: the column sums of FF_MERGE tiles and more
#pragma unroll
  for (int e = 0; e < EPQ; ++e) {
    ch[e][0] = ch[e][1] = cl[e][0] = cl[e][1] = 0.f;
    if (!REAL) dh[e][0] = dh[e][1] = dl[e][0] = dl[e][1] = 0.f;
  }
  auto merge_cols = [&] {
#pragma unroll
    for (int e = 0; e < EPQ; ++e)
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        ff_add(dh[REAL ? 0 : e][z], dl[REAL ? 0 : e][z], ch[e][z], cl[e][z]);
        ch[e][z] = cl[e][z] = 0.f;
      }
  };
  auto flush_cols = [&](int c) {
    if (!REAL) merge_cols();
    const int j0 = c * SEG + EPQ * qc;
#pragma unroll
    for (int e = 0; e < EPQ; ++e) {
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        float& h = REAL ? ch[e][z] : dh[REAL ? 0 : e][z];
        float& l = REAL ? cl[e][z] : dl[REAL ? 0 : e][z];
        if (j0 + e < n) atomicAdd(reinterpret_cast<double*>(out + j0 + e) + z, scale * ((double)h + (double)l));
        h = l = 0.f;
      }
    }
  };
  auto load_x = [&](int c) {  // x of the slot's columns (zero past the padded row)
    const int j0 = c * SEG + EPQ * qc;
#pragma unroll
    for (int e = 0; e < EPQ; ++e) {
      const bool in = j0 + e < ld;
      xjh[e] = in ? xh[j0 + e] : make_float2(0.f, 0.f);
      xjl[e] = in ? xl[j0 + e] : make_float2(0.f, 0.f);
    }
  };
  int c = c0, rb = rb0, nrb = (int)G.nrb(c);
  load_x(c);
  Ring<NST> q;
  bool ok = true;
  for (int i = 0; i < cnt; ++i, q.next()) {
    const int s = q.s;
    const uint32_t parity = q.parity;
    ok = __all_sync(0xffffffffu, mbar_wait(&full[s], parity));
    if (!ok) {
      if (lane == 0) atomicExch(err, 32);
      break;
    }
    const int cb = c * SEG, row0 = rb * ROWS;
    uint8_t* st = smem + s * S::BYTES;
    float h[V], l[V];
    if (qc < min(SEG, ld - cb) * ESZ / 16) {
      const int j = cb + EPQ * qc;
      if (row0 + ROWS > cb) ff_tile<REAL, CONJ, true>(st, qc, row0, n, j, xjh, xjl, h, l, ch, cl);
      else ff_tile<REAL, CONJ, false>(st, qc, row0, n, j, xjh, xjl, h, l, ch, cl);
    } else {
#pragma unroll
      for (int k = 0; k < V; ++k) h[k] = l[k] = 0.f;
    }
    if (!REAL && i % FF_MERGE == FF_MERGE - 1) merge_cols();
    if (i % FF_FLUSH == FF_FLUSH - 1) flush_cols(c);
    warp_reduce_scatter_ff<V>(h, l, lane);
    float2* red = reinterpret_cast<float2*>(st + S::RED);  // [SROWS warps][V]
    if (lane % (32 / V) == 0) red[warp * V + lane * V / 32] = make_float2(h[0], l[0]);
    __syncwarp();
    if (lane == 0) mbar_arrive(&rfull[s]);
    if (warp == i % SROWS) {
      const bool got = __all_sync(0xffffffffu, mbar_wait(&rfull[s], parity));
      if (!got) {
        if (lane == 0) atomicExch(err, 34);
        ok = false;
        break;
      }
      if (lane < V) {
        float sh = 0.f, sl = 0.f;
#pragma unroll
        for (int w2 = 0; w2 < SROWS; ++w2) {
          const float2 v = red[w2 * V + lane];
          ff_add(sh, sl, v.x, v.y);
        }
        const int row = row0 + (lane >> 1);
        if (row < n)
          atomicAdd(reinterpret_cast<double*>(out + row) + (lane & 1), scale * ((double)sh + (double)sl));
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[s]);
    if (++rb == nrb) {
      flush_cols(c);
      nrb = (int)G.nrb(++c);
      rb = 0;
      if (i + 1 < cnt) load_x(c);
    }
  }
  if (ok && rb > 0) flush_cols(c);
}

// Two CTAs per SM where the registers allow (the real two-column variant needs more than half
// the register file): twice the warps to hide the consumers' latency (complex T_A product at
// N = 30720: 0.659 ms with one CTA of four stages, 0.585 ms with two CTAs of two stages,
// 0.557 ms with two CTAs of three stages: the measured copy bandwidth).
// CTAs of the first of two jobs (b may be empty): in proportion to their units, at least one each
int gemv_split_ctas(const GemvJob& a, const GemvJob& b, int grid) {
  if (b.units == 0) return grid;
  long long g = (grid * a.units + (a.units + b.units) / 2) / (a.units + b.units);
  g = std::max<long long>(std::max<long long>(1, grid - b.units), std::min<long long>(g, std::min<long long>(grid - 1, a.units)));
  return (int)g;
}

template <int NR, bool REAL, bool CONJ>
cudaError_t launch_sym(GemvJob a, GemvJob b, GemvScratch& w, cudaStream_t s) {
  constexpr int SEG = SBYTES_ROW / (REAL ? 4 : 8);
  constexpr int NCTA = REAL && NR == 2 ? 1 : 2;
  constexpr int SMEM = SymStage<NR, REAL, NCTA>::SMEM;
  auto k = gemv_sym_kernel<NR, REAL, CONJ, NCTA>;
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  static int sms = 0;
  std::call_once(once, [&] {
    attr = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
    int dev = 0;
    if (attr == cudaSuccess) attr = cudaGetDevice(&dev);
    if (attr == cudaSuccess) attr = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  });
  if (attr != cudaSuccess) return attr;
  if (!w.err) return cudaErrorInvalidValue;
  for (GemvJob* q : {&a, &b}) {
    if (q->n <= 0) continue;
    const SymGeom G = sym_geom(q->n, q->ld, SEG);
    q->units = G.off(G.S);
  }
  const int grid = (int)std::max(1LL, std::min<long long>(a.units + b.units, (long long)NCTA * sms));
  k<<<grid, STHREADS, SMEM, s>>>(a, b, gemv_split_ctas(a, b, grid), w.err);
  return cudaGetLastError();
}

template <bool CONJ>
cudaError_t launch_stream_ff(GemvJob a, GemvJob b, GemvScratch& w, cudaStream_t s) {
  constexpr int SEG = FF_ROW / 8;
  auto k = gemv_stream_ff_kernel<CONJ>;
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  static int sms = 0;
  std::call_once(once, [&] {
    attr = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, FF_NST * FF_STAGE + 256);
    int dev = 0;
    if (attr == cudaSuccess) attr = cudaGetDevice(&dev);
    if (attr == cudaSuccess) attr = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  });
  if (attr != cudaSuccess) return attr;
  if (!w.err || !w.xl) return cudaErrorInvalidValue;
  for (GemvJob* q : {&a, &b}) {
    if (q->n <= 0) continue;
    q->units = (long long)((q->n + SROWS - 1) / SROWS) * ((q->ld + SEG - 1) / SEG);
  }
  const int grid = (int)std::max(1LL, std::min<long long>(a.units + b.units, (long long)FF_NCTA * sms));
  k<<<grid, STHREADS, FF_NST * FF_STAGE + 256, s>>>(a, b, gemv_split_ctas(a, b, grid), w.err);
  return cudaGetLastError();
}

GemvJob gemv_job(const void* M, int ld, int n, const GemvScratch& w) {
  return GemvJob{M, w.xh, w.xl, w.out, w.scale, 0, ld, n};
}

template <bool REAL, bool CONJ>
cudaError_t launch_sym_ff(const void* M, const void* Mlo, int ld, int n, int nr, GemvScratch& w, cudaStream_t s) {
  using S = FfStage<REAL>;
  auto k = gemv_sym_ff_kernel<REAL, CONJ>;
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  static int sms = 0;
  std::call_once(once, [&] {
    attr = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, S::SMEM);
    int dev = 0;
    if (attr == cudaSuccess) attr = cudaGetDevice(&dev);
    if (attr == cudaSuccess) attr = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  });
  if (attr != cudaSuccess) return attr;
  if (!w.err || !w.xl || !w.symmetric) return cudaErrorInvalidValue;
  const SymGeom G = sym_geom(n, ld, S::SEG, S::ROWS);
  const long long units = G.off(G.S);
  const int grid = (int)std::max(1LL, std::min<long long>(units, 2LL * sms));
  k<<<dim3(grid, nr), STHREADS, S::SMEM, s>>>(static_cast<const char*>(M), static_cast<const char*>(Mlo), ld, n, w.xh,
                                              w.xl, w.out, w.scale, units, w.err);
  return cudaGetLastError();
}

}  // namespace

template <int NR>
cudaError_t gemv_stream_c64(const float2* M, int ld, int n, bool conj, GemvScratch& w, cudaStream_t s) {
  if (!w.symmetric) return cudaErrorInvalidValue;
  const GemvJob a = gemv_job(M, ld, n, w);
  return conj ? launch_sym<NR, false, true>(a, GemvJob{}, w, s) : launch_sym<NR, false, false>(a, GemvJob{}, w, s);
}
template <int NR>
cudaError_t gemv_stream_r32(const float* M, int ld, int n, GemvScratch& w, cudaStream_t s) {
  if (!w.symmetric) return cudaErrorInvalidValue;
  return launch_sym<NR, true, false>(gemv_job(M, ld, n, w), GemvJob{}, w, s);
}
cudaError_t gemv_stream_c64_ff(const float2* M, int ld, int n, int nr, bool conj, GemvScratch& w, cudaStream_t s) {
  // One complex column takes the full pass: 1.46 ms against 1.8 here at N = 30720, where neither waits for HBM
  // (7.55 GB in 1.11 ms) and the pass over whole rows keeps no column sums.
  const GemvJob a = gemv_job(M, ld, n, w);
  if (nr == 1) return conj ? launch_stream_ff<true>(a, GemvJob{}, w, s) : launch_stream_ff<false>(a, GemvJob{}, w, s);
  return conj ? launch_sym_ff<false, true>(M, nullptr, ld, n, nr, w, s)
              : launch_sym_ff<false, false>(M, nullptr, ld, n, nr, w, s);
}
cudaError_t gemv_stream_r32_ff(const float* hi, const float* lo, int ld, int n, int nr, GemvScratch& w, cudaStream_t s) {
  return launch_sym_ff<true, false>(hi, lo, ld, n, nr, w, s);
}
cudaError_t gemv_stream_pair(const GemvPart& a, const GemvPart& b, int nr, bool conj, GemvMode mode, GemvScratch& w,
                             cudaStream_t s) {
  if (!w.symmetric) return cudaErrorInvalidValue;
  GemvJob J[2];
  for (int i = 0; i < 2; ++i) {
    const GemvPart& p = i ? b : a;
    J[i] = GemvJob{p.M, p.xh, p.xl, p.out, p.scale, 0, padded_ld(p.n), p.n};
  }
  if (mode == GEMV_FF) {
    if (nr != 1) return cudaErrorInvalidValue;
    return conj ? launch_stream_ff<true>(J[0], J[1], w, s) : launch_stream_ff<false>(J[0], J[1], w, s);
  }
  if (nr == 1) return conj ? launch_sym<1, false, true>(J[0], J[1], w, s) : launch_sym<1, false, false>(J[0], J[1], w, s);
  return conj ? launch_sym<2, false, true>(J[0], J[1], w, s) : launch_sym<2, false, false>(J[0], J[1], w, s);
}
template cudaError_t gemv_stream_c64<1>(const float2*, int, int, bool, GemvScratch&, cudaStream_t);
template cudaError_t gemv_stream_c64<2>(const float2*, int, int, bool, GemvScratch&, cudaStream_t);
template cudaError_t gemv_stream_r32<1>(const float*, int, int, GemvScratch&, cudaStream_t);
template cudaError_t gemv_stream_r32<2>(const float*, int, int, GemvScratch&, cudaStream_t);

RF_LAUNCH_READER(launches_gemv_stream)

}  // namespace rfcmp
