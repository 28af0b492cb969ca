// Compressed T_A and V (Sec. 4: the system matrix compressed by an adaptive cross approximation at
// tolerance 1e-4; at extremely low frequency the vector potential compressed apart from the scalar
// one).  Each of T_A (RWG functions) and V (cells) becomes a symmetric hierarchical matrix: a
// cluster tree of its index set, the blocks of the block tree on and above the block diagonal, the
// admissible ones as low-rank crosses U Vt found by ACA with partial pivoting on the GPU, the rest
// dense; a block off the diagonal also stands for its transpose below it, so the compressed
// matrices stay exactly complex symmetric like T_A and V.
//
// Host: cluster trees (median bisection across the longest side of the item centres' extent, items
// carrying support boxes), the admissibility test min(diam a, diam b) <= eta dist(a, b) on
// boxes that do not touch (dist > 0), the block list.  Device: a warp or a CTA per admissible block runs the cross approximation on the
// resident dense matrix (rows and columns gathered through the cluster permutation), blocks whose
// crosses reach the rank cap, or would take at least the block's own entries, stay dense, and the factors and dense blocks are packed into one
// buffer per matrix.  The product y = H x (FP64 accumulation) runs over cross items and row tiles.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <climits>
#include <atomic>
#include <cmath>
#include <cstring>
#include <future>
#include <memory>
#include <mutex>
#include <new>
#include <string>
#include <system_error>
#include <utility>
#include <vector>

#include "rfcmp_internal.h"

namespace rfcmp {

namespace cg = cooperative_groups;

RF_LAUNCH_READER(launches_hmatrix)

// ---------------------------------------------------------------- host partition
namespace {

struct HmNode {
  int start = 0, stop = 0;
  double lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
  int child[2] = {-1, -1};
  double diam = 0.0;  // of the box
};

// Recursive bisection: a cluster of more than `leaf` items is sorted (stably) along the axis of
// the largest extent of its item centres and split at the middle position.
int build_tree(const double* cen, const double* slo, const double* shi, int start, int stop, int leaf,
               std::vector<int32_t>& perm, std::vector<HmNode>& nodes, std::vector<std::pair<double, int32_t>>& keys) {
  const int id = (int)nodes.size();
  nodes.emplace_back();
  HmNode node;
  node.start = start;
  node.stop = stop;
  for (int d = 0; d < 3; ++d) {
    node.lo[d] = HUGE_VAL;
    node.hi[d] = -HUGE_VAL;
  }
  double clo[3] = {HUGE_VAL, HUGE_VAL, HUGE_VAL}, chi[3] = {-HUGE_VAL, -HUGE_VAL, -HUGE_VAL};
  for (int p = start; p < stop; ++p) {
    const int i = perm[p];
    for (int d = 0; d < 3; ++d) {
      node.lo[d] = std::min(node.lo[d], slo[3 * i + d]);
      node.hi[d] = std::max(node.hi[d], shi[3 * i + d]);
      clo[d] = std::min(clo[d], cen[3 * i + d]);
      chi[d] = std::max(chi[d], cen[3 * i + d]);
    }
  }
  {
    double d2 = 0.0;
    for (int d = 0; d < 3; ++d) d2 += (node.hi[d] - node.lo[d]) * (node.hi[d] - node.lo[d]);
    node.diam = std::sqrt(d2);
  }
  if (stop - start > leaf) {
    int axis = 0;  // the first axis of the largest extent
    for (int d = 1; d < 3; ++d)
      if (chi[d] - clo[d] > chi[axis] - clo[axis]) axis = d;
    keys.resize(stop - start);  // (coordinate, item): the sort reads each coordinate once
    for (int p = start; p < stop; ++p) keys[p - start] = {cen[3 * perm[p] + axis], perm[p]};
    std::stable_sort(keys.begin(), keys.end(), [](const auto& a, const auto& b) { return a.first < b.first; });
    for (int p = start; p < stop; ++p) perm[p] = keys[p - start].second;
    const int mid = start + (stop - start) / 2;
    node.child[0] = build_tree(cen, slo, shi, start, mid, leaf, perm, nodes, keys);
    node.child[1] = build_tree(cen, slo, shi, mid, stop, leaf, perm, nodes, keys);
  }
  nodes[id] = node;
  return id;
}

double box_distance(const HmNode& a, const HmNode& b) {
  double s = 0.0;
  for (int d = 0; d < 3; ++d) {
    const double g = std::max(0.0, std::max(a.lo[d] - b.hi[d], b.lo[d] - a.hi[d]));
    s += g * g;
  }
  return std::sqrt(s);
}

struct HmBlockHost {
  int r0, r1, c0, c1;
  int admissible;
};

// Leaves of the block tree on and above the block diagonal (r0 <= c0), ordered by (r0, c0).  A pair
// that is not admissible splits into the children of whichever clusters have children; two leaves
// that are not admissible form a dense block.
std::vector<HmBlockHost> block_list(const std::vector<HmNode>& nodes, double eta) {
  std::vector<HmBlockHost> out;
  if (nodes.empty() || nodes[0].stop == 0) return out;
  std::vector<std::pair<int, int>> stack{{0, 0}};
  while (!stack.empty()) {
    const auto [ia, ib] = stack.back();
    stack.pop_back();
    const HmNode &a = nodes[ia], &b = nodes[ib];
    if (a.start > b.start) continue;  // below the diagonal: the transpose of a mirrored block
    const double dist = box_distance(a, b);
    if (dist > 0.0 && std::min(a.diam, b.diam) <= eta * dist) {  // boxes that touch: never
      out.push_back({a.start, a.stop, b.start, b.stop, 1});
    } else if (a.child[0] < 0 && b.child[0] < 0) {
      out.push_back({a.start, a.stop, b.start, b.stop, 0});
    } else {
      const int as[2] = {a.child[0] < 0 ? ia : a.child[0], a.child[1]};
      const int bs[2] = {b.child[0] < 0 ? ib : b.child[0], b.child[1]};
      const int na = a.child[0] < 0 ? 1 : 2, nb = b.child[0] < 0 ? 1 : 2;
      for (int x = 0; x < na; ++x)
        for (int y = 0; y < nb; ++y) stack.push_back({as[x], bs[y]});
    }
  }
  std::sort(out.begin(), out.end(), [](const HmBlockHost& p, const HmBlockHost& q) {
    return p.r0 != q.r0 ? p.r0 < q.r0 : p.c0 < q.c0;
  });
  return out;
}

int check_partition_args(int64_t n, int32_t leaf, double eta) {
  if (n < 0 || n > (int64_t)INT32_MAX) return set_error(RFCMP_ERR_INVALID_ARG, "item count out of range");
  if (leaf < 1 || leaf > 65536) return set_error(RFCMP_ERR_INVALID_ARG, "leaf must be in [1, 65536]");
  if (!(eta >= 0.0) || !std::isfinite(eta)) return set_error(RFCMP_ERR_INVALID_ARG, "eta must be finite and >= 0");
  return RFCMP_OK;
}

void partition(const double* cen, const double* slo, const double* shi, int n, int leaf, double eta,
               std::vector<int32_t>& perm, std::vector<HmBlockHost>& blocks) {
  perm.resize(n);
  for (int i = 0; i < n; ++i) perm[i] = i;
  std::vector<HmNode> nodes;
  std::vector<std::pair<double, int32_t>> keys;
  if (n > 0) build_tree(cen, slo, shi, 0, n, leaf, perm, nodes, keys);
  blocks = block_list(nodes, eta);
}

}  // namespace
}  // namespace rfcmp

// ---------------------------------------------------------------- device
namespace rfcmp {
namespace {

constexpr int HM_THREADS = 256;
constexpr int HM_MAX_RANK = 256;              // largest rank cap a caller may ask for
constexpr int HM_MAX_ITER = HM_MAX_RANK + 16;  // crosses plus rows skipped for a zero residual
constexpr unsigned FULL = 0xffffffffu;

// one block of the compressed form: rows [r0, r1) and columns [c0, c1) in cluster order; rank < 0
// for a dense block (m x n row-major at off), else U (rank x m, one cross per row of U) at off and
// Vt (rank x n) at off + rank m; t0: its first entry of a product's cross sums (rank of Vt x, rank
// of U x)
struct HmBlockDev {
  int32_t r0, r1, c0, c1;
  int32_t rank, t0;
  long long off;
};

__device__ __forceinline__ void argmax_merge(float& v, int& i, float v2, int i2) {
  if (v2 > v || (v2 == v && i2 < i)) {
    v = v2;
    i = i2;
  }
}

// largest v over the CTA (ties: smallest i); every thread receives it
__device__ void block_argmax(float v, int i, float* sv, int* si, float& bv, int& bi) {
  for (int o = 16; o > 0; o >>= 1) argmax_merge(v, i, __shfl_down_sync(FULL, v, o), __shfl_down_sync(FULL, i, o));
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) {
    sv[w] = v;
    si[w] = i;
  }
  __syncthreads();
  if (w == 0) {
    v = l < HM_THREADS / 32 ? sv[l] : -1.f;
    i = l < HM_THREADS / 32 ? si[l] : INT_MAX;
    for (int o = 16; o > 0; o >>= 1) argmax_merge(v, i, __shfl_down_sync(FULL, v, o), __shfl_down_sync(FULL, i, o));
    if (l == 0) {
      sv[HM_THREADS / 32] = v;
      si[HM_THREADS / 32] = i;
    }
  }
  __syncthreads();
  bv = sv[HM_THREADS / 32];
  bi = si[HM_THREADS / 32];
  __syncthreads();
}

__device__ __forceinline__ float2 cmulf(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}

__device__ __forceinline__ bool row_used(const int* used, int nused, int p) {
  for (int k = 0; k < nused; ++k)
    if (used[k] == p) return true;
  return false;
}

// FP32 -> FP64 by moving the bits: exponent rebased by 896, mantissa shifted by 29.  Zeros,
// subnormals, infinities and NaN take the conversion instruction.
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f);
  if ((u & 0x7f800000u) - 0x00800000u >= 0x7f000000u) return (double)f;
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}

// Warp sums of V = 2^k values a lane: afterwards v[0] of lane l is the sum of value l * V / 32 (each
// exchange halves the values a lane holds: V - 1 + max(0, 5 - k) additions instead of 5 V).
template <int V>
__device__ __forceinline__ void warp_sums(double (&v)[V], int lane) {
#pragma unroll
  for (int step = 0; step < 5; ++step) {
    const int off = 16 >> step, h = V >> (step + 1);
    if (h == 0) {
      v[0] += __shfl_xor_sync(FULL, v[0], off);
    } else {
      const bool up = (lane & off) != 0;
#pragma unroll
      for (int k = 0; k < h; ++k) {
        const double send = up ? v[k] : v[k + h], keep = up ? v[k + h] : v[k];
        v[k] = keep + __shfl_xor_sync(FULL, send, off);
      }
    }
  }
}

constexpr int ACA_SMALL = 128;  // blocks of at most this many rows and columns take one warp
constexpr int ACA_GROUP = 8;    // crosses whose four norm products a warp sums together

// ACA with partial pivoting of one admissible block per team of WARPS warps (a CTA holds 8 / WARPS
// teams), on the dense matrix A (row stride ld) through the cluster permutation.  The crosses go to the
// block's slot: U (cap x m) at slot[b], Vt (cap x n) after it.  rank_out[b] = crosses kept, status_out[b]
// = 0 when the stopping rule ||u|| ||v|| <= eps ||S||_F held (or every row was used), 1 when the rank cap
// or the iteration cap ended the loop first.  All loops are bounded by the caps and the block's size.
//
// Most blocks are a few dozen rows: a CTA each left seven of its eight warps idle and cost a reduction
// of FP64 sums over all of them per earlier cross, 160 warp additions on the slow FP64 pipe, which bound
// the kernel.  A warp per small block synchronises with itself only, and the products of eight earlier
// crosses are summed together, 31 additions.  GB300, T_A and V of 7680 functions and 5120 cells: 8.75 ->
// 1.94 ms.
template <int WARPS>
__global__ void __launch_bounds__(HM_THREADS)
    hm_aca_kernel(const float2* __restrict__ A, long long ld, const int32_t* __restrict__ perm,
                  const HmBlockDev* __restrict__ blk, const int32_t* __restrict__ list, int nlist,
                  const long long* __restrict__ slot, int cap, int iter_cap, float eps, float2* __restrict__ slots,
                  int32_t* __restrict__ rank_out, int32_t* __restrict__ status_out) {
  RF_COUNT_LAUNCH();
  constexpr int T = 32 * WARPS;  // threads of a team
  __shared__ float sv[HM_THREADS / 32 + 1];
  __shared__ int si[HM_THREADS / 32 + 1];
  __shared__ double sd[WARPS][33];
  __shared__ int used[WARPS == 1 ? 1 : HM_MAX_ITER];
  __shared__ int s_next;
  const int team = blockIdx.x * (HM_THREADS / T) + threadIdx.x / T;
  if (team >= nlist) return;  // whole teams only
  const int b = list[team], tid = threadIdx.x % T, lane = threadIdx.x & 31, w = tid >> 5;
  auto sync = [] {
    if (WARPS == 1) __syncwarp();
    else __syncthreads();
  };
  // largest v over the team (ties: smallest i); every thread receives it
  auto argmax = [&](float v, int i, float& bv, int& bi) {
    if (WARPS == 1) {
      for (int o = 16; o > 0; o >>= 1) argmax_merge(v, i, __shfl_xor_sync(FULL, v, o), __shfl_xor_sync(FULL, i, o));
      bv = v;
      bi = i;
    } else {
      block_argmax(v, i, sv, si, bv, bi);
    }
  };
  // sums over the team of 32 values a thread, value l in lane l of every warp
  auto team_sums = [&](double (&v)[32]) -> double {
    warp_sums<32>(v, lane);
    if (WARPS == 1) return v[0];
    sd[w][lane] = v[0];
    __syncthreads();
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < WARPS; ++k) s += sd[k][lane];
    __syncthreads();
    return s;
  };
  const HmBlockDev B = blk[b];
  const int m = B.r1 - B.r0, n = B.c1 - B.c0;
  const int32_t* rp = perm + B.r0;
  const int32_t* cp = perm + B.c0;
  float2* U = slots + slot[b];
  float2* Vt = U + (size_t)cap * m;
  int rank = 0, nused = 0, status = 1, i = 0;
  unsigned mine = 0;   // one warp: bit q for row lane + 32 q, set once the row was a pivot row
  double norm2 = 0.0;  // ||S_rank||_F^2, the same in every thread
  auto is_used = [&](int p) { return WARPS == 1 ? (mine >> (p >> 5) & 1u) != 0 : row_used(used, nused, p); };
  for (int it = 0; it < iter_cap && rank < cap; ++it) {
    if (WARPS == 1) {
      if ((i & 31) == lane) mine |= 1u << (i >> 5);
    } else if (tid == 0) {
      used[nused] = i;
    }
    ++nused;
    // residual row i into the next cross's Vt row, and its largest entry
    float bv = -1.f;
    int bj = INT_MAX;
    const float2* Arow = A + (size_t)rp[i] * ld;
    for (int j = tid; j < n; j += T) {
      float2 r = Arow[cp[j]];
#pragma unroll 4
      for (int l = 0; l < rank; ++l) {
        const float2 p = cmulf(U[(size_t)l * m + i], Vt[(size_t)l * n + j]);
        r.x -= p.x;
        r.y -= p.y;
      }
      Vt[(size_t)rank * n + j] = r;
      argmax_merge(bv, bj, r.x * r.x + r.y * r.y, j);
    }
    sync();
    int js;
    argmax(bv, bj, bv, js);
    if (!(bv >= FLT_MIN)) {
      // the residual vanishes on this row (to below the normal range, where 1 / pivot would
      // overflow): the next row not yet used
      if (WARPS == 1) {
        int c = INT_MAX;
        for (int p = lane; p < m && c == INT_MAX; p += 32)
          if (!is_used(p)) c = p;
        c = __reduce_min_sync(FULL, c);
        i = c == INT_MAX ? -1 : c;
      } else {
        if (tid == 0) {
          int c = -1;
          for (int p = 0; p < m && c < 0; ++p)
            if (!row_used(used, nused, p)) c = p;
          s_next = c;
        }
        __syncthreads();
        i = s_next;
        __syncthreads();
      }
      if (i < 0) {
        status = 0;  // every row reproduced
        break;
      }
      continue;
    }
    const float2 piv = Vt[(size_t)rank * n + js];
    sync();  // every thread holds the pivot before its entry is rescaled
    const float dd = piv.x * piv.x + piv.y * piv.y;
    const float2 ip = make_float2(piv.x / dd, -piv.y / dd);
    double nrm[2] = {0.0, 0.0};  // |u|^2, |v|^2 of this thread's entries
    for (int j = tid; j < n; j += T) {
      const float2 v = cmulf(Vt[(size_t)rank * n + j], ip);
      Vt[(size_t)rank * n + j] = v;
      const double x = widen(v.x), y = widen(v.y);
      nrm[1] = fma(x, x, fma(y, y, nrm[1]));
    }
    sync();
    // residual column js into the next cross's U row, and the next pivot row
    float bu = -1.f;
    int bp = INT_MAX;
    for (int p = tid; p < m; p += T) {
      float2 u = A[(size_t)rp[p] * ld + cp[js]];
#pragma unroll 4
      for (int l = 0; l < rank; ++l) {
        const float2 q = cmulf(Vt[(size_t)l * n + js], U[(size_t)l * m + p]);
        u.x -= q.x;
        u.y -= q.y;
      }
      U[(size_t)rank * m + p] = u;
      const double x = widen(u.x), y = widen(u.y);
      nrm[0] = fma(x, x, fma(y, y, nrm[0]));
      if (!is_used(p)) argmax_merge(bu, bp, u.x * u.x + u.y * u.y, p);
    }
    sync();  // the new cross is complete in global memory
    // ||S + u v^T||^2 = ||S||^2 + 2 Re sum_l (u_l^H u)(v_l^H v) + ||u||^2 ||v||^2: the four products of
    // up to ACA_GROUP earlier crosses at a time, the norms in the first group's last places
    double cross = 0.0, uu = 0.0, vv = 0.0;
    for (int l0 = 0; l0 == 0 || l0 < rank; l0 += l0 == 0 ? ACA_GROUP - 1 : ACA_GROUP) {
      const int nl = min(l0 == 0 ? ACA_GROUP - 1 : ACA_GROUP, rank - l0);
      double c[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) c[k] = 0.0;
      for (int p = tid; p < m; p += T) {
        const float2 ub = U[(size_t)rank * m + p];
        const double x = widen(ub.x), y = widen(ub.y);
#pragma unroll
        for (int l = 0; l < ACA_GROUP; ++l) {
          if (l >= nl) break;
          const float2 ua = U[(size_t)(l0 + l) * m + p];
          const double ax = widen(ua.x), ay = widen(ua.y);
          c[4 * l] = fma(ax, x, fma(ay, y, c[4 * l]));  // conj(a) b
          c[4 * l + 1] = fma(ax, y, fma(-ay, x, c[4 * l + 1]));
        }
      }
      for (int j = tid; j < n; j += T) {
        const float2 vb = Vt[(size_t)rank * n + j];
        const double x = widen(vb.x), y = widen(vb.y);
#pragma unroll
        for (int l = 0; l < ACA_GROUP; ++l) {
          if (l >= nl) break;
          const float2 va = Vt[(size_t)(l0 + l) * n + j];
          const double ax = widen(va.x), ay = widen(va.y);
          c[4 * l + 2] = fma(ax, x, fma(ay, y, c[4 * l + 2]));
          c[4 * l + 3] = fma(ax, y, fma(-ay, x, c[4 * l + 3]));
        }
      }
      if (l0 == 0) {
        c[30] = nrm[0];
        c[31] = nrm[1];
      }
      const double s = team_sums(c);
      // lanes 4 l .. 4 l + 3 hold c0 .. c3 of cross l: c0 c2 - c1 c3
      const double t = __shfl_down_sync(FULL, s, 2);
      double q = lane & 1 ? -s * t : s * t;
      if ((lane & 3) > 1 || (lane >> 2) >= nl) q = 0.0;
      for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(FULL, q, o);
      cross += q;
      if (l0 == 0) {
        uu = __shfl_sync(FULL, s, 30);
        vv = __shfl_sync(FULL, s, 31);
      }
    }
    norm2 += 2.0 * cross + uu * vv;
    ++rank;
    if (sqrt(uu * vv) <= (double)eps * sqrt(fmax(norm2, 0.0))) {
      status = 0;
      break;
    }
    int np;
    argmax(bu, bp, bu, np);
    if (bu < 0.f) {
      status = 0;  // every row used
      break;
    }
    i = np;
  }
  if (tid == 0) {
    rank_out[b] = rank;
    status_out[b] = status;
  }
}

// Packs the final blocks into one buffer: a dense block gathered from A (m x n row-major), a
// low-rank block copied from its slot (the first rank rows of U and of Vt).
__global__ void __launch_bounds__(HM_THREADS)
    hm_pack_kernel(const float2* __restrict__ A, long long ld, const int32_t* __restrict__ perm,
                   const HmBlockDev* __restrict__ blk, const long long* __restrict__ slot, int cap,
                   const float2* __restrict__ slots, float2* __restrict__ out) {
  RF_COUNT_LAUNCH();
  const HmBlockDev B = blk[blockIdx.x];
  const int m = B.r1 - B.r0, n = B.c1 - B.c0;
  float2* dst = out + B.off;
  if (B.rank < 0) {
    const long long total = (long long)m * n;
    for (long long e = threadIdx.x; e < total; e += HM_THREADS) {
      const int i = (int)(e / n), j = (int)(e % n);
      dst[e] = A[(size_t)perm[B.r0 + i] * ld + perm[B.c0 + j]];
    }
  } else {
    const float2* U = slots + slot[blockIdx.x];
    const float2* Vt = U + (size_t)cap * m;
    const long long nu = (long long)B.rank * m, nv = (long long)B.rank * n;
    for (long long e = threadIdx.x; e < nu; e += HM_THREADS) dst[e] = U[e];
    for (long long e = threadIdx.x; e < nv; e += HM_THREADS) dst[nu + e] = Vt[e];
  }
}

// ---- the product y = H x ----
// Three launches per group of columns (at most HM_COLS columns a group):
//   hm_gather   x into cluster order, the columns of a group interleaved
//   hm_cross    t = Vt x[c0..c1) and t' = U x[r0..r1) of every low-rank block, one warp per four
//               crosses of one side, so an x entry is read once for four crosses
//   hm_rows     y of one tile of at most 32 rows per CTA or cluster of CTAs: every block that covers the tile adds U t
//               (or Vt^T t' below the diagonal, or its dense entries), lane = row, the blocks dealt to
//               its warps; one store per row through the permutation
// Every stored entry is used once per side, so no sum crosses a cluster: no atomics, no zeroed output,
// and a product is the same bits on every run.  Bound: the FP64 pipe (2 lanes per clock and SM, 90 to
// 93 % busy), 8 multiply-adds per stored entry and column; the FP32 entries are widened with integer
// operations, which keeps the conversions off that pipe.  Measured on GB300: both products of an
// ellipsoid of 17280 functions and 11520 cells (47.8 M stored entries), 8 columns: 10.1 ms; one CTA
// per block and column with a row a thread and FP64 atomics took 20.2 ms.
constexpr int HM_COLS = 4;        // columns of a group
constexpr int HM_TILE = 32;       // rows of a tile (one lane each)
constexpr int HM_CROSS = 4;       // crosses of one warp's item
constexpr int HM_CROSS_THREADS = 128;
constexpr int HM_ROW_WARPS = HM_THREADS / 32;
constexpr size_t HM_SCRATCH = (size_t)256 << 20;  // cross sums of one pass over the columns

struct HmTile {
  int32_t row0, rows;      // rows [row0, row0 + rows) in cluster order
  int32_t begin, end;      // its entries of the cover list: 2 block + (1: as columns)
};

// xp: group g (columns 4 g ..) at 4 g n, entry p, column c of the group at p * (columns of the group) + c
__global__ void hm_gather_kernel(const double2* __restrict__ x, const int32_t* __restrict__ perm, int n, int nrhs,
                                 double2* __restrict__ xp) {
  RF_COUNT_LAUNCH();
  const long long total = (long long)n * nrhs;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(e / n), p = (int)(e - (long long)c * n);
    const int g = c / HM_COLS, nc = min(HM_COLS, nrhs - g * HM_COLS);
    xp[(size_t)g * HM_COLS * n + (size_t)p * nc + (c - g * HM_COLS)] = x[(size_t)c * n + perm[p]];
  }
}

// t[(l0 + q) nrhs + c] = sum_j f[q len + j] x[j NC + c] for q < nl crosses (NC columns)
template <int NC>
__device__ __forceinline__ void cross_dots(const float2* __restrict__ f, int len, int nl, const double2* __restrict__ x,
                                           double2* __restrict__ t, int nrhs, int lane) {
  constexpr int V = HM_CROSS * (NC == 3 ? 4 : NC) * 2;
  double acc[V];
#pragma unroll
  for (int k = 0; k < V; ++k) acc[k] = 0.0;
  for (int j = lane; j < len; j += 32) {
    double2 xv[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) xv[c] = x[(size_t)j * NC + c];
#pragma unroll
    for (int q = 0; q < HM_CROSS; ++q) {
      const float2 e = q < nl ? f[(size_t)q * len + j] : make_float2(0.f, 0.f);
      if (q >= nl) continue;
      const double er = widen(e.x), ei = widen(e.y);
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        double& re = acc[(q * (NC == 3 ? 4 : NC) + c) * 2];
        double& im = acc[(q * (NC == 3 ? 4 : NC) + c) * 2 + 1];
        re = fma(er, xv[c].x, fma(-ei, xv[c].y, re));
        im = fma(er, xv[c].y, fma(ei, xv[c].x, im));
      }
    }
  }
  warp_sums<V>(acc, lane);
  if (V < 32 && (lane & (32 / V - 1))) return;
  const int v = lane * V / 32, q = v / (V / HM_CROSS), c = (v / 2) % (V / HM_CROSS / 2);
  if (q < nl && c < NC) reinterpret_cast<double*>(t + (size_t)q * nrhs + c)[v & 1] = acc[0];
}

// items: x = 2 block + (1: U, the row side), y = first cross
__global__ void __launch_bounds__(HM_CROSS_THREADS)
    hm_cross_kernel(const HmBlockDev* __restrict__ blk, const int2* __restrict__ items, int nitems,
                    const float2* __restrict__ H, const double2* __restrict__ xp, double2* __restrict__ t, int n,
                    int nrhs) {
  RF_COUNT_LAUNCH();
  const int it = blockIdx.x * (HM_CROSS_THREADS / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (it >= nitems) return;
  const int2 item = items[it];
  const HmBlockDev B = blk[item.x >> 1];
  const int side = item.x & 1, m = B.r1 - B.r0, nn = B.c1 - B.c0, len = side ? m : nn;
  const int g = blockIdx.y * HM_COLS, nc = min(HM_COLS, nrhs - g), nl = min(HM_CROSS, B.rank - item.y);
  const float2* f = H + B.off + (side ? 0 : (size_t)B.rank * m) + (size_t)item.y * len;
  const double2* x = xp + (size_t)g * n + (size_t)(side ? B.r0 : B.c0) * nc;
  double2* o = t + ((size_t)B.t0 + (side ? B.rank : 0) + item.y) * nrhs + g;
  switch (nc) {
    case 1: return cross_dots<1>(f, len, nl, x, o, nrhs, lane);
    case 2: return cross_dots<2>(f, len, nl, x, o, nrhs, lane);
    case 3: return cross_dots<3>(f, len, nl, x, o, nrhs, lane);
    default: return cross_dots<4>(f, len, nl, x, o, nrhs, lane);
  }
}

template <int NC>
__device__ __forceinline__ void madd(double (&acc)[2 * HM_COLS], float2 e, const double2* __restrict__ x) {
  const double er = widen(e.x), ei = widen(e.y);
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const double2 v = x[c];
    acc[2 * c] = fma(er, v.x, fma(-ei, v.y, acc[2 * c]));
    acc[2 * c + 1] = fma(er, v.y, fma(ei, v.x, acc[2 * c + 1]));
  }
}

// The sums of one row (row0 + `row`) of a tile over the cover entries begin + first, begin + first + step, ...  Each entry
// is `count` products of a stored value (f, fs values apart) and NC columns (x, xs values apart), so that groups of
// lanes with entries of different kinds run one loop.
template <int NC>
__device__ __forceinline__ void tile_rows(const HmTile& T, const int32_t* __restrict__ cover,
                                          const HmBlockDev* __restrict__ blk, const float2* __restrict__ H,
                                          const double2* __restrict__ xg, const double2* __restrict__ t, int nrhs,
                                          int first, int step, int row, double (&acc)[2 * HM_COLS]) {
  for (int q = T.begin + first; q < T.end; q += step) {
    const int code = cover[q];
    const HmBlockDev B = blk[code >> 1];
    const int cols = code & 1, m = B.r1 - B.r0, nn = B.c1 - B.c0;
    const int i = T.row0 + row - (cols ? B.c0 : B.r0);
    const float2* f = H + B.off + i;
    const double2* x = xg + (size_t)(cols ? B.r0 : B.c0) * NC;
    int count = cols ? m : nn, fs = nn, xs = NC;
    if (B.rank >= 0) {  // U t, or Vt^T t' below the diagonal
      if (cols) f += (size_t)B.rank * m;
      else fs = m;
      x = t + ((size_t)B.t0 + (cols ? B.rank : 0)) * nrhs;
      count = B.rank;
      xs = nrhs;
    } else if (!cols && B.r0 != B.c0) {  // along a row; a diagonal block is symmetric, a transposed one lies so
      f += (size_t)i * (nn - 1);
      fs = 1;
    }
#pragma unroll 4
    for (int l = 0; l < count; ++l, f += fs, x += xs) madd<NC>(acc, *f, x);
  }
}

// A cluster of CTAs per tile and group, the cover entries dealt to all their warps; the first adds their sums in order.
// Where a tile has at most 16 or 8 rows (small leaves) and more entries than warps, a warp takes two or four entries at
// a time, one per 16 or 8 lanes: leaves of 8, both products of 14520 functions and 9680 cells, one column, 3.4 ms
// with an entry a warp and 1.5 so.
__global__ void __launch_bounds__(HM_THREADS)
    hm_rows_kernel(const HmTile* __restrict__ tiles, const int32_t* __restrict__ cover,
                   const HmBlockDev* __restrict__ blk, const float2* __restrict__ H, const double2* __restrict__ xp,
                   const double2* __restrict__ t, const int32_t* __restrict__ perm, double2* __restrict__ y, int n,
                   int nrhs) {
  RF_COUNT_LAUNCH();
  __shared__ double part[HM_ROW_WARPS][2 * HM_COLS][HM_TILE];
  __shared__ double sums[HM_THREADS];
  const cg::cluster_group cl = cg::this_cluster();
  const int team = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const HmTile T = tiles[blockIdx.x / team];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = blockIdx.y * HM_COLS, nc = min(HM_COLS, nrhs - g);
  const double2* xg = xp + (size_t)g * n;
  const bool many = T.end - T.begin > HM_ROW_WARPS * team;
  const int R = many && T.rows <= 8 ? 8 : (many && T.rows <= 16 ? 16 : HM_TILE), subs = HM_TILE / R;  // lanes of an entry
  const int first = (w * team + rank) * subs + lane / R, step = HM_ROW_WARPS * team * subs;
  const int row = lane % R < T.rows ? lane % R : 0;
  double acc[2 * HM_COLS];
#pragma unroll
  for (int k = 0; k < 2 * HM_COLS; ++k) acc[k] = 0.0;
  switch (nc) {
    case 1: tile_rows<1>(T, cover, blk, H, xg, t + g, nrhs, first, step, row, acc); break;
    case 2: tile_rows<2>(T, cover, blk, H, xg, t + g, nrhs, first, step, row, acc); break;
    case 3: tile_rows<3>(T, cover, blk, H, xg, t + g, nrhs, first, step, row, acc); break;
    default: tile_rows<4>(T, cover, blk, H, xg, t + g, nrhs, first, step, row, acc); break;
  }
#pragma unroll
  for (int k = 0; k < 2 * HM_COLS; ++k) part[w][k][lane] = acc[k];
  __syncthreads();
  static_assert(HM_THREADS == 2 * HM_COLS * HM_TILE, "one thread per (value, row) of a tile");
  const int k = threadIdx.x / HM_TILE, i = threadIdx.x % HM_TILE;
  double s = 0.0;
#pragma unroll
  for (int v = 0; v < HM_ROW_WARPS; ++v) s += part[v][k][i];
  for (int z = i + R; i < R && z < HM_TILE; z += R)  // the other entries of the warps
#pragma unroll
    for (int v = 0; v < HM_ROW_WARPS; ++v) s += part[v][k][z];
  if (team > 1) {
    sums[threadIdx.x] = s;
    cl.sync();
    if (rank == 0)
      for (int r = 1; r < team; ++r) s += cl.map_shared_rank(sums, r)[threadIdx.x];
    cl.sync();  // no CTA leaves while its sums may be read
    if (rank != 0) return;
  }
  if (i >= T.rows || k >= 2 * nc) return;
  reinterpret_cast<double*>(y + (size_t)(g + k / 2) * n + perm[T.row0 + i])[k & 1] = s;
}

// The FP64 pipe of an SM works on a tile as long as its CTAs are there: small matrices have fewer tiles than SMs
// (1080 functions: about 60).  Up to 8 CTAs share a tile while there are fewer than 4 an SM: 1080 functions and 720
// cells, both products of one and of four columns 128 and 302 us with one CTA a tile, 77 and 151 so; 18000
// functions and 12000 cells, one column 1.09 and 1.03 ms.  Cutting the entries into pieces of 16 or 32 terms as
// well gave nothing.
// CTAs beyond the entries of every tile would have no work (225 functions in four blocks a row, 40 columns: 90 us with 8
// CTAs a tile, 49 with 4).
int hm_team(long long ctas, int entries) {
  int team = 1;
  while (team < 8 && ctas * team < 4 * 152 && team < entries) team *= 2;
  return team;
}

}  // namespace

// one compressed matrix (T_A or V)
struct HmPart {
  int n = 0;
  int nblocks = 0;
  int32_t* perm = nullptr;       // cluster order -> original index (device)
  HmBlockDev* blocks = nullptr;  // (device)
  float2* data = nullptr;        // dense blocks and crosses (device)
  int2* items = nullptr;         // cross items of the low-rank blocks, longest first (device)
  HmTile* tiles = nullptr;       // row tiles (device)
  int32_t* cover = nullptr;      // blocks over each tile (device)
  int nitems = 0, ntiles = 0, entries = 0, ncross = 0;  // entries: most over one tile
  long long elems = 0;
  int64_t n_lowrank = 0, n_dense = 0, n_capped = 0, n_small = 0;
  int max_rank = 0;
  uint64_t bytes = 0;
};

#define HM_CUDA(call)                                                                                \
  do {                                                                                               \
    cudaError_t e_ = (call);                                                                         \
    if (e_ != cudaSuccess) return set_error(RFCMP_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

// Frees the temporaries of one build on every path out of it.
struct HmTemps {
  std::vector<void*> p;
  ~HmTemps() { clear(); }
  void clear() {
    for (void* q : p) dev_free(q);
    p.clear();
  }
  template <class T>
  cudaError_t alloc(T** q, size_t bytes) {
    cudaError_t e = dev_malloc(q, bytes);
    if (e == cudaSuccess) p.push_back(*q);
    return e;
  }
};

// What a product runs over.  Tiles: at most 32 rows that no block boundary cuts, each with the blocks
// that cover it (2 block, + 1 where the tile lies in the block's columns).
struct CoverLists {
  std::vector<HmTile> tiles;
  std::vector<int32_t> cover;
};

CoverLists cover_lists(const std::vector<HmBlockHost>& blk, int n) {
  CoverLists L;
  std::vector<uint8_t> cut((size_t)n + 1, 0);
  for (const HmBlockHost& B : blk) cut[B.r0] = cut[B.r1] = cut[B.c0] = cut[B.c1] = 1;
  std::vector<int32_t> first((size_t)n + 1, 0);  // first[p]: tiles that start below p
  for (int p = 0; p < n;) {
    int q = p + 1;
    while (q < n && q - p < HM_TILE && !cut[q]) ++q;
    for (int i = p + 1; i <= q; ++i) first[i] = (int32_t)L.tiles.size() + 1;
    L.tiles.push_back({p, q - p, 0, 0});
    p = q;
  }
  auto each = [&](auto&& f) {
    for (size_t b = 0; b < blk.size(); ++b) {
      const HmBlockHost& B = blk[b];
      for (int i = first[B.r0]; i < first[B.r1]; ++i) f(i, (int32_t)(2 * b));
      if (B.r0 != B.c0)
        for (int i = first[B.c0]; i < first[B.c1]; ++i) f(i, (int32_t)(2 * b + 1));
    }
  };
  each([&](int i, int32_t) { ++L.tiles[i].end; });
  int32_t total = 0;
  for (HmTile& t : L.tiles) {
    const int32_t c = t.end;
    t.begin = t.end = total;
    total += c;
  }
  L.cover.resize(total);
  each([&](int i, int32_t code) { L.cover[L.tiles[i].end++] = code; });
  return L;
}

// The cross items of the low-rank blocks, the longest first (by binary order of magnitude), so that
// the last ones to run are short.
std::vector<int2> cross_items(const std::vector<HmBlockDev>& blk) {
  size_t count[32] = {}, at[32], total = 0;
  auto each = [&](auto&& f) {
    for (size_t b = 0; b < blk.size(); ++b)
      for (int side = 0; side < 2 && blk[b].rank > 0; ++side) {
        int len = side ? blk[b].r1 - blk[b].r0 : blk[b].c1 - blk[b].c0, mag = 0;
        for (; len > 1; len >>= 1) ++mag;
        for (int l = 0; l < blk[b].rank; l += HM_CROSS) f(mag, make_int2((int)(2 * b) + side, l));
      }
  };
  each([&](int mag, int2) { ++count[mag]; });
  for (int mag = 31; mag >= 0; --mag) {
    at[mag] = total;
    total += count[mag];
  }
  std::vector<int2> items(total);
  each([&](int mag, int2 v) { items[at[mag]++] = v; });
  return items;
}

// One matrix on its way to the compressed form: the partition (host), the cross approximations (queued
// on the legacy stream) and what the packing reads.
struct PartBuild {
  std::vector<int32_t> perm;
  std::vector<HmBlockHost> blocks;
  std::vector<HmBlockDev> cand;  // the admissible blocks
  std::vector<long long> slot;
  int32_t *rank_d = nullptr, *status_d = nullptr;
  float2* slots = nullptr;
  CoverLists lists;
  HmTemps tmp;
};

// Queues the cross approximations of the dense n x n matrix A (row stride ld, both triangles stored)
// partitioned in b.  owned receives the part's device buffers; budget_left bounds the bytes it may hold
// at the peak of the build.
int start_part(const float2* A, int ld, int n, const rfcmp_hm_opts& o, uint64_t budget_left, PartBuild& b, HmPart& out,
               std::vector<void*>& owned) {
  out.n = n;
  const int cap = o.max_rank;
  std::vector<int32_t> order;  // candidates, the large ones (a CTA each) before the small ones (a warp each)
  long long slot_elems = 0, worst = 0;
  uint64_t item_bytes = 0;
  for (const HmBlockHost& h : b.blocks) {
    const long long m = h.r1 - h.r0, nn = h.c1 - h.c0;
    worst += m * nn;  // at worst every block is stored dense
    if (h.admissible) {
      b.cand.push_back({h.r0, h.r1, h.c0, h.c1, 0, 0, 0});
      b.slot.push_back(slot_elems);
      slot_elems += (long long)cap * (m + nn);
      // a low-rank block keeps fewer crosses than make its own entries
      const long long most = std::min<long long>(cap, m * nn / (m + nn));
      item_bytes += 2 * sizeof(int2) * (uint64_t)((most + HM_CROSS - 1) / HM_CROSS);
    }
  }
  if (budget_left != UINT64_MAX) {
    // the blocks and, beside them, first the slots and lists of the approximations, then the lists of the product
    b.lists = cover_lists(b.blocks, n);
    const uint64_t nb = b.blocks.size(), nc = b.cand.size();
    const uint64_t temps = 8ull * (uint64_t)slot_elems + nc * (sizeof(HmBlockDev) + 20);
    const uint64_t keeps = item_bytes + sizeof(HmTile) * b.lists.tiles.size() + 4ull * b.lists.cover.size();
    const uint64_t peak = 8ull * (uint64_t)worst + (sizeof(HmBlockDev) + 8) * nb + 4ull * n + std::max(temps, keeps);
    if (peak > budget_left)
      return set_error(RFCMP_ERR_OUT_OF_BUDGET, "compression needs up to " + std::to_string(peak) +
                                                    " bytes, budget has " + std::to_string(budget_left));
  }
  HM_CUDA(dev_malloc(&out.perm, std::max<size_t>(4 * (size_t)n, 4)));
  owned.push_back(out.perm);
  if (n > 0) HM_CUDA(cudaMemcpy(out.perm, b.perm.data(), 4 * (size_t)n, cudaMemcpyHostToDevice));
  if (b.cand.empty()) return RFCMP_OK;
  auto is_small = [&](const HmBlockDev& c) { return std::max(c.r1 - c.r0, c.c1 - c.c0) <= ACA_SMALL; };
  order.reserve(b.cand.size());
  for (size_t c = 0; c < b.cand.size(); ++c)
    if (!is_small(b.cand[c])) order.push_back((int32_t)c);
  const int large = (int)order.size(), small = (int)b.cand.size() - large, per = HM_THREADS / 32;
  for (size_t c = 0; c < b.cand.size(); ++c)
    if (is_small(b.cand[c])) order.push_back((int32_t)c);
  HmBlockDev* cand_d = nullptr;
  long long* slot_d = nullptr;
  int32_t* order_d = nullptr;
  HM_CUDA(b.tmp.alloc(&cand_d, b.cand.size() * sizeof(HmBlockDev)));
  HM_CUDA(b.tmp.alloc(&slot_d, b.slot.size() * sizeof(long long)));
  HM_CUDA(b.tmp.alloc(&order_d, 4 * order.size()));
  HM_CUDA(b.tmp.alloc(&b.slots, 8 * (size_t)slot_elems));
  HM_CUDA(b.tmp.alloc(&b.rank_d, 4 * b.cand.size()));
  HM_CUDA(b.tmp.alloc(&b.status_d, 4 * b.cand.size()));
  HM_CUDA(cudaMemcpy(cand_d, b.cand.data(), b.cand.size() * sizeof(HmBlockDev), cudaMemcpyHostToDevice));
  HM_CUDA(cudaMemcpy(slot_d, b.slot.data(), b.slot.size() * sizeof(long long), cudaMemcpyHostToDevice));
  HM_CUDA(cudaMemcpy(order_d, order.data(), 4 * order.size(), cudaMemcpyHostToDevice));
  const int iter_cap = std::min(cap + 16, HM_MAX_ITER);
  ProfScope prof("hm_aca", 8.0 * (double)slot_elems, 0.0, 0);
  if (large > 0)
    hm_aca_kernel<8><<<large, HM_THREADS>>>(A, ld, out.perm, cand_d, order_d, large, slot_d, cap, iter_cap,
                                            (float)o.eps, b.slots, b.rank_d, b.status_d);
  if (small > 0)
    hm_aca_kernel<1><<<(small + per - 1) / per, HM_THREADS>>>(A, ld, out.perm, cand_d, order_d + large, small, slot_d,
                                                              cap, iter_cap, (float)o.eps, b.slots, b.rank_d,
                                                              b.status_d);
  HM_CUDA(cudaGetLastError());
  return RFCMP_OK;
}

// Waits for the cross approximations and packs the final blocks: the admissible ones whose crosses met the
// stopping rule in low rank, the rest dense.  The slots and lists of the approximations end here, so that
// one matrix's are not held beside the other's, nor beside the product's lists.
int finish_part(const float2* A, int ld, int n, const rfcmp_hm_opts& o, PartBuild& b, HmPart& out,
                std::vector<void*>& owned) {
  const int cap = o.max_rank;
  if (b.lists.tiles.empty()) b.lists = cover_lists(b.blocks, n);  // while the crosses are found
  const CoverLists& lists = b.lists;
  std::vector<int32_t> rank(b.cand.size(), 0), status(b.cand.size(), 1);
  if (!b.cand.empty()) {
    HM_CUDA(cudaMemcpy(rank.data(), b.rank_d, 4 * b.cand.size(), cudaMemcpyDeviceToHost));
    HM_CUDA(cudaMemcpy(status.data(), b.status_d, 4 * b.cand.size(), cudaMemcpyDeviceToHost));
  }
  std::vector<HmBlockDev> fin;
  std::vector<long long> fin_slot;
  fin.reserve(b.blocks.size());
  fin_slot.reserve(b.blocks.size());
  long long off = 0;
  size_t ci = 0;
  for (const HmBlockHost& h : b.blocks) {
    const long long m = h.r1 - h.r0, nn = h.c1 - h.c0;
    HmBlockDev d{h.r0, h.r1, h.c0, h.c1, -1, 0, off};
    long long s = 0;
    if (h.admissible) {
      const size_t c = ci++;
      if (status[c] != 0 || rank[c] < 0 || rank[c] > cap) {
        ++out.n_capped;
      } else if ((long long)rank[c] * (m + nn) >= m * nn) {
        ++out.n_small;  // the crosses would take at least the block's own entries
      } else {
        d.rank = rank[c];
        d.t0 = out.ncross;
        out.ncross += 2 * d.rank;
        s = b.slot[c];
        ++out.n_lowrank;
        out.max_rank = std::max(out.max_rank, rank[c]);
      }
    }
    if (d.rank < 0) ++out.n_dense;
    off += d.rank < 0 ? m * nn : (long long)d.rank * (m + nn);
    fin.push_back(d);
    fin_slot.push_back(s);
  }
  out.elems = off;
  out.nblocks = (int)fin.size();
  HM_CUDA(dev_malloc(&out.data, std::max<size_t>(8 * (size_t)off, 8)));
  owned.push_back(out.data);
  if (!fin.empty()) {
    const size_t nb = fin.size(), at = nb * sizeof(HmBlockDev);
    std::vector<char> buf(at + 8 * nb);  // the blocks, then their slots
    std::memcpy(buf.data(), fin.data(), at);
    std::memcpy(buf.data() + at, fin_slot.data(), 8 * nb);
    char* d = nullptr;
    HM_CUDA(dev_malloc(&d, buf.size()));
    owned.push_back(d);
    HM_CUDA(cudaMemcpy(d, buf.data(), buf.size(), cudaMemcpyHostToDevice));
    out.blocks = reinterpret_cast<HmBlockDev*>(d);
    hm_pack_kernel<<<(unsigned)nb, HM_THREADS>>>(A, ld, out.perm, out.blocks, reinterpret_cast<long long*>(d + at), cap,
                                                 b.slots, out.data);
    HM_CUDA(cudaGetLastError());
  }
  const std::vector<int2> items = cross_items(fin);
  b.tmp.clear();
  HM_CUDA(cudaStreamSynchronize(0));  // packed, and the pool has the temporaries back
  out.nitems = (int)items.size();
  out.ntiles = (int)lists.tiles.size();
  for (const HmTile& t : lists.tiles) out.entries = std::max(out.entries, t.end - t.begin);
  // the product's lists in one buffer (an upload each took as long as the rest of a small body's compression)
  const size_t at_tiles = sizeof(int2) * items.size(), at_cover = at_tiles + sizeof(HmTile) * lists.tiles.size();
  std::vector<char> buf(at_cover + 4 * lists.cover.size());
  if (!buf.empty()) {
    if (!items.empty()) std::memcpy(buf.data(), items.data(), at_tiles);
    std::memcpy(buf.data() + at_tiles, lists.tiles.data(), at_cover - at_tiles);
    std::memcpy(buf.data() + at_cover, lists.cover.data(), buf.size() - at_cover);
    char* d = nullptr;
    HM_CUDA(dev_malloc(&d, buf.size()));
    owned.push_back(d);
    HM_CUDA(cudaMemcpy(d, buf.data(), buf.size(), cudaMemcpyHostToDevice));
    out.items = reinterpret_cast<int2*>(d);
    out.tiles = reinterpret_cast<HmTile*>(d + at_tiles);
    out.cover = reinterpret_cast<int32_t*>(d + at_cover);
  }
  out.bytes = 8ull * (uint64_t)off + (sizeof(HmBlockDev) + 8) * fin.size() + 4ull * n + sizeof(int2) * items.size() +
              sizeof(HmTile) * lists.tiles.size() + 4ull * lists.cover.size();
  return RFCMP_OK;
}

}  // namespace rfcmp

// ============================================================================ C ABI
struct rfcmp_hm {
  int device = 0;
  rfcmp::HmPart part[2];  // RFCMP_HM_T_A, RFCMP_HM_V
  std::vector<void*> owned;
  std::atomic<uint64_t>* ctx_bytes = nullptr;
  std::atomic<int>* ctx_live = nullptr;
  uint64_t bytes = 0;
  rfcmp_hm_opts opts{};
  std::mutex mu;                          // guards nb_streams
  std::vector<cudaStream_t> nb_streams;   // non-blocking streams products were queued on
  ~rfcmp_hm() {
    for (void* p : owned) rfcmp::dev_free(p);
  }
};

using namespace rfcmp;

namespace {

// supports of the cells (centroid; box of the three vertices) and of the RWG functions (edge
// midpoint; box of the vertices of both cells)
void supports(const Topology& top, const double* verts, std::vector<double>& ccen, std::vector<double>& clo,
              std::vector<double>& chi, std::vector<double>& ecen, std::vector<double>& elo, std::vector<double>& ehi) {
  const int64_t nc = top.nc, ne = top.ne;
  ccen.assign(3 * nc, 0.0);
  clo.assign(3 * nc, 0.0);
  chi.assign(3 * nc, 0.0);
  for (int64_t c = 0; c < nc; ++c) {
    const double* p0 = verts + 3 * (int64_t)top.tris[3 * c];
    const double* p1 = verts + 3 * (int64_t)top.tris[3 * c + 1];
    const double* p2 = verts + 3 * (int64_t)top.tris[3 * c + 2];
    for (int d = 0; d < 3; ++d) {
      ccen[3 * c + d] = (p0[d] + p1[d] + p2[d]) / 3.0;
      clo[3 * c + d] = std::min(std::min(p0[d], p1[d]), p2[d]);
      chi[3 * c + d] = std::max(std::max(p0[d], p1[d]), p2[d]);
    }
  }
  ecen.assign(3 * ne, 0.0);
  elo.assign(3 * ne, 0.0);
  ehi.assign(3 * ne, 0.0);
  for (int64_t e = 0; e < ne; ++e) {
    const double* a = verts + 3 * (int64_t)top.edge_verts[2 * e];
    const double* b = verts + 3 * (int64_t)top.edge_verts[2 * e + 1];
    const int64_t cp = top.edge_cells[2 * e], cm = top.edge_cells[2 * e + 1];
    for (int d = 0; d < 3; ++d) {
      ecen[3 * e + d] = 0.5 * (a[d] + b[d]);
      elo[3 * e + d] = std::min(clo[3 * cp + d], clo[3 * cm + d]);
      ehi[3 * e + d] = std::max(chi[3 * cp + d], chi[3 * cm + d]);
    }
  }
}

int check_opts(const rfcmp_hm_opts& o) {
  for (int i = 0; i < 6; ++i)
    if (o.reserved[i] != 0) return set_error(RFCMP_ERR_INVALID_ARG, "opts.reserved must be zero");
  if (!(o.eps > 0.0 && o.eps < 1.0)) return set_error(RFCMP_ERR_INVALID_ARG, "eps must be in (0, 1)");
  if (!(o.eta > 0.0) || !std::isfinite(o.eta)) return set_error(RFCMP_ERR_INVALID_ARG, "eta must be positive");
  if (o.leaf < 8 || o.leaf > 1024) return set_error(RFCMP_ERR_INVALID_ARG, "leaf must be in [8, 1024]");
  if (o.max_rank < 1 || o.max_rank > HM_MAX_RANK) return set_error(RFCMP_ERR_INVALID_ARG, "max_rank must be in [1, 256]");
  return RFCMP_OK;
}

}  // namespace

extern "C" {

void rfcmp_hm_opts_default(rfcmp_hm_opts* o) {
  if (!o) return;
  std::memset(o, 0, sizeof(*o));
  o->eps = 1e-4;
  o->eta = 1.0;
  o->leaf = 32;
  o->max_rank = 64;
}

int rfcmp_hm_partition(const double* centres, const double* sup_lo, const double* sup_hi, int64_t n, int32_t leaf,
                       double eta, int32_t* perm, int32_t* blocks, int64_t capacity, int64_t* n_blocks) {
  if (!n_blocks || !perm || (n > 0 && (!centres || !sup_lo || !sup_hi)))
    return set_error(RFCMP_ERR_INVALID_ARG, "NULL argument");
  int rc = check_partition_args(n, leaf, eta);
  if (rc != RFCMP_OK) return rc;
  for (int64_t i = 0; i < 3 * n; ++i)
    if (!std::isfinite(centres[i]) || !std::isfinite(sup_lo[i]) || !std::isfinite(sup_hi[i]))
      return set_error(RFCMP_ERR_INVALID_ARG, "non-finite coordinate");
  std::vector<int32_t> p;
  std::vector<HmBlockHost> b;
  partition(centres, sup_lo, sup_hi, (int)n, leaf, eta, p, b);
  *n_blocks = (int64_t)b.size();
  if (n > 0) std::memcpy(perm, p.data(), 4 * (size_t)n);
  if (!blocks) return RFCMP_OK;
  if (capacity < (int64_t)b.size()) return set_error(RFCMP_ERR_INVALID_ARG, "blocks capacity too small");
  for (size_t i = 0; i < b.size(); ++i) {
    blocks[5 * i] = b[i].r0;
    blocks[5 * i + 1] = b[i].r1;
    blocks[5 * i + 2] = b[i].c0;
    blocks[5 * i + 3] = b[i].c1;
    blocks[5 * i + 4] = b[i].admissible;
  }
  return RFCMP_OK;
}

int rfcmp_hm_create(rfcmp_op* op, const rfcmp_hm_opts* opts_in, rfcmp_hm** out) {
  if (!op || !out) return set_error(RFCMP_ERR_INVALID_ARG, "NULL argument");
  *out = nullptr;
  rfcmp_hm_opts o;
  rfcmp_hm_opts_default(&o);
  if (opts_in) o = *opts_in;
  int rc = check_opts(o);
  if (rc != RFCMP_OK) return rc;
  OpDenseView v;
  if (!op_dense_view(op, &v)) return set_error(RFCMP_ERR_INVALID_ARG, "op has no resident T_A and V");
  HM_CUDA(cudaSetDevice(v.device));
  auto hm = std::make_unique<rfcmp_hm>();
  hm->device = v.device;
  hm->opts = o;
  try {
    std::vector<double> ccen, clo, chi, ecen, elo, ehi;
    supports(*v.top, v.verts, ccen, clo, chi, ecen, elo, ehi);
    const float2* mats[2] = {v.TA, v.V};
    const int lds[2] = {v.ldN, v.ldC}, ns[2] = {v.n, v.nc};
    PartBuild part[2];
    // the host partitions V beside T_A (a thread of its own, or after it where none can be had or V's partition takes
    // no longer than to start one); the builds follow one another, so that the peak is one matrix's slots
    auto split_v = [&] { partition(ccen.data(), clo.data(), chi.data(), v.nc, o.leaf, o.eta, part[1].perm, part[1].blocks); };
    std::future<void> other;
    try {
      if (v.nc >= 12 * o.leaf) other = std::async(std::launch::async, split_v);
    } catch (const std::system_error&) {
    }
    partition(ecen.data(), elo.data(), ehi.data(), v.n, o.leaf, o.eta, part[0].perm, part[0].blocks);
    for (int w = 0; w < 2 && rc == RFCMP_OK; ++w) {
      uint64_t left = UINT64_MAX;
      if (v.budget) {
        const uint64_t used = v.ctx_bytes->load() + hm->bytes;
        left = v.budget > used ? v.budget - used : 0;
      }
      if (w == 1) {
        if (other.valid()) other.get();
        else split_v();
      }
      rc = start_part(mats[w], lds[w], ns[w], o, left, part[w], hm->part[w], hm->owned);
      if (rc == RFCMP_OK) rc = finish_part(mats[w], lds[w], ns[w], o, part[w], hm->part[w], hm->owned);
      hm->bytes += hm->part[w].bytes;
    }
  } catch (const std::bad_alloc&) {
    return set_error(RFCMP_ERR_CUDA, "out of host memory");
  }
  if (rc != RFCMP_OK) return rc;
  hm->ctx_bytes = v.ctx_bytes;
  hm->ctx_live = v.ctx_live;
  *hm->ctx_bytes += hm->bytes;
  ++*hm->ctx_live;
  *out = hm.release();
  return RFCMP_OK;
}

int rfcmp_hm_apply(rfcmp_hm* hm, int which, const rfcmp_c128* x, rfcmp_c128* y, int64_t nrhs, void* stream) {
  if (!hm || !x || !y || nrhs < 1 || nrhs > 65535 || (which != RFCMP_HM_T_A && which != RFCMP_HM_V))
    return set_error(RFCMP_ERR_INVALID_ARG, "invalid argument");
  if ((const void*)x == (const void*)y) return set_error(RFCMP_ERR_INVALID_ARG, "x and y must not alias");
  const HmPart& P = hm->part[which];
  HM_CUDA(cudaSetDevice(hm->device));
  cudaStream_t st = (cudaStream_t)stream;
  if (st) {
    unsigned int flags = 0;
    HM_CUDA(cudaStreamGetFlags(st, &flags));
    if (flags & cudaStreamNonBlocking) {
      std::lock_guard<std::mutex> lk(hm->mu);
      if (std::find(hm->nb_streams.begin(), hm->nb_streams.end(), st) == hm->nb_streams.end())
        hm->nb_streams.push_back(st);
    }
  }
  if (P.n == 0) return RFCMP_OK;
  // scratch: x in cluster order and the cross sums, at most HM_SCRATCH bytes of sums at a time
  const size_t per_col = 16 * (size_t)std::max(P.ncross, 1);
  const int64_t most = std::max<int64_t>(HM_COLS, (int64_t)(HM_SCRATCH / per_col) / HM_COLS * HM_COLS);
  const int64_t width = std::min<int64_t>(nrhs, most);
  double2* xp = nullptr;
  HM_CUDA(cudaMallocAsync(&xp, (16 * (size_t)P.n + per_col) * (size_t)width, st));
  double2* t = xp + (size_t)P.n * width;
  cudaError_t launched = cudaSuccess;
  for (int64_t c = 0; c < nrhs; c += width) {
    const int nr = (int)std::min<int64_t>(width, nrhs - c);
    const long long total = (long long)P.n * nr;
    const unsigned groups = (unsigned)((nr + HM_COLS - 1) / HM_COLS);
    const int grid = (int)std::min<long long>((total + HM_THREADS - 1) / HM_THREADS, 152 * 8);
    hm_gather_kernel<<<grid, HM_THREADS, 0, st>>>(reinterpret_cast<const double2*>(x) + (size_t)c * P.n, P.perm, P.n,
                                                  nr, xp);
    ProfScope prof("hm_apply", 8.0 * (double)P.elems + 32.0 * (double)total, 16.0 * (double)P.elems * nr, st);
    if (P.nitems > 0) {
      const int per = HM_CROSS_THREADS / 32;
      hm_cross_kernel<<<dim3((P.nitems + per - 1) / per, groups), HM_CROSS_THREADS, 0, st>>>(
          P.blocks, P.items, P.nitems, P.data, xp, t, P.n, nr);
    }
    const int team = hm_team((long long)P.ntiles * groups, P.entries);
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = (unsigned)team;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(P.ntiles * team), groups);
    cfg.blockDim = dim3(HM_THREADS);
    cfg.stream = st;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    launched = cudaLaunchKernelEx(&cfg, hm_rows_kernel, (const HmTile*)P.tiles, (const int32_t*)P.cover,
                                  (const HmBlockDev*)P.blocks, (const float2*)P.data, (const double2*)xp,
                                  (const double2*)t, (const int32_t*)P.perm,
                                  reinterpret_cast<double2*>(y) + (size_t)c * P.n, P.n, nr);
    if (launched != cudaSuccess) break;
  }
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = launched;
  cudaFreeAsync(xp, st);
  if (e != cudaSuccess) return set_error(RFCMP_ERR_CUDA, std::string("rfcmp_hm_apply: ") + cudaGetErrorString(e));
  return RFCMP_OK;
}

int rfcmp_hm_info_get(const rfcmp_hm* hm, rfcmp_hm_info* out) {
  if (!hm || !out) return set_error(RFCMP_ERR_INVALID_ARG, "NULL argument");
  std::memset(out, 0, sizeof(*out));
  for (int w = 0; w < 2; ++w) {
    const HmPart& P = hm->part[w];
    out->n[w] = P.n;
    out->lowrank_blocks[w] = P.n_lowrank;
    out->dense_blocks[w] = P.n_dense;
    out->capped_blocks[w] = P.n_capped;
    out->small_blocks[w] = P.n_small;
    out->bytes[w] = P.bytes;
    out->max_rank[w] = P.max_rank;
  }
  return RFCMP_OK;
}

int rfcmp_hm_destroy(rfcmp_hm* hm) {
  if (!hm) return RFCMP_OK;
  cudaSetDevice(hm->device);
  // frees are queued on the legacy stream: make it wait for the streams products ran on
  if (!hm->nb_streams.empty()) {
    cudaEvent_t ev = nullptr;
    if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) == cudaSuccess) {
      for (cudaStream_t s : hm->nb_streams)
        if (cudaEventRecord(ev, s) == cudaSuccess) cudaStreamWaitEvent(0, ev, 0);
      cudaEventDestroy(ev);
    } else {
      for (cudaStream_t s : hm->nb_streams) cudaStreamSynchronize(s);
    }
  }
  if (hm->ctx_bytes) *hm->ctx_bytes -= hm->bytes;
  if (hm->ctx_live) --*hm->ctx_live;
  delete hm;
  return RFCMP_OK;
}

}  // extern "C"
