// Device packer: Alg. 1 (Sec. 4.1) applied to every row panel of A.
//
// Alg. 1 walks a tile column by column and, within a column, row by row,
// appending each nonzero to A_p / loc_m and, for a non-empty column, its
// index to col_ind and its count to nnz.  On the GPU the per-(panel, column)
// counts are independent, so the walk becomes count / scan / scatter:
//   count   one thread per (panel, column): nonzeros of that panel column
//   scan    exclusive prefix sums of (count, count != 0) in panel-major,
//           column-ascending order = Alg. 1's append order
//   scatter one thread per (panel, column): writes its column record and
//           its values/rows (rows ascending) at the scanned offsets
// The execution layouts of the SpMM (row stream, touched-row gather, dense
// BF16 tile copies) are built the same way, and the independent passes share
// launches: phase 1 is one counting launch and one three-array scan, phase 2
// one writing launch, with one host round trip between them (pack_typed).
// Threads of a warp own consecutive columns (or, for row passes, one warp owns
// a row), so every read of A is a coalesced row segment.
#include <algorithm>
#include <cstring>
#include <new>
#include <type_traits>
#include <vector>

#include "handle.hpp"

namespace rosko {
namespace {

constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;
constexpr int kScanTile = kScanThreads * kScanItems;

// ----------------------------------------------------------------------------
// Value test and conversion per (source, packed) type pair.
template <class S, class D> struct Conv;
template <> struct Conv<float, float> {
  __device__ static bool get(float a, float, float& out) { out = a; return a != 0.0f; }
};
template <> struct Conv<float, __nv_bfloat16> {
  // The mask is taken from the FP32 value; a value that rounds to 0 stays packed.
  __device__ static bool get(float a, float, __nv_bfloat16& out) {
    out = __float2bfloat16_rn(a);
    return a != 0.0f;
  }
};
template <> struct Conv<float, double> {
  __device__ static bool get(float a, float, double& out) { out = (double)a; return a != 0.0f; }
};
template <> struct Conv<float, int8_t> {
  // Symmetric per-row code q = clamp(rint(a / s), -127, 127); the mask is q != 0.
  __device__ static bool get(float a, float s, int8_t& out) {
    float q = rintf(__fdiv_rn(a, s));
    q = fminf(fmaxf(q, -127.0f), 127.0f);
    out = (int8_t)(int)q;
    return out != 0;
  }
};
template <> struct Conv<__nv_bfloat16, __nv_bfloat16> {
  __device__ static bool get(__nv_bfloat16 a, float, __nv_bfloat16& out) {
    out = a;
    return __bfloat162float(a) != 0.0f;
  }
};
template <> struct Conv<int8_t, int8_t> {
  __device__ static bool get(int8_t a, float, int8_t& out) { out = a; return a != 0; }
};

// One nonzero record (value + panel-relative row), see handle.hpp.
__device__ __forceinline__ void put_rec(void* nz, int64_t e, float v, int r) {
  reinterpret_cast<uint2*>(nz)[e] = make_uint2((uint32_t)r, __float_as_uint(v));
}
__device__ __forceinline__ void put_rec(void* nz, int64_t e, __nv_bfloat16 v, int r) {
  reinterpret_cast<uint32_t*>(nz)[e] = ((uint32_t)__bfloat16_as_ushort(v) << 16) | (uint32_t)r;
}
__device__ __forceinline__ void put_rec(void* nz, int64_t e, int8_t v, int r) {
  reinterpret_cast<uint32_t*>(nz)[e] = ((uint32_t)(uint8_t)v << 16) | (uint32_t)r;
}
__device__ __forceinline__ void put_rec(void* nz, int64_t e, double v, int r) {
  RecF64 w;
  w.a = v;
  w.r = r;
  w.pad = 0;
  reinterpret_cast<RecF64*>(nz)[e] = w;
}
__device__ __forceinline__ float get_val(const void* nz, int64_t e, float) {
  return __uint_as_float(reinterpret_cast<const uint2*>(nz)[e].y);
}
__device__ __forceinline__ __nv_bfloat16 get_val(const void* nz, int64_t e, __nv_bfloat16) {
  return __ushort_as_bfloat16((unsigned short)(reinterpret_cast<const uint32_t*>(nz)[e] >> 16));
}
__device__ __forceinline__ int8_t get_val(const void* nz, int64_t e, int8_t) {
  return (int8_t)(uint8_t)(reinterpret_cast<const uint32_t*>(nz)[e] >> 16);
}
__device__ __forceinline__ double get_val(const void* nz, int64_t e, double) {
  return reinterpret_cast<const RecF64*>(nz)[e].a;
}
__device__ __forceinline__ int get_row(const void* nz, int64_t e, float) {
  return (int)reinterpret_cast<const uint2*>(nz)[e].x;
}
template <class D>
__device__ __forceinline__ int get_row(const void* nz, int64_t e, D) {
  return (int)(reinterpret_cast<const uint32_t*>(nz)[e] & 0xFFFFu);
}
__device__ __forceinline__ int get_row(const void* nz, int64_t e, double) {
  return reinterpret_cast<const RecF64*>(nz)[e].r;
}

// Per-row symmetric INT8 scale s_i = max_k |a_ik| / 127 (1 for an all-zero row).
__global__ void rowscale_kernel(const float* __restrict__ A, int64_t M, int64_t K, int64_t lda,
                                float* __restrict__ scale) {
  const int64_t row = (int64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (row >= M) return;
  float m = 0.0f;
  for (int64_t k = lane; k < K; k += 32) m = fmaxf(m, fabsf(A[row * lda + k]));
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) scale[row] = (m == 0.0f) ? 1.0f : __fdiv_rn(m, 127.0f);
}

__device__ __forceinline__ int2 add2(int2 a, int2 b) { return make_int2(a.x + b.x, a.y + b.y); }

__device__ __forceinline__ int2 warp_incl_scan(int2 v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int2 t;
    t.x = __shfl_up_sync(0xffffffffu, v.x, o);
    t.y = __shfl_up_sync(0xffffffffu, v.y, o);
    if (lane >= o) v = add2(v, t);
  }
  return v;
}

// Exclusive block scan of one int2 per thread; returns the block total in *total.
__device__ int2 block_excl_scan(int2 v, int2* total) {
  __shared__ int2 warp_sums[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int2 inc = warp_incl_scan(v);
  if (lane == 31) warp_sums[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    int2 w = (lane < (int)(blockDim.x >> 5)) ? warp_sums[lane] : make_int2(0, 0);
    w = warp_incl_scan(w);
    warp_sums[lane] = w;
  }
  __syncthreads();
  int2 base = warp ? warp_sums[warp - 1] : make_int2(0, 0);
  *total = warp_sums[(blockDim.x >> 5) - 1];
  __syncthreads();
  return make_int2(base.x + inc.x - v.x, base.y + inc.y - v.y);
}

// Up to three independent exclusive scans of int2 arrays in place, sharing
// each of the three launches of a tiled scan: job i owns blocks
// [first[i], first[i+1]) of the tile passes and block i of the spine pass.
// data[n] receives the total; sums holds nb + 1 entries (nb = tiles of job).
struct ScanJob {
  int2* data;
  int64_t n;
  int2* sums;
  int64_t nb;
};
struct ScanSet {
  ScanJob job[3];
  int64_t first[4];
  int count;
};

__device__ __forceinline__ int scan_job_of(const ScanSet& s, int64_t b) {
  int i = 0;
  while (i + 1 < s.count && b >= s.first[i + 1]) ++i;
  return i;
}

// Tile pass A: per-tile sums.
__global__ void scan_reduce_kernel(ScanSet s) {
  pdl_wait();
  pdl_trigger();
  const int j = scan_job_of(s, blockIdx.x);
  const ScanJob J = s.job[j];
  const int64_t base = ((int64_t)blockIdx.x - s.first[j]) * kScanTile;
  int2 v = make_int2(0, 0);
  for (int i = 0; i < kScanItems; ++i) {
    const int64_t idx = base + (int64_t)i * kScanThreads + threadIdx.x;
    if (idx < J.n) v = add2(v, J.data[idx]);
  }
  int2 total;
  block_excl_scan(v, &total);
  if (threadIdx.x == 0) J.sums[blockIdx.x - s.first[j]] = total;
}

// Spine pass B: exclusive scan of one job's tile sums (chunked), total to
// sums[nb].
__global__ void scan_spine_kernel(ScanSet s) {
  pdl_wait();
  pdl_trigger();
  const ScanJob J = s.job[blockIdx.x];
  int2 carry = make_int2(0, 0);
  for (int64_t c0 = 0; c0 < J.nb; c0 += kScanThreads) {
    const int64_t idx = c0 + threadIdx.x;
    int2 v = idx < J.nb ? J.sums[idx] : make_int2(0, 0);
    int2 total;
    int2 ex = block_excl_scan(v, &total);
    if (idx < J.nb) J.sums[idx] = add2(ex, carry);
    carry = add2(carry, total);
    __syncthreads();
  }
  if (threadIdx.x == 0) J.sums[J.nb] = carry;
}

// Tile pass C: in-place exclusive scan of each tile with its offset.
__global__ void scan_down_kernel(ScanSet s) {
  pdl_wait();
  pdl_trigger();
  const int j = scan_job_of(s, blockIdx.x);
  const ScanJob J = s.job[j];
  const int64_t tile = (int64_t)blockIdx.x - s.first[j];
  const int64_t base = tile * kScanTile + (int64_t)threadIdx.x * kScanItems;
  int2 v[kScanItems];
  int2 sum = make_int2(0, 0);
  for (int i = 0; i < kScanItems; ++i) {
    v[i] = (base + i < J.n) ? J.data[base + i] : make_int2(0, 0);
    sum = add2(sum, v[i]);
  }
  int2 total;
  int2 off = add2(block_excl_scan(sum, &total), J.sums[tile]);
  for (int i = 0; i < kScanItems; ++i) {
    if (base + i < J.n) J.data[base + i] = off;
    off = add2(off, v[i]);
  }
  if (tile == 0 && threadIdx.x == 0) J.data[J.n] = J.sums[J.nb];
}

// Dense BF16 copies of 128-row tiles for the tensor-core dense-panel path:
// row block c holds rows tile_order[c]*128 .. +127 of A (zero past M and past
// K; row stride Kpad), converted exactly as the packer converts them.
__device__ __forceinline__ __nv_bfloat16 to_bf16(__nv_bfloat16 a) { return a; }
// INT8 codes are integers of magnitude <= 127: exact in BF16
__device__ __forceinline__ __nv_bfloat16 to_bf16(int8_t a) { return __float2bfloat16_rn((float)a); }

// Row-slot stream records (value + column k) and the per-row sentinel.
__device__ __forceinline__ void put_row_rec(void* rnz, int64_t e, float v, int k) {
  reinterpret_cast<uint2*>(rnz)[e] = make_uint2((uint32_t)k, __float_as_uint(v));
}
__device__ __forceinline__ void put_row_rec(void* rnz, int64_t e, __nv_bfloat16 v, int k) {
  reinterpret_cast<uint32_t*>(rnz)[e] = ((uint32_t)__bfloat16_as_ushort(v) << 16) | (uint32_t)k;
}
__device__ __forceinline__ void put_row_rec(void* rnz, int64_t e, int8_t v, int k) {
  reinterpret_cast<uint32_t*>(rnz)[e] = ((uint32_t)(uint8_t)v << 16) | (uint32_t)k;
}
__device__ __forceinline__ void put_row_rec(void* rnz, int64_t e, double v, int k) {
  RecF64 w;
  w.a = v;
  w.r = k;
  w.pad = 0;
  reinterpret_cast<RecF64*>(rnz)[e] = w;
}
template <class D>
__device__ __forceinline__ void put_row_sentinel(void* rnz, int64_t e) {
  if constexpr (sizeof(D) <= 2) {
    reinterpret_cast<uint32_t*>(rnz)[e] = 0xFFFFu;
  } else if constexpr (sizeof(D) == 4) {
    reinterpret_cast<uint2*>(rnz)[e] = make_uint2(0x7FFFFFFFu, 0u);
  } else {
    RecF64 w;
    w.a = 0.0;
    w.r = 0x7FFFFFFF;
    w.pad = 0;
    reinterpret_cast<RecF64*>(rnz)[e] = w;
  }
}

// ----------------------------------------------------------------------------
// The passes of one phase share a launch: a 1-D grid of 256-thread blocks in
// consecutive ranges, one range per pass (a block runs exactly one pass).
constexpr int kPackThreads = 256;
constexpr int kRowsPerBlock = kPackThreads / 32;   // row passes: one warp per row
constexpr int kRowBatch = 16;   // column passes: rows of a column in flight together

struct PackGeom {
  int64_t M, K, lda, P, T;
  int m_r;
  int64_t gx;   // 256-column groups, ceil(K / 256)
};

// Counting pass, Alg. 1's per-column nnz: cnt[p*K + k] = (nonzeros of column
// k in panel p, 1 if non-empty); a column's first nonzero seen anywhere
// counts it as touched.  The same visit of the panel yields the other two
// counts: the nonzeros of each row (a ballot per row across the warp, summed
// over the block in shared memory, one atomic add per row and block into
// rcnt, which starts at 0; the block of columns 0..255 adds the row's
// sentinel) and, for the gather stream, flag[t*K + k].x = 1 when column k of
// 128-row tile t is non-empty (flag starts at 0).
template <class S, class D>
__device__ void col_count(const S* __restrict__ A, const PackGeom& g,
                          const float* __restrict__ scale, int64_t b, int2* __restrict__ cnt,
                          int* __restrict__ touched, int* __restrict__ touched_total,
                          int2* __restrict__ rcnt, int2* __restrict__ flag) {
  __shared__ int row_sum[32];   // m_r <= 32
  const int64_t bx = b % g.gx;
  const int64_t k = bx * kPackThreads + threadIdx.x;
  const int64_t p = b / g.gx;
  const bool in = k < g.K;
  const int lane = threadIdx.x & 31;
  const int64_t m0 = p * g.m_r, m1 = min(g.M, m0 + g.m_r);
  if (rcnt) {
    if (threadIdx.x < 32) row_sum[threadIdx.x] = 0;
    __syncthreads();
  }
  int c = 0;
  // bounds are uniform across the block: every lane takes every ballot.  A
  // panel's loads are issued sixteen rows at a time, before any is tested.
  for (int64_t mb = m0; mb < m1; mb += kRowBatch) {
    S a[kRowBatch];
#pragma unroll
    for (int i = 0; i < kRowBatch; ++i)
      a[i] = in && mb + i < m1 ? A[(mb + i) * g.lda + k] : S(0);
#pragma unroll
    for (int i = 0; i < kRowBatch; ++i) {
      if (mb + i >= m1) break;
      D v;
      const bool nz = in && Conv<S, D>::get(a[i], scale ? scale[mb + i] : 1.0f, v);
      c += nz ? 1 : 0;
      if (rcnt) {
        const unsigned mask = __ballot_sync(0xffffffffu, nz);
        if (lane == 0 && mask) atomicAdd(&row_sum[mb + i - m0], __popc(mask));
      }
    }
  }
  if (rcnt) {
    __syncthreads();
    const int64_t r = m0 + threadIdx.x;
    if (threadIdx.x < 32 && r < m1) {
      const int add = row_sum[threadIdx.x] + (bx == 0 ? 1 : 0);
      if (add) atomicAdd(&rcnt[r].x, add);
    }
  }
  if (!in) return;
  cnt[p * g.K + k] = make_int2(c, c != 0);
  if (c && atomicExch(&touched[k], 1) == 0) atomicAdd(touched_total, 1);
  if (c && flag) flag[(m0 / kDenseTileRows) * g.K + k] = make_int2(1, 0);
}

// Counting pass of the row-slot stream: rcnt[row] = (nonzeros of the row + 1
// sentinel, 0); lanes over consecutive columns (coalesced).
template <class S, class D>
__device__ void row_count(const S* __restrict__ A, const PackGeom& g,
                          const float* __restrict__ scale, int64_t b, int2* __restrict__ rcnt) {
  const int64_t row = b * kRowsPerBlock + threadIdx.x / 32;
  const int lane = threadIdx.x & 31;
  if (row >= g.M) return;
  const float sc = scale ? scale[row] : 1.0f;
  int c = 0;
#pragma unroll 8
  for (int64_t k = lane; k < g.K; k += 32) {
    D v;
    c += Conv<S, D>::get(A[row * g.lda + k], sc, v) ? 1 : 0;
  }
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if (lane == 0) rcnt[row] = make_int2(c + 1, 0);
}

// Phase 1 in one launch: blocks [0, b_col) count panel columns (and rows and
// tile columns, see col_count); with K = 0 there are no column blocks and
// the remaining blocks give each row its sentinel count instead.
template <class S, class D>
__global__ void __launch_bounds__(kPackThreads)
    pack_count_kernel(const S* __restrict__ A, PackGeom g, const float* __restrict__ scale,
                      int2* __restrict__ cnt, int* __restrict__ touched,
                      int* __restrict__ touched_total, int2* __restrict__ rcnt,
                      int2* __restrict__ flag, int64_t b_col) {
  pdl_wait();
  pdl_trigger();
  const int64_t b = blockIdx.x;
  if (b < b_col) {
    col_count<S, D>(A, g, scale, b, cnt, touched, touched_total, rcnt, flag);
    return;
  }
  row_count<S, D>(A, g, scale, b - b_col, rcnt);
}

// Pointers and block ranges of the writing phase.  Scanned offsets:
// cnt[p*K+k] = (first nonzero, first packed column) of a panel column,
// rcnt[row].x = first record of a row, flag[t*K+k].x = slot of column k in
// tile t's union list (plus the tile's base).
struct WriteArgs {
  const int2* cnt;
  int2* colrec;
  void* nz;
  int32_t* panel_col;
  int64_t* panel_nnz;
  const int2* rcnt;
  int32_t* rowptr;
  void* rnz;
  const int2* flag;
  int32_t* gu_start;
  int32_t* gu_k;
  void* gnz;
  const int32_t* tile_order;
  __nv_bfloat16* dense_A;
  int64_t dense_rows, Kpad, gxd, ry;
  int64_t nnz, n_cols, gu_total;
  int zero_panels, a_vec, row_warps;
  int64_t b_scatter, b_row, b_union, b_dense;
};

// Alg. 1's append: each non-empty panel column writes its column record and
// its values with rows ascending at the scanned offsets.
template <class S, class D>
__device__ void scatter(const S* __restrict__ A, const PackGeom& g,
                        const float* __restrict__ scale, int64_t b, const WriteArgs& w) {
  const int64_t k = (b % g.gx) * kPackThreads + threadIdx.x;
  const int64_t p = b / g.gx;
  if (k >= g.K) return;
  const int64_t pk = p * g.K + k;
  const int2 o = w.cnt[pk];
  if (k == 0) {
    w.panel_col[p] = o.y;
    w.panel_nnz[p] = o.x;
  }
  const int cnt = w.cnt[pk + 1].x - o.x;
  if (cnt == 0) return;
  w.colrec[o.y] = make_int2((int32_t)k, o.x);
  const int64_t m0 = p * g.m_r, m1 = min(g.M, m0 + g.m_r);
  int64_t e = o.x;
  for (int64_t mb = m0; mb < m1; mb += kRowBatch) {
    S a[kRowBatch];
#pragma unroll
    for (int i = 0; i < kRowBatch; ++i) a[i] = mb + i < m1 ? A[(mb + i) * g.lda + k] : S(0);
#pragma unroll
    for (int i = 0; i < kRowBatch; ++i) {
      D v;
      if (mb + i < m1 && Conv<S, D>::get(a[i], scale ? scale[mb + i] : 1.0f, v)) {
        put_rec(w.nz, e, v, (int)(mb + i - m0));
        ++e;
      }
    }
  }
}

// Row-slot stream: each row's records (k ascending) at its scanned offset,
// then its sentinel; with the gather stream, the same record re-addressed by
// the slot of k in the tile's union list goes to the same position of gnz.
// W warps share a row (W = kRowsPerBlock: the whole block) and take turns of
// 256 columns each: a step's loads are issued together, the step after is
// fetched while this one is written, and a warp starts where the counts of
// the warps before it end.
template <class S, class D, int W>
__device__ void row_write(const S* __restrict__ A, const PackGeom& g,
                          const float* __restrict__ scale, int64_t b, const WriteArgs& w) {
  __shared__ int cnt[2][kRowsPerBlock];
  const int wid = threadIdx.x / 32, lane = threadIdx.x & 31;
  const int64_t row = W == 1 ? b * kRowsPerBlock + wid : b;
  if (row >= g.M) return;   // (uniform over a block that shares a row)
  const float sc = scale ? scale[row] : 1.0f;
  int64_t pos = w.rcnt[row].x;
  const bool first = lane == 0 && (W == 1 || wid == 0);
  if (first) w.rowptr[row] = (int32_t)pos;
  const int2* tf = w.flag ? w.flag + (row / kDenseTileRows) * g.K : nullptr;
  const int32_t base = tf ? tf[0].x : 0;
  constexpr int G = 8;
  const int64_t kw = W == 1 ? 0 : wid * 32 * G;
  S nx[G];
  auto fetch = [&](int64_t k0) {
#pragma unroll
    for (int u = 0; u < G; ++u) {
      const int64_t k = k0 + kw + u * 32 + lane;
      nx[u] = k < g.K ? A[row * g.lda + k] : S(0);
    }
  };
  fetch(0);
  int turn = 0;
  for (int64_t k0 = 0; k0 < g.K; k0 += 32 * G * W) {
    D v[G];
    unsigned mask[G];
    int total = 0;
#pragma unroll
    for (int u = 0; u < G; ++u) {
      const int64_t k = k0 + kw + u * 32 + lane;
      mask[u] = __ballot_sync(0xffffffffu, k < g.K && Conv<S, D>::get(nx[u], sc, v[u]));
      total += __popc(mask[u]);
    }
    fetch(k0 + 32 * G * W);
    int64_t q0 = pos;
    if constexpr (W > 1) {
      // (two sets of counts in turn: one barrier per step)
      if (lane == 0) cnt[turn][wid] = total;
      __syncthreads();
#pragma unroll
      for (int i = 0; i < W; ++i) {
        const int c = cnt[turn][i];
        if (i < wid) q0 += c;
        pos += c;
      }
      turn ^= 1;
    } else {
      pos += total;
    }
#pragma unroll
    for (int u = 0; u < G; ++u) {
      if (mask[u] >> lane & 1u) {
        const int64_t k = k0 + kw + u * 32 + lane;
        const int64_t q = q0 + __popc(mask[u] & ((1u << lane) - 1u));
        put_row_rec(w.rnz, q, v[u], (int)k);
        if (tf) put_row_rec(w.gnz, q, v[u], (int)(tf[k].x - base));
      }
      q0 += __popc(mask[u]);
    }
  }
  if (first) {
    put_row_sentinel<D>(w.rnz, pos);
    if (tf) put_row_sentinel<D>(w.gnz, pos);
  }
}

// Gather stream: the union list gu_k of each tile and its offset gu_start.
__device__ void tile_union(const PackGeom& g, int64_t b, const WriteArgs& w) {
  const int64_t k = (b % g.gx) * kPackThreads + threadIdx.x;
  const int64_t t = b / g.gx;
  if (k >= g.K) return;
  const int64_t i = t * g.K + k;
  if (k == 0) w.gu_start[t] = w.flag[i].x;
  if (w.flag[i + 1].x != w.flag[i].x) w.gu_k[w.flag[i].x] = (int32_t)k;
}

// The dense copy holds each entry converted exactly as the packer converts
// it (BF16 packs: the BF16 value; INT8 packs: the INT8 code, exact in BF16).
// A thread writes eight columns of a row (16 bytes; Kpad is a multiple of
// eight), read with 16-byte loads where A's rows are 16-byte aligned.
template <class S, class D>
__device__ void densify(const S* __restrict__ A, const PackGeom& g,
                        const float* __restrict__ scale, int64_t b, const WriteArgs& w) {
  const int64_t k = ((b % w.gxd) * kPackThreads + threadIdx.x) * 8;
  if (k >= w.Kpad) return;
  const bool vec = w.a_vec && k + 8 <= g.K;
  for (int64_t rr = b / w.gxd; rr < w.dense_rows; rr += w.ry) {
    const int64_t row = (int64_t)w.tile_order[rr / kDenseTileRows] * kDenseTileRows +
                        rr % kDenseTileRows;
    alignas(16) __nv_bfloat16 o[8];
    alignas(16) S a[8];
    const bool in = row < g.M;
    const S* src = A + row * g.lda + k;
    if (vec && in) {
      constexpr int W = (int)sizeof(S) * 8;   // 8, 16 or 32 bytes
      if constexpr (W == 8) {
        *reinterpret_cast<uint2*>(a) = __ldg(reinterpret_cast<const uint2*>(src));
      } else {
#pragma unroll
        for (int i = 0; i < W / 16; ++i)
          reinterpret_cast<uint4*>(a)[i] = __ldg(reinterpret_cast<const uint4*>(src) + i);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) a[i] = in && k + i < g.K ? src[i] : S(0);
    }
    const float sc = scale && in ? scale[row] : 1.0f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      D q;
      Conv<S, D>::get(a[i], sc, q);
      o[i] = in && k + i < g.K ? to_bf16(q) : __float2bfloat16_rn(0.0f);
    }
    *reinterpret_cast<uint4*>(w.dense_A + rr * w.Kpad + k) = *reinterpret_cast<const uint4*>(o);
  }
}

// Terminating entries: panel_col[P] = packed columns, panel_nnz[P] = nnz,
// colrec[n_cols] = colrec[n_cols + 1] = {INT32_MAX, nnz}, rowptr[M] = nnz + M
// (row stream), gu_start[T] = union total (gather stream); with no scatter
// (K = 0) every panel starts at 0.
__device__ void tails(const PackGeom& g, const WriteArgs& w) {
  if (w.zero_panels)
    for (int64_t p = threadIdx.x; p < g.P; p += blockDim.x) {
      w.panel_col[p] = 0;
      w.panel_nnz[p] = 0;
    }
  if (threadIdx.x == 0) {
    w.panel_col[g.P] = (int32_t)w.n_cols;
    w.panel_nnz[g.P] = w.nnz;
    w.colrec[w.n_cols] = make_int2(INT32_MAX, (int32_t)w.nnz);
    w.colrec[w.n_cols + 1] = make_int2(INT32_MAX, (int32_t)w.nnz);
    if (w.rowptr) w.rowptr[g.M] = (int32_t)(w.nnz + g.M);
    if (w.gu_start) w.gu_start[g.T] = (int32_t)w.gu_total;
  }
}

// Phase 2 in one launch: scatter, row write (+ gather records), union lists,
// dense copies, then one block of terminating entries.  A is read from L2 by
// each of them; what bounds the launch is loads in flight, so a panel column
// fetches its sixteen rows together, a row its next 256 columns while it writes
// the last, and a dense copy eight columns per thread (512 x 4608 at 95 %:
// 35 -> 16 us; transposed 35 -> 14).
template <class S, class D>
__global__ void __launch_bounds__(kPackThreads)
    pack_write_kernel(const S* __restrict__ A, PackGeom g, const float* __restrict__ scale,
                      WriteArgs w) {
  pdl_wait();
  pdl_trigger();
  int64_t b = blockIdx.x;
  if (b < w.b_scatter) {
    scatter<S, D>(A, g, scale, b, w);
    return;
  }
  b -= w.b_scatter;
  if (b < w.b_row) {
    if (w.row_warps > 1)
      row_write<S, D, kRowsPerBlock>(A, g, scale, b, w);
    else
      row_write<S, D, 1>(A, g, scale, b, w);
    return;
  }
  b -= w.b_row;
  if (b < w.b_union) {
    tile_union(g, b, w);
    return;
  }
  b -= w.b_union;
  if constexpr (std::is_same<D, __nv_bfloat16>::value || std::is_same<D, int8_t>::value) {
    if (b < w.b_dense) {
      densify<S, D>(A, g, scale, b, w);
      return;
    }
  }
  tails(g, w);
}

template <class D>
__global__ void unpack_kernel(const int32_t* __restrict__ panel_col,
                              const int2* __restrict__ colrec, const void* __restrict__ nz,
                              int m_r, int64_t lda, D* __restrict__ out) {
  const int64_t p = blockIdx.x;
  for (int64_t c = panel_col[p] + threadIdx.x; c < panel_col[p + 1]; c += blockDim.x) {
    const int64_t k = colrec[c].x;
    for (int32_t e = colrec[c].y; e < colrec[c + 1].y; ++e)
      out[(p * m_r + get_row(nz, e, D())) * lda + k] = get_val(nz, e, D());
  }
}

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Stream-ordered scratch from the library's pool, released in the order of
// its stream (so an early return never frees memory that queued work uses).
struct PoolScratch {
  void* p = nullptr;
  cudaStream_t st = nullptr;
  ~PoolScratch() { pool_free(p, st); }
};

__global__ void fill_kernel(float* __restrict__ out, int64_t n, float v) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = v;
}

// ---- work segments of the row-direct traversal (see rosko_packed_s) --------
// Planned on the device: the host only learns how many pieces each panel has.
// (Planned on the host, the piece lists and their sorting took 266 us of the
// 388 us pack of a 4608 x 512 matrix, and 1.9 of 2.7 ms for 11008 x 4096.)
// What bounds the writing kernel is the chain of row -> records -> entries of a
// half-warp: one block per 256 rows took 33 us for 512 x 4608 at 95 % (two
// blocks); several blocks that plan the same rows and share the writing, four
// pieces of a row in flight: 8 us.
//
// lpt order: pieces by length class, longest first, ties in row order.  A
// class is a range of lengths (kSegClasses of them between the list's piece
// length and 0), so the order is a stable counting sort: the summary kernel
// counts each block's pieces per class, its last block turns the counts into
// offsets, and the writing kernel ranks the pieces inside a block.
constexpr int kSegRows = 256;      // rows per block of both kernels
constexpr int kSegClasses = 64;
constexpr int kSegBatch = 4;       // pieces of a row that are in flight together

__host__ __device__ inline int seg_class_shift(int seg) {
  int s = 0;
  while ((seg >> s) >= kSegClasses) ++s;
  return s;
}
// Pieces of a row of nr nonzeros: the first ns - 1 hold seg records each, the
// last one rem.
struct RowPieces {
  int ns, rem, cls;
};
__device__ __forceinline__ RowPieces row_pieces(int nr, int seg, int shift) {
  RowPieces p;
  p.ns = nr > seg ? (nr + seg - 1) / seg : 1;
  p.rem = nr - (p.ns - 1) * seg;
  p.cls = (seg - p.rem) >> shift;
  return p;
}

// The counting half of the plan, run by pack_summary_kernel.
struct SegCount {
  const int2* rcnt;      // scanned row offsets; NULL: no row stream
  int32_t* panel_segs;   // [2][P]: pieces of a panel, bit 31: a row of it is cut
  int32_t* hist;         // [2][kSegClasses][nblk] counts, then exclusive offsets
  int* ticket;           // blocks done (starts at 0)
  int m_r, nblk;
};

// What the host needs to lay out the handle, gathered from the scans into one
// array so that a single copy brings it back:
//   sum64[0..3]    nonzeros, packed columns, touched columns, gather-union total
//   sum64[4..4+P]  nonzero offset of every panel, then the total
//   panel_segs     per list and panel the work segments (row stream only)
__global__ void __launch_bounds__(kSegRows)
    pack_summary_kernel(const int2* __restrict__ cnt, int64_t n, int64_t P, int64_t K,
                        const int* __restrict__ touched_total, int64_t M,
                        const int2* __restrict__ flag, int64_t nf, int64_t* __restrict__ sum64,
                        SegCount sc) {
  pdl_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int nnz = cnt[n].x;
  if (i == 0) {
    sum64[0] = nnz;
    sum64[1] = cnt[n].y;
    sum64[2] = *touched_total;
    sum64[3] = flag ? flag[nf].x : 0;
  }
  if (i <= P) sum64[4 + i] = i < P ? cnt[i * K].x : nnz;
  if (!sc.rcnt || (int)blockIdx.x >= sc.nblk) return;   // uniform over the block
  __shared__ int h[2 * kSegClasses];
  __shared__ bool last;
  if (threadIdx.x < 2 * kSegClasses) h[threadIdx.x] = 0;
  __syncthreads();
  const bool in = i < M;
  const int nr = in ? sc.rcnt[i + 1].x - sc.rcnt[i].x - 1 : 0;
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const int seg = g ? (int)seg_records_for(nnz, M) : kSegRecords;
    RowPieces p = row_pieces(nr, seg, seg_class_shift(seg));
    if (!in) p.ns = 0;
    if (in) {
      atomicAdd(&h[g * kSegClasses + p.cls], 1);
      if (p.ns > 1) atomicAdd(&h[g * kSegClasses], p.ns - 1);
    }
    // the rows of a panel are m_r (8, 16 or 32) neighbouring lanes
    int sum = p.ns, cut = p.ns > 1 ? 1 : 0;
    for (int o = 1; o < sc.m_r; o <<= 1) {
      sum += __shfl_xor_sync(0xffffffffu, sum, o);
      cut |= __shfl_xor_sync(0xffffffffu, cut, o);
    }
    if (in && i % sc.m_r == 0)
      sc.panel_segs[(int64_t)g * P + i / sc.m_r] = (int)((uint32_t)sum | ((uint32_t)cut << 31));
  }
  __syncthreads();
  if (threadIdx.x < 2 * kSegClasses)
    sc.hist[(int64_t)threadIdx.x * sc.nblk + blockIdx.x] = h[threadIdx.x];
  // the last block turns each list's counts into offsets
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(sc.ticket, 1) == sc.nblk - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  const int64_t len = (int64_t)kSegClasses * sc.nblk;
  const int64_t per = (len + kSegRows - 1) / kSegRows;
  const int64_t j0 = min((int64_t)threadIdx.x * per, len), j1 = min(j0 + per, len);
  int2 v = make_int2(0, 0);
  for (int64_t j = j0; j < j1; ++j) {
    v.x += __ldcg(&sc.hist[j]);
    v.y += __ldcg(&sc.hist[len + j]);
  }
  int2 total;
  int2 off = block_excl_scan(v, &total);
  for (int64_t j = j0; j < j1; ++j) {
    const int a = __ldcg(&sc.hist[j]), b = __ldcg(&sc.hist[len + j]);
    sc.hist[j] = off.x;
    sc.hist[len + j] = off.y;
    off.x += a;
    off.y += b;
  }
}

// The writing half: the entries of every list (one when both piece lengths
// are the same) from the row stream.  A block plans its 256 rows (a thread
// per row and list), then each half-warp writes the entries of a row at a
// time, one 4-byte word per lane: {row, first record, end record, cut} and
// the piece's first 48 bytes of records (zero past its end).
struct SegWrite {
  const int2* rcnt;
  const uint32_t* rnz;
  const int32_t* hist;        // offsets of (class, block), per list
  const int32_t* ord_base;    // [2][P]: first piece of a panel in panel order
  SegEntry* ord[2];           // NULL: no panel order
  SegEntry* lpt[2];
  int64_t M, P;
  int seg[2];
  int rec_words, m_r, nblk, lists;
};
__global__ void __launch_bounds__(2 * kSegRows) seg_write_kernel(const SegWrite w) {
  pdl_wait();
  __shared__ int first[kSegRows], len[kSegRows];
  __shared__ int at_full[2][kSegRows], at_rem[2][kSegRows], at_ord[2][kSegRows];
  __shared__ int base[2][kSegRows / 32][kSegClasses];   // per warp and class
  const int g = threadIdx.x >> 8, r = threadIdx.x & (kSegRows - 1);
  const int wr = r >> 5, lane = threadIdx.x & 31;
  const int64_t row = (int64_t)blockIdx.x * kSegRows + r;
  const bool in = row < w.M && g < w.lists;
  for (int i = threadIdx.x; i < 2 * (kSegRows / 32) * kSegClasses; i += 2 * kSegRows)
    (&base[0][0][0])[i] = 0;
  const int e0 = in ? w.rcnt[row].x : 0;
  const int nr = in ? w.rcnt[row + 1].x - e0 - 1 : 0;
  if (g == 0) {
    first[r] = e0;
    len[r] = in ? nr : -1;
  }
  __syncthreads();
  const int seg = w.seg[g];
  RowPieces p = row_pieces(nr, seg, seg_class_shift(seg));
  if (!in) p.ns = 0;
  // class 0 takes the row's full pieces (and its last one when that is in
  // class 0 too); the other classes at most the last piece
  const int n0 = in ? p.ns - 1 + (p.cls == 0 ? 1 : 0) : 0;
  int incl = n0;
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const int key = in && p.cls > 0 ? p.cls : 0;
  const unsigned same = __match_any_sync(0xffffffffu, key);
  const int rank = __popc(same & ((1u << lane) - 1u));
  if (key > 0 && rank == 0) base[g][wr][key] = __popc(same);
  if (lane == 31) base[g][wr][0] = incl;
  // this panel's pieces before this row
  int before = p.ns;
  for (int o = 1; o < w.m_r; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, before, o);
    if ((lane & (w.m_r - 1)) >= o) before += t;
  }
  before -= p.ns;
  __syncthreads();
  if (r < kSegClasses && g < w.lists) {
    int at = w.hist[((int64_t)g * kSegClasses + r) * w.nblk + blockIdx.x];
    for (int i = 0; i < kSegRows / 32; ++i) {
      const int c = base[g][i][r];
      base[g][i][r] = at;
      at += c;
    }
  }
  __syncthreads();
  if (in) {
    const int full0 = base[g][wr][0] + incl - n0;
    at_full[g][r] = full0;
    at_rem[g][r] = p.cls == 0 ? full0 + p.ns - 1 : base[g][wr][p.cls] + rank;
    at_ord[g][r] = w.ord[g] ? w.ord_base[(int64_t)g * w.P + row / w.m_r] + before : 0;
  }
  __syncthreads();
  const int l16 = threadIdx.x & 15;
  const int words = 12 / w.rec_words * w.rec_words;   // inline words of whole records
  const int groups = 2 * kSegRows / 16;
  for (int it = blockIdx.y * groups + (threadIdx.x >> 4); it < w.lists * kSegRows;
       it += gridDim.y * groups) {
    const int gg = it >> 8, rr = it & (kSegRows - 1);
    const int n = len[rr];
    if (n < 0) continue;
    const int sg = w.seg[gg];
    const int ns = n > sg ? (n + sg - 1) / sg : 1;
    for (int k0 = 0; k0 < ns; k0 += kSegBatch) {
      uint32_t v[kSegBatch];
#pragma unroll
      for (int i = 0; i < kSegBatch; ++i) {
        const int k = k0 + i, a = first[rr] + k * sg;
        const int e = k + 1 < ns ? a + sg : first[rr] + n;
        v[i] = 0;
        if (l16 == 0) v[i] = (uint32_t)(blockIdx.x * kSegRows + rr);
        else if (l16 == 1) v[i] = (uint32_t)a;
        else if (l16 == 2) v[i] = (uint32_t)e;
        else if (l16 == 3) v[i] = ns > 1 ? 1u : 0u;
        else if (k < ns && l16 - 4 < words && l16 - 4 < (e - a) * w.rec_words)
          v[i] = w.rnz[(int64_t)a * w.rec_words + l16 - 4];
      }
#pragma unroll
      for (int i = 0; i < kSegBatch; ++i) {
        const int k = k0 + i;
        if (k >= ns) break;
        const int to = k + 1 < ns ? at_full[gg][rr] + k : at_rem[gg][rr];
        reinterpret_cast<uint32_t*>(&w.lpt[gg][to])[l16] = v[i];
        if (w.ord[gg]) reinterpret_cast<uint32_t*>(&w.ord[gg][at_ord[gg][rr] + k])[l16] = v[i];
      }
    }
  }
}

// Dense-panel split bookkeeping (BF16 packs): 128-row tiles sorted by density,
// descending; the tiles at or above dense_min_pm per mille get a dense copy;
// panel_order lists the panels tile by tile in ascending density.
void plan_dense_tiles(rosko_packed_s* h, int32_t dense_min_pm) {
  const int64_t M = h->M, K = h->K, P = h->P;
  const int64_t T = (M + kDenseTileRows - 1) / kDenseTileRows;
  const int64_t ppt = kDenseTileRows / h->m_r;
  std::vector<double> dens((size_t)T);
  h->tile_panels.assign((size_t)T, 0);
  for (int64_t t = 0; t < T; ++t) {
    const int64_t p0 = t * ppt, p1 = std::min<int64_t>(P, p0 + ppt);
    const int64_t rows = std::min<int64_t>(kDenseTileRows, M - t * kDenseTileRows);
    dens[(size_t)t] = (double)(h->panel_nnz[(size_t)p1] - h->panel_nnz[(size_t)p0]) /
                      ((double)rows * (double)K);
    h->tile_panels[(size_t)t] = (int32_t)(p1 - p0);
  }
  h->tile_order.resize((size_t)T);
  for (int64_t t = 0; t < T; ++t) h->tile_order[(size_t)t] = (int32_t)t;
  std::stable_sort(h->tile_order.begin(), h->tile_order.end(),
                   [&](int32_t a, int32_t b) { return dens[(size_t)a] > dens[(size_t)b]; });
  h->tile_density.resize((size_t)T);
  int64_t n_copy = 0;
  for (int64_t c = 0; c < T; ++c) {
    h->tile_density[(size_t)c] = dens[(size_t)h->tile_order[(size_t)c]];
    if (h->tile_density[(size_t)c] * 1000.0 >= (double)dense_min_pm) n_copy = c + 1;
  }
  std::vector<int32_t>& panel_order = h->panel_order_host;
  panel_order.clear();
  panel_order.reserve((size_t)P);
  for (int64_t c = T - 1; c >= 0; --c) {
    const int64_t t = h->tile_order[(size_t)c];
    for (int64_t q = 0; q < h->tile_panels[(size_t)t]; ++q)
      panel_order.push_back((int32_t)(t * ppt + q));
  }
  h->n_tiles = T;
  h->n_copy = n_copy;
  h->Kpad = (K + 7) / 8 * 8;
}

// The host's part of the work segments: per list the pieces and cut panels
// among the first i panels of panel_order (or of the natural order), and each
// panel's first piece in that order.
void plan_segments(rosko_packed_s* h, const int32_t* panel_segs, bool panel_order,
                   std::vector<int32_t>* ord_base) {
  const int64_t P = h->P;
  ord_base->assign((size_t)(2 * P), 0);
  for (int g = 0; g < 2; ++g) {
    rosko_packed_s::SegList& L = h->segs[g];
    L.records = g ? (int32_t)seg_records_for(h->nnz, h->M) : kSegRecords;
    L.prefix.assign((size_t)P + 1, 0);
    L.split.assign((size_t)P + 1, 0);
    for (int64_t i = 0; i < P; ++i) {
      const int64_t p = panel_order ? h->panel_order_host[(size_t)i] : i;
      const uint32_t v = (uint32_t)panel_segs[(size_t)(g * P + p)];
      (*ord_base)[(size_t)(g * P + p)] = (int32_t)L.prefix[(size_t)i];
      L.prefix[(size_t)i + 1] = L.prefix[(size_t)i] + (int64_t)(v & 0x7FFFFFFFu);
      L.split[(size_t)i + 1] = L.split[(size_t)i] + (int32_t)(v >> 31);
    }
  }
}

// Bump allocator over byte offsets, each region 256-byte aligned.
struct Layout {
  size_t top = 0;
  size_t take(size_t bytes, size_t align = 256) {
    top = align_up(top, align);
    const size_t at = top;
    top += bytes;
    return at;
  }
};

// The whole pack in two phases with one host round trip:
//   1. every counting pass (per panel column: Alg. 1's counts; per row: the
//      row stream; per 128-row tile and column: the gather union), their
//      scans, and one summary array copied back;
//   2. the host lays out the handle in one allocation (plus the tile order
//      and segment lists it derives from the summary, staged in one copy),
//      then every writing pass runs.
template <class S, class D>
rosko_status pack_typed(const S* A, int64_t lda, const float* scale_in, bool quantize_rows,
                        int32_t dense_min_pm, rosko_packed_s* h, cudaStream_t st) {
  const int64_t M = h->M, K = h->K, P = h->P;
  const int64_t n = P * K;
  const int64_t T = (M + kDenseTileRows - 1) / kDenseTileRows;
  const bool rows = M > 0 && K < kRowSlotMaxK;
  const bool gather = rows && h->m_r == 16 && K > 0;
  const bool dense = (std::is_same<D, __nv_bfloat16>::value || std::is_same<D, int8_t>::value) &&
                     dense_min_pm <= 1000 && M > 0 && K > 0;
  const int64_t nf = gather ? T * K : 0;
  auto blocks_for = [](int64_t x) { return (x + kScanTile - 1) / kScanTile + 1; };

  // ---- phase 1: counts ------------------------------------------------------
  Layout s;
  const size_t o_cnt = s.take((size_t)(n + 1) * sizeof(int2));
  const size_t o_sums = s.take((size_t)blocks_for(n) * sizeof(int2));
  const size_t o_touch = s.take((size_t)std::max<int64_t>(K, 1) * sizeof(int));
  const size_t o_tot = s.take(16);
  const size_t o_rcnt = s.take(rows ? (size_t)(M + 1) * sizeof(int2) : 0);
  const size_t o_rsums = s.take(rows ? (size_t)blocks_for(M) * sizeof(int2) : 0);
  const size_t o_flag = s.take((size_t)(nf + 1) * sizeof(int2));
  const size_t o_fsums = s.take((size_t)blocks_for(nf) * sizeof(int2));
  const size_t o_scale = s.take(quantize_rows ? (size_t)M * 4 : 0);
  const size_t o_sum64 = s.take((size_t)(P + 5) * 8);
  const size_t o_psegs = s.take(rows ? (size_t)(2 * P) * 4 : 0);
  const size_t summary_bytes = s.top - o_sum64;
  const int64_t nblk = (M + kSegRows - 1) / kSegRows;
  PoolScratch scr;
  scr.st = st;
  if (pool_malloc(&scr.p, s.top + 256, st) != cudaSuccess) return ROSKO_ERR_OOM;
  // the segment plan's class counts (packs with a row stream)
  PoolScratch seg_scr;
  seg_scr.st = st;
  if (rows && pool_malloc(&seg_scr.p, (size_t)(2 * kSegClasses * nblk) * 4, st) != cudaSuccess)
    return ROSKO_ERR_OOM;
  int32_t* seg_hist = static_cast<int32_t*>(seg_scr.p);
  char* sb = static_cast<char*>(scr.p);
  int2* cnt = reinterpret_cast<int2*>(sb + o_cnt);
  int* touched = reinterpret_cast<int*>(sb + o_touch);
  int* tot = reinterpret_cast<int*>(sb + o_tot);
  int2* rcnt = rows ? reinterpret_cast<int2*>(sb + o_rcnt) : nullptr;
  int2* flag = gather ? reinterpret_cast<int2*>(sb + o_flag) : nullptr;

  // touched flags, totals, row counts (and their tile sums) and tile flags
  // are adjacent: one memset
  if (cudaMemsetAsync(touched, 0, o_fsums - o_touch, st) != cudaSuccess ||
      (n == 0 && cudaMemsetAsync(cnt, 0, sizeof(int2), st) != cudaSuccess))
    return ROSKO_ERR_CUDA;
  const float* scale = nullptr;
  if (quantize_rows) {
    scale = reinterpret_cast<float*>(sb + o_scale);
    const int wpb = 8;
    if (M > 0) {
      rowscale_kernel<<<(unsigned)((M + wpb - 1) / wpb), wpb * 32, 0, st>>>(
          reinterpret_cast<const float*>(A), M, K, lda, const_cast<float*>(scale));
      count_launches(1);
    }
  }
  PackGeom geo;
  geo.M = M;
  geo.K = K;
  geo.lda = lda;
  geo.P = P;
  geo.T = T;
  geo.m_r = h->m_r;
  geo.gx = (K + kPackThreads - 1) / kPackThreads;
  const int64_t b_col = n > 0 ? geo.gx * P : 0;
  // rows are counted by the column blocks; without columns (K = 0) every row
  // still gets its sentinel from a row block
  const int64_t b_row_count = (rows && n == 0) ? (M + kRowsPerBlock - 1) / kRowsPerBlock : 0;
  if (b_col + b_row_count > 0) {
    // (the launches of a phase are programmatic dependents of one another:
    // each is scheduled while the one before it ends)
    if (launch_dependent(pack_count_kernel<S, D>, dim3((unsigned)(b_col + b_row_count)),
                         dim3(kPackThreads), 0, st, A, geo, scale, cnt, touched, tot + 2, rcnt,
                         flag, b_col) != cudaSuccess)
      return ROSKO_ERR_CUDA;
    count_launches(1);
  }
  // the writing phase's ranges
  // A warp per row is a chain of steps of 256 columns, which few rows leave
  // exposed: up to 16 warps per SM a block shares each row (whole pack, BF16,
  // a warp per row -> a block: 512x4608 at 50 % 148 -> 119 us, at 95 % 118 -> 98;
  // above that it only adds barriers: 4608x512 110 -> 131, 4096x4096 241 -> 250).
  // Rows of one step stay with a warp.
  const bool share_rows = M <= 16 * (int64_t)num_sms() && K > 256;
  const int64_t b_row = !rows ? 0 : share_rows ? M : (M + kRowsPerBlock - 1) / kRowsPerBlock;
  const int64_t b_tile = gather ? geo.gx * T : 0;
  {
    ScanSet ss;
    std::memset(&ss, 0, sizeof(ss));
    auto add = [&](int2* data, int64_t len, size_t o_s) {
      if (len <= 0) return;
      ScanJob& J = ss.job[ss.count];
      J.data = data;
      J.n = len;
      J.sums = reinterpret_cast<int2*>(sb + o_s);
      J.nb = (len + kScanTile - 1) / kScanTile;
      ss.first[ss.count + 1] = ss.first[ss.count] + J.nb;
      ++ss.count;
    };
    add(cnt, n, o_sums);
    if (rows) add(rcnt, M, o_rsums);
    if (gather) add(flag, nf, o_fsums);
    if (ss.count > 0) {
      const unsigned tiles = (unsigned)ss.first[ss.count];
      if (launch_dependent(scan_reduce_kernel, dim3(tiles), dim3(kScanThreads), 0, st, ss) !=
              cudaSuccess ||
          launch_dependent(scan_spine_kernel, dim3((unsigned)ss.count), dim3(kScanThreads), 0, st,
                           ss) != cudaSuccess ||
          launch_dependent(scan_down_kernel, dim3(tiles), dim3(kScanThreads), 0, st, ss) !=
              cudaSuccess)
        return ROSKO_ERR_CUDA;
      count_launches(3);
    }
  }
  {
    const int64_t span = std::max<int64_t>(P, M) + 1;
    SegCount sc;
    std::memset(&sc, 0, sizeof(sc));
    if (rows) {
      sc.rcnt = rcnt;
      sc.panel_segs = reinterpret_cast<int32_t*>(sb + o_psegs);
      sc.hist = seg_hist;
      sc.ticket = tot + 3;
      sc.m_r = h->m_r;
      sc.nblk = (int)nblk;
    }
    if (launch_dependent(pack_summary_kernel, dim3((unsigned)((span + kSegRows - 1) / kSegRows)),
                         dim3(kSegRows), 0, st, cnt, n, P, K, tot + 2, M, flag, nf,
                         reinterpret_cast<int64_t*>(sb + o_sum64), sc) != cudaSuccess)
      return ROSKO_ERR_CUDA;
    count_launches(1);
  }
  std::vector<int64_t> summary((summary_bytes + 7) / 8);
  if (cudaGetLastError() != cudaSuccess ||
      cudaMemcpyAsync(summary.data(), sb + o_sum64, summary_bytes, cudaMemcpyDeviceToHost, st) !=
          cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return ROSKO_ERR_CUDA;

  // ---- host: sizes, dense tiles, segments, layout ----------------------------
  h->nnz = summary[0];
  h->n_cols = summary[1];
  h->touched_k = summary[2];
  h->gu_total = gather ? summary[3] : 0;
  h->panel_nnz.assign(summary.begin() + 4, summary.begin() + 5 + P);
  if (dense) plan_dense_tiles(h, dense_min_pm);
  std::vector<int32_t> ord_base;
  if (rows)
    plan_segments(h,
                  reinterpret_cast<const int32_t*>(reinterpret_cast<const char*>(summary.data()) +
                                                   (o_psegs - o_sum64)),
                  dense, &ord_base);
  // both piece lengths the same: one list serves as both
  const int lists = !rows ? 0 : (h->segs[0].records == h->segs[1].records ? 1 : 2);

  const size_t rsz = rec_size(h->dt);
  const int64_t nnz = h->nnz, n_cols = h->n_cols;
  Layout L;
  // staged from the host in one copy
  const size_t o_to = L.take(dense ? (size_t)T * 4 : 0);
  const size_t o_po = L.take(dense ? (size_t)P * 4 : 0);
  const size_t o_ob = L.take(dense && rows ? ord_base.size() * 4 : 0);
  const size_t staged = L.top;
  size_t o_ord[2] = {0, 0}, o_lpt[2] = {0, 0};
  for (int g = 0; g < lists; ++g) {
    const size_t bytes = (size_t)h->segs[g].prefix[(size_t)P] * sizeof(SegEntry);
    o_ord[g] = L.take(dense ? bytes : 0);
    o_lpt[g] = L.take(bytes);
  }
  // written on the device
  const size_t o_pc = L.take((size_t)(P + 1) * 4);
  const size_t o_pn = L.take((size_t)(P + 1) * 8);
  const size_t o_rs = L.take((size_t)std::max<int64_t>(M, 1) * 4);
  const size_t o_ft = L.take(256);
  const size_t o_cr = L.take((size_t)(n_cols + 2) * 8);
  const size_t o_nz = L.take((size_t)(nnz + 1) * rsz);
  const size_t o_rowptr = L.take(rows ? (size_t)(M + 1) * 4 : 0);
  const size_t o_rnz = L.take(rows ? (size_t)(nnz + M) * rsz : 0);
  const size_t o_gs = L.take(gather ? (size_t)(T + 1) * 4 : 0);
  const size_t o_gk = L.take(gather ? (size_t)std::max<int64_t>(h->gu_total, 1) * 4 : 0);
  const size_t o_gnz = L.take(gather ? (size_t)(nnz + M) * rsz : 0);
  const size_t o_da =
      L.take(dense ? (size_t)h->n_copy * kDenseTileRows * (size_t)h->Kpad * 2 : 0, 1024);
  if (pool_malloc(&h->base, L.top + 256, st) != cudaSuccess) return ROSKO_ERR_OOM;
  h->base_bytes = L.top + 256;
  char* b = static_cast<char*>(h->base);
  h->panel_col = reinterpret_cast<int32_t*>(b + o_pc);
  h->panel_nnz_dev = reinterpret_cast<int64_t*>(b + o_pn);
  h->row_scale = reinterpret_cast<float*>(b + o_rs);
  h->feat_dev = reinterpret_cast<float*>(b + o_ft);
  h->colrec = reinterpret_cast<int2*>(b + o_cr);
  h->nz = b + o_nz;
  if (rows) {
    h->rowptr = reinterpret_cast<int32_t*>(b + o_rowptr);
    h->rnz = b + o_rnz;
    for (int g = 0; g < 2; ++g) {
      const int l = g < lists ? g : 0;
      h->segs[g].ord = dense ? reinterpret_cast<SegEntry*>(b + o_ord[l]) : nullptr;
      h->segs[g].lpt = reinterpret_cast<SegEntry*>(b + o_lpt[l]);
    }
  }
  if (gather) {
    h->gu_start = reinterpret_cast<int32_t*>(b + o_gs);
    h->gu_k = reinterpret_cast<int32_t*>(b + o_gk);
    h->gnz = b + o_gnz;
  }
  if (dense) {
    h->tile_order_dev = reinterpret_cast<int32_t*>(b + o_to);
    h->panel_order_dev = reinterpret_cast<int32_t*>(b + o_po);
    h->dense_A = b + o_da;
  }
  if (staged > 0) {
    std::vector<char> stage(staged, 0);
    if (dense) {
      std::memcpy(stage.data() + o_to, h->tile_order.data(), (size_t)T * 4);
      std::memcpy(stage.data() + o_po, h->panel_order_host.data(), (size_t)P * 4);
      if (rows) std::memcpy(stage.data() + o_ob, ord_base.data(), ord_base.size() * 4);
    }
    // a pageable source is staged before the call returns
    if (cudaMemcpyAsync(b, stage.data(), staged, cudaMemcpyHostToDevice, st) != cudaSuccess)
      return ROSKO_ERR_CUDA;
  }

  // ---- phase 2: writes ------------------------------------------------------
  if (quantize_rows) {
    if (M > 0 && cudaMemcpyAsync(h->row_scale, scale, (size_t)M * 4, cudaMemcpyDeviceToDevice,
                                 st) != cudaSuccess)
      return ROSKO_ERR_CUDA;
  } else if (h->dt == ROSKO_I8 && M > 0) {
    if (scale_in) {
      if (cudaMemcpyAsync(h->row_scale, scale_in, (size_t)M * 4, cudaMemcpyDeviceToDevice, st) !=
          cudaSuccess)
        return ROSKO_ERR_CUDA;
    } else {
      fill_kernel<<<(unsigned)std::min<int64_t>((M + 255) / 256, 1024), 256, 0, st>>>(
          h->row_scale, M, 1.0f);
      count_launches(1);
    }
  }
  WriteArgs w;
  std::memset(&w, 0, sizeof(w));
  w.cnt = cnt;
  w.colrec = h->colrec;
  w.nz = h->nz;
  w.panel_col = h->panel_col;
  w.panel_nnz = h->panel_nnz_dev;
  w.rcnt = rcnt;
  w.rowptr = h->rowptr;
  w.rnz = h->rnz;
  w.flag = flag;
  w.gu_start = h->gu_start;
  w.gu_k = h->gu_k;
  w.gnz = h->gnz;
  w.nnz = nnz;
  w.n_cols = n_cols;
  w.gu_total = h->gu_total;
  w.zero_panels = n == 0 ? 1 : 0;
  w.b_scatter = b_col;
  w.b_row = b_row;
  w.row_warps = share_rows ? kRowsPerBlock : 1;
  w.b_union = b_tile;
  if (dense && h->n_copy > 0) {
    w.tile_order = h->tile_order_dev;
    w.dense_A = reinterpret_cast<__nv_bfloat16*>(h->dense_A);
    w.dense_rows = h->n_copy * kDenseTileRows;
    w.Kpad = h->Kpad;
    w.gxd = (h->Kpad / 8 + kPackThreads - 1) / kPackThreads;
    w.a_vec = reinterpret_cast<uintptr_t>(A) % 16 == 0 && (lda * (int64_t)sizeof(S)) % 16 == 0;
    w.ry = std::min<int64_t>(w.dense_rows, 2048);
    w.b_dense = w.gxd * w.ry;
  }
  if (launch_dependent(pack_write_kernel<S, D>,
                       dim3((unsigned)(w.b_scatter + w.b_row + w.b_union + w.b_dense + 1)),
                       dim3(kPackThreads), 0, st, A, geo, scale, w) != cudaSuccess)
    return ROSKO_ERR_CUDA;
  count_launches(1);
  if (rows) {
    // the work segments, once the row stream is written
    SegWrite sw;
    std::memset(&sw, 0, sizeof(sw));
    sw.rcnt = rcnt;
    sw.rnz = static_cast<const uint32_t*>(h->rnz);
    sw.hist = seg_hist;
    sw.ord_base = dense ? reinterpret_cast<const int32_t*>(b + o_ob) : nullptr;
    for (int g = 0; g < 2; ++g) {
      sw.ord[g] = h->segs[g].ord;
      sw.lpt[g] = h->segs[g].lpt;
      sw.seg[g] = h->segs[g].records;
    }
    sw.M = M;
    sw.P = P;
    sw.rec_words = (int)(rsz / 4);
    sw.m_r = h->m_r;
    sw.nblk = (int)nblk;
    sw.lists = lists;
    // several blocks plan the same rows and share the writing until the SMs
    // have a block each (a part for every half-warp's one row at most)
    const int64_t parts =
        std::min<int64_t>(lists * 16 / 2, std::max<int64_t>(1, num_sms() / std::max<int64_t>(nblk, 1)));
    if (launch_dependent(seg_write_kernel, dim3((unsigned)nblk, (unsigned)parts),
                         dim3(2 * kSegRows), 0, st, sw) != cudaSuccess)
      return ROSKO_ERR_CUDA;
    count_launches(1);
  }
  // the scratch is released on return: wait for the writes that read it
  if (cudaStreamSynchronize(st) != cudaSuccess || cudaGetLastError() != cudaSuccess)
    return ROSKO_ERR_CUDA;
  return ROSKO_OK;
}

// out[c][r] = in[r][c] for an R x C matrix of E-byte elements (row-major,
// leading dimensions ld_in / ld_out); 32 x 32 tiles through shared memory.
template <class E>
__global__ void transpose_kernel(const E* __restrict__ in, int64_t R, int64_t C, int64_t ld_in,
                                 E* __restrict__ out, int64_t ld_out) {
  __shared__ E tile[32][33];
  const int64_t r0 = (int64_t)blockIdx.y * 32, c0 = (int64_t)blockIdx.x * 32;
  for (int j = threadIdx.y; j < 32; j += 8) {
    const int64_t r = r0 + j, c = c0 + threadIdx.x;
    if (r < R && c < C) tile[j][threadIdx.x] = in[r * ld_in + c];
  }
  __syncthreads();
  for (int j = threadIdx.y; j < 32; j += 8) {
    const int64_t c = c0 + j, r = r0 + threadIdx.x;
    if (r < R && c < C) out[c * ld_out + r] = tile[threadIdx.x][j];
  }
}

}  // namespace

// Dense K x M transpose of a row-major M x K matrix into `out` (ld = M).
rosko_status transpose_impl(const void* A, rosko_dtype dt, int64_t M, int64_t K, int64_t lda,
                            void* out, cudaStream_t st) {
  if (M == 0 || K == 0) return ROSKO_OK;
  const dim3 grid((unsigned)((K + 31) / 32), (unsigned)((M + 31) / 32));
  if (grid.y > 65535) return ROSKO_ERR_INVALID_ARG;
  const dim3 block(32, 8);
  const size_t es = dtype_size(dt);
  if (es == 4)
    transpose_kernel<uint32_t><<<grid, block, 0, st>>>(static_cast<const uint32_t*>(A), M, K, lda,
                                                       static_cast<uint32_t*>(out), M);
  else if (es == 2)
    transpose_kernel<uint16_t><<<grid, block, 0, st>>>(static_cast<const uint16_t*>(A), M, K, lda,
                                                       static_cast<uint16_t*>(out), M);
  else
    transpose_kernel<uint8_t><<<grid, block, 0, st>>>(static_cast<const uint8_t*>(A), M, K, lda,
                                                      static_cast<uint8_t*>(out), M);
  count_launches(1);
  return cudaGetLastError() == cudaSuccess ? ROSKO_OK : ROSKO_ERR_CUDA;
}

rosko_status pack_impl(const void* A, rosko_dtype a_dt, int64_t M, int64_t K, int64_t lda,
                       rosko_dtype p_dt, const float* row_scale_in, int32_t m_r,
                       int32_t dense_min_pm, cudaStream_t stream, rosko_packed_s** out) {
  rosko_packed_s* h = new (std::nothrow) rosko_packed_s();
  if (!h) return ROSKO_ERR_OOM;
  cudaGetDevice(&h->device);
  h->M = M;
  h->K = K;
  h->m_r = m_r;
  h->P = (M + m_r - 1) / m_r;
  h->dt = p_dt;
  rosko_status s = ROSKO_ERR_UNSUPPORTED;
  const int32_t dm = dense_min_pm;
  if (a_dt == ROSKO_F32 && p_dt == ROSKO_F32)
    s = pack_typed<float, float>((const float*)A, lda, nullptr, false, dm, h, stream);
  else if (a_dt == ROSKO_F32 && p_dt == ROSKO_BF16)
    s = pack_typed<float, __nv_bfloat16>((const float*)A, lda, nullptr, false, dm, h, stream);
  else if (a_dt == ROSKO_F32 && p_dt == ROSKO_F64)
    s = pack_typed<float, double>((const float*)A, lda, nullptr, false, dm, h, stream);
  else if (a_dt == ROSKO_F32 && p_dt == ROSKO_I8)
    s = pack_typed<float, int8_t>((const float*)A, lda, nullptr, true, dm, h, stream);
  else if (a_dt == ROSKO_BF16 && p_dt == ROSKO_BF16)
    s = pack_typed<__nv_bfloat16, __nv_bfloat16>((const __nv_bfloat16*)A, lda, nullptr, false, dm,
                                                 h, stream);
  else if (a_dt == ROSKO_I8 && p_dt == ROSKO_I8)
    s = pack_typed<int8_t, int8_t>((const int8_t*)A, lda, row_scale_in, false, dm, h, stream);
  if (s != ROSKO_OK) {
    pool_free(h->base, stream);
    delete h;
    return s;
  }
  h->magic = kHandleMagic;
  *out = h;
  return ROSKO_OK;
}

rosko_status unpack_impl(rosko_packed_s* h, void* A_out, int64_t lda, cudaStream_t st) {
  const size_t esz = dtype_size(h->dt);
  if (h->M > 0 && h->K > 0 &&
      cudaMemset2DAsync(A_out, (size_t)lda * esz, 0, (size_t)h->K * esz, (size_t)h->M, st) !=
          cudaSuccess)
    return ROSKO_ERR_CUDA;
  if (h->P == 0 || h->nnz == 0) return ROSKO_OK;
  const unsigned g = (unsigned)h->P;
  switch (h->dt) {
    case ROSKO_F32:
      unpack_kernel<float><<<g, 256, 0, st>>>(h->panel_col, h->colrec, h->nz, h->m_r, lda,
                                              (float*)A_out);
      break;
    case ROSKO_BF16:
      unpack_kernel<__nv_bfloat16><<<g, 256, 0, st>>>(h->panel_col, h->colrec, h->nz, h->m_r,
                                                      lda, (__nv_bfloat16*)A_out);
      break;
    case ROSKO_I8:
      unpack_kernel<int8_t><<<g, 256, 0, st>>>(h->panel_col, h->colrec, h->nz, h->m_r, lda,
                                               (int8_t*)A_out);
      break;
    case ROSKO_F64:
      unpack_kernel<double><<<g, 256, 0, st>>>(h->panel_col, h->colrec, h->nz, h->m_r, lda,
                                               (double*)A_out);
      break;
    default:
      return ROSKO_ERR_UNSUPPORTED;
  }
  count_launches(1);
  return cudaGetLastError() == cudaSuccess ? ROSKO_OK : ROSKO_ERR_CUDA;
}

}  // namespace rosko
