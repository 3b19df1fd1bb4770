// Dense-panel path on the 5th-generation tensor cores (tcgen05, sm_103a).
//
// Row tiles of A (128 rows = several packed panels) whose density is high
// enough that a dense contraction beats row skipping on CUDA cores are kept
// as dense BF16 copies.  For such tiles the whole K-first schedule of
// Sec. 4.2 runs on the tensor core: the C tile lives in tensor memory (TMEM)
// for the full K range, K slabs of A (128 x 64, K-major) and B (64 x TN,
// N-major: B is row-major K x N) stream through a ring of shared memory
// stages filled by TMA, one elected thread issues tcgen05.mma (K = 16 per
// instruction) and C is written once.
//
// Workers.  A worker is a pair of CTAs on two neighbouring SMs (CG = 2,
// cta_group::2) whenever the work has at least two row tiles, else one CTA
// (CG = 1).  A pair computes a 256 x TN tile of C: each CTA loads its own 128
// rows of A and half of B's columns, the MMA (M = 256, N = TN) reads both
// halves of B from the two shared memories, and each CTA's TMEM receives its
// own 128 x TN half of C.  What bounds this kernel is feeding the tensor
// pipe: a 128 x 256 x 64 slab takes 512 cycles of it; one CTA alone has to
// write 48 KB into shared memory and read 48 KB of operands in that time
// (96 + 96 bytes per cycle of 128), a CTA of a pair 32 KB (64 + 64), and the
// L2 -> SM traffic falls by the same third.  The smaller stages also make the
// ring six slabs deep instead of four.
//
// Warp roles: 0 = TMA producer, 1 = MMA issuer (and TMEM owner), 4-11 =
// epilogue (warp w reads TMEM lanes 32 (w % 4) .. 32 (w % 4) + 31).  The
// producer and MMA warps wait as whole warps and one elected lane issues
// (elect.sync, see elect_one: with a plain `lane == 0` branch a slab's four
// MMAs took 640-670 cycles to issue, more than the 512 that the pipe needs;
// elected, the loop runs at 508, and 11008x4096x2048 went from 115 to 96 us;
// with the chunk sums below it takes 101-112 over boxes, one CTA per tile 141).
// In a pair both CTAs run a producer (their copies complete on the even CTA's
// barrier) and an epilogue; the even CTA's MMA warp issues for both and its
// commits arrive on both CTAs' barriers.
//
// Schedule.  Workers are persistent.  A single problem with at least as many
// tiles as workers gives each worker one whole tile per round, in an order
// that keeps the tiles of a round a compact block of C (8 column tiles wide),
// so that a round reads few distinct slabs of A and B; what is left (fewer
// tiles than workers, or the whole of a batch) is cut into one equal
// contiguous share per worker along (tile, K slab), so every worker finishes
// together and layers with few row tiles still fill the GPU.  A share's ends
// snap to the tile boundary when it is closer than kMinPiece slabs.  A tile
// whose K range is cut is added into C by its pieces; only those tiles are
// zero-filled first, by a small kernel of which this launch is a programmatic
// dependent: the ring fills and MMAs start at once and only the epilogue
// waits (griddepcontrol.wait), so the fill runs under the MMAs.  Every other
// tile is stored.  Two TMEM accumulators alternate so that the epilogue of
// one range overlaps the MMAs of the next.
//
// Epilogue: each epilogue warp moves its 32 TMEM lanes (C rows) 32 columns
// at a time into a 32 x 32 FP32 staging tile in shared memory (128-byte
// swizzle, so the row-per-lane writes are bank-conflict free) and one lane
// hands the tile to TMA: a tensor store for a whole tile, a tensor
// reduce-add (element-wise add in L2) for a cut tile or C += A.B.
//
// Accumulators end every kChunkSlabs K slabs (kShortSlabs in a short range);
// the epilogue adds each chunk to its sums in registers while the next chunk's
// MMAs run, and writes C once per range.  INT8 packs run through the same BF16
// pipe (GB300's INT8 tensor rate is far below it): the codes are exact in BF16, every chunk's FP32 sum
// is still an exact integer and is converted and summed in INT32; C is INT32,
// or FP32 times the row and column scales.  (Adding every chunk into INT32 C in
// global memory instead cost an epilogue per 1,024 K: 162 against 115 us for
// 4096x11008x2048, and kept the scaled result off the tensor cores.)
// C whose rows are not 16-byte aligned falls back to direct stores and
// 16-byte atomics.
#include <algorithm>
#include <cstring>
#include <vector>

#include "handle.hpp"
#include "tc_common.cuh"
#include "wait_gate.hpp"

namespace rosko {
namespace {

constexpr int kTM = 128;             // rows of a dense tile
constexpr int kTK = 64;              // K per stage: 64 BF16 = one 128-byte swizzle row
constexpr uint32_t kABytes = kTM * kTK * 2;   // 16 KB
constexpr uint32_t kStageC = 32 * 32 * 4;      // one 32 x 32 FP32 staging tile
// Epilogue warps: two per TMEM lane quarter, and 128 columns of sums per lane in
// registers.  On 256-column tiles the two share a tile (half of its columns
// each); on 128-column ones they take the tiles in turn, so that one tile's
// waits, loads and stores overlap the next one's (with few K slabs per tile
// that chain is the whole time: 4650x239x4720 31.9 us shared, 26.7 in turn).
constexpr int kEpiWarps = 8;
// Staging tiles of a warp: one beside a 256-column ring (32 KB stages, six of
// them), two beside a 128-column one (a tile of few K slabs is bound by its
// stores, which then overlap).
template <int TN> constexpr int kStagePerWarp = TN == 128 ? 2 : 1;
template <int TN> constexpr uint32_t kEpiBytes = kEpiWarps * kStagePerWarp<TN> * kStageC;
// Warps 0-3 (producer, MMA issuer, two idle) give registers to the epilogue's
// two warpgroups: 128 sums and what the stores need do not fit the 168 that
// 384 threads can get at launch (they spilled: 108 against 98 us for
// 11008x4096x2048).  152 at launch leave room on an SM for a block of the next
// call's zero fill, which so starts before this grid has ended (1 us of a
// 512x4608x3136 call).  The shares add up to no more than the launch's total.
constexpr int kFirstEpi = 4;
constexpr int kThreads = 32 * (kFirstEpi + kEpiWarps);
constexpr int kRegsLaunch = 152, kRegsRest = 56, kRegsEpi = 200;
static_assert(128 * kRegsRest + 32 * kEpiWarps * kRegsEpi <= kThreads * kRegsLaunch,
              "setmaxnreg would wait for registers that the block does not have");
// K slabs of 64 that one accumulator sums before the epilogue takes it over
// into registers.  INT8 codes: 16 slabs = 1024 products of magnitude <= 127^2,
// so a partial sum stays below 1024 * 16129 < 2^24 and is exact in the FP32
// accumulator.  BF16: the tensor core truncates each addition, an error that
// grows with the length of the chain (2048x4096x2048 at 50 %, against 64
// bits: 2.1e-6 in chains of 54 slabs, 1.0e-6 of 27); chunks of 16 slabs added
// with round-to-nearest keep it below 1e-6 whatever K and the split are, and
// draining them costs nothing (the MMAs of the next chunk run meanwhile).
// Short ranges (a whole tile of 16 to 32 slabs, a piece of up to 16, any range
// of a batch) close their sums every 8 at the latest: a split of all the work
// over every SM would cut them there, and dealing them whole must not cost
// precision (1827x1157x1232 at 80 %: 2.6e-7 with a chain of 16 slabs, 1.4e-7
// so; 175x3497x2048 at 77 % in a batch: 1.7e-7, 1.0e-7).  For all ranges 8
// would cost the long ones 8 % (11008x4096x2048 102 -> 111 us: the drains take
// TMEM from the MMAs), 4 would cost 36 %; tiles of fewer than 16 slabs, which
// no split of a single product cuts, 7 % (7541x545x6775 184 -> 198 us).
constexpr int kChunkSlabs = 16;
constexpr int kShortSlabs = 8;
template <bool I8>
__device__ __forceinline__ int chunk_slabs(int range, bool whole, bool batch) {
  const bool is_short = batch ? range > kShortSlabs
                              : whole ? range >= kChunkSlabs && range <= 2 * kChunkSlabs
                                      : range <= kChunkSlabs;
  if (I8 || !is_short) return kChunkSlabs;
  const int n = (range + kShortSlabs - 1) / kShortSlabs;   // equal chunks
  return (range + n - 1) / n;
}
// A tile's cost in K slabs is at least its epilogue's time (128 KB per
// 128 x 256 accumulator at ~28 B/clk: about nine slabs of 512 cycles; the
// same ratio for 128-column tiles).
constexpr int kEpiCost = 9;
// Stream-K pieces shorter than this many K slabs cost more in reductions
// (every piece adds its partial tile into C) than they gain in balance.
constexpr int kMinPiece = 8;
// Column tiles of a round's block (see the schedule above).
constexpr int kGroupN = 8;

// One problem of the batch (a single SpMM is a batch of one).
struct DenseProb {
  const int32_t* tile_order;  // dense copy c holds rows tile_order[c]*128 ...
  float* C;
  int64_t ldc;
  int M, N;
  int n_copy;        // 128-row tiles (dense copies) in the work
  int mtiles;        // worker tiles: ceil(n_copy / CG) rows of them
  int ntn;           // TN-wide column tiles
  int tiles;         // mtiles * ntn
  int slabs;         // K slabs of 64 per tile
  int cost;          // max(slabs, kEpiCost)
  int cost0;         // first cost unit of this problem in the shared space
  int accumulate;
  int tma_c;         // C tensor map usable (16-byte aligned rows)
  int b3d;           // B tensor map is 3-D (64 columns x K x N / 64 chunks)
};

// The split of the work between the workers.  Rounds of whole tiles (one
// problem only): tile r * workers + w for r < rounds; then the tiles from
// tile0 on, cut along the cost space [0, units).
// cut = 0: every share ends on a tile boundary (see cut_rest; a batch with at
// least two tiles per worker: its problems would otherwise be zero-filled
// whole).
struct DenseSplit {
  int count, workers, rounds, tile0, units, cut;
};

// A position in the cut part of the work: problem, tile in it, K slab.
struct DensePos {
  int q, tile, slab;
};
constexpr int kMaxWorkers = 160;   // persistent: at most one per SM

// The whole batch travels in the kernel parameters (no device allocation):
// per problem its A and B tensor maps and its scalars.
template <int NP>
struct DenseTable {
  CUtensorMap tmA[NP];
  CUtensorMap tmB[NP];
  CUtensorMap tmC[NP];   // FP32 C, 32 x 32 boxes, 128-byte swizzle
  DenseProb p[NP];
  DenseSplit split;
  // where each worker's share begins (computed on the host: the divisions
  // cost a worker about a microsecond at its start)
  DensePos start[kMaxWorkers + 1];
  // INT8 packs: the scales of an FP32 result (NULL: C is INT32)
  const float* row_scale;
  const float* col_scale;
  // 1: the launch follows a zero fill of C that started after everything
  // before it had completed, so A and B may be read at once
  int early_ab;
  int batch;   // the launch is (part of) a batch, of one problem or more
  int* status;
};

// Where worker b's share begins (b = workers: the end of the work).  The
// cost space is divided evenly (U < 2^31 and b <= workers < 2^16, so
// floor(U b / G) is (U / G) b + ((U % G) b) / G in 32-bit divisions); a cut
// closer than kMinPiece slabs to a tile boundary moves onto it, as does every
// cut of a tile whose cost is its epilogue.
inline DensePos dense_pos(const DenseSplit& S, const DenseProb* p, int b) {
  DensePos r = {S.count, 0, 0};
  if (b >= S.workers) return r;
  const uint32_t U = (uint32_t)S.units, G = (uint32_t)S.workers;
  const uint32_t quo = U / G, rem = U - quo * G;
  const uint32_t x = quo * (uint32_t)b + rem * (uint32_t)b / G;
  if (x >= U) return r;
  int q = 0;
  while (q + 1 < S.count && x >= (uint32_t)p[q + 1].cost0) ++q;
  const uint32_t lx = x - (uint32_t)p[q].cost0, cost = (uint32_t)p[q].cost;
  int tile = (int)(lx / cost);
  int slab = (int)(lx - (uint32_t)tile * cost);
  if (!S.cut || p[q].slabs != (int)cost) {
    tile += 2 * slab >= (int)cost ? 1 : 0;
    slab = 0;
  } else if (slab < kMinPiece) {
    slab = 0;
  } else if ((int)cost - slab < kMinPiece) {
    ++tile;
    slab = 0;
  }
  tile += S.tile0;
  if (tile >= p[q].tiles) {
    ++q;
    tile = 0;
  }
  r.q = q;
  r.tile = tile;
  r.slab = slab;
  return r;
}

// Row and column of a worker tile: column groups of kGroupN tiles, inside a
// group columns fastest.
__host__ __device__ inline void dense_tile_at(const DenseProb& p, int tile, int* mt, int* nt) {
  const int per = kGroupN * p.mtiles;
  const int g = tile / per;
  const int r = tile - g * per;
  const int w = p.ntn - g * kGroupN < kGroupN ? p.ntn - g * kGroupN : kGroupN;
  *mt = r / w;
  *nt = g * kGroupN + (r - *mt * w);
}

// A worker's segments: the K slabs [s0, s1) of one tile each, in the same
// order for its three roles.
struct DenseSeg {
  int q, mt, nt, s0, s1;
  bool whole;
};
template <int NP>
struct SegIter {
  const DenseTable<NP>& T;
  int worker, round;
  DensePos c, e;
  __device__ __forceinline__ SegIter(const DenseTable<NP>& t, int w)
      : T(t), worker(w), round(0), c(t.start[w]), e(t.start[w + 1]) {}
  __device__ __forceinline__ bool next(DenseSeg& s) {
    int tile;
    if (round < T.split.rounds) {
      s.q = 0;
      tile = round * T.split.workers + worker;
      s.s0 = 0;
      s.s1 = T.p[0].slabs;
      ++round;
    } else {
      if (c.q > e.q || (c.q == e.q && (c.tile > e.tile || (c.tile == e.tile && c.slab >= e.slab))))
        return false;
      s.q = c.q;
      tile = c.tile;
      s.s0 = c.slab;
      s.s1 = (c.q == e.q && c.tile == e.tile) ? e.slab : T.p[c.q].slabs;
      c.slab = 0;
      if (++c.tile == T.p[c.q].tiles) {
        c.tile = 0;
        ++c.q;
      }
    }
    dense_tile_at(T.p[s.q], tile, &s.mt, &s.nt);
    s.whole = s.s0 == 0 && s.s1 == T.p[s.q].slabs;
    return true;
  }
};

template <int TN, int NP, int CG, bool I8>
__global__ void __cluster_dims__(CG, 1, 1) __maxnreg__(kRegsLaunch)
    dense_panel_kernel(const __grid_constant__ DenseTable<NP> T, int S) {
  constexpr int BN = TN / CG;                             // B columns this CTA loads
  constexpr uint32_t kBBytes = (uint32_t)BN * kTK * 2;
  constexpr uint32_t kStageBytes = kABytes + kBBytes;
  constexpr int NBUF = 512 / TN;                          // TMEM accumulators
  constexpr int kParts = TN / 128;                        // epilogue warps that share a tile's rows
  // 256-column tiles: both accumulators serve every tile in turn.  128-column
  // ones: two for each warpgroup's tiles, so that a group only ever waits on
  // barriers whose every phase is its own (a parity says nothing about a
  // phase further ahead).
  static_assert(NBUF == 4 / kParts, "two accumulators per group of epilogue warps");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* stage_c = smem + (size_t)S * kStageBytes;   // 1024-aligned: stages are 1 KB multiples
  uint64_t* full = reinterpret_cast<uint64_t*>(stage_c + kEpiBytes<TN>);
  uint64_t* empty = full + S;
  uint64_t* acc_full = empty + S;    // [NBUF] MMA -> epilogue: accumulator ready
  uint64_t* acc_empty = acc_full + NBUF;  // [NBUF] epilogue -> MMA: accumulator drained
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + NBUF);

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int rank = CG == 2 ? (int)cluster_rank() : 0;
  const int worker = (int)blockIdx.x / CG;
  // the next launch in the stream may be scheduled from now on (it waits for
  // this grid in its own pdl_wait)
  if (threadIdx.x == 0) pdl_trigger();

  // Set-up, overlapped per warp: the producer initialises the barriers and
  // starts its copies as soon as both CTAs' barriers exist, while warp 1
  // allocates TMEM (the epilogue's and MMA warps' barrier 1 hands it over).
  // Launched as a programmatic dependent, all of it also overlaps the tail of
  // the launch before it.
  if (warp == 0) {
    if (lane == 0) {
      for (int s = 0; s < S; ++s) {
        mbar_init(&full[s], 1);
        mbar_init(&empty[s], 1);
      }
      for (int b = 0; b < NBUF; ++b) {
        mbar_init(&acc_full[b], 1);
        mbar_init(&acc_empty[b], CG * 4 * kParts);
      }
      fence_barrier_init();
    }
    __syncwarp();
  }
  // the peer's copies and commits arrive on this CTA's barriers: both CTAs
  // must have initialised theirs
  if constexpr (CG == 2) cluster_arrive();
  else __syncthreads();
  if (warp == 1) {
    tc::tmem_alloc<CG>(tmem_slot, NBUF * TN);
    tc::tmem_relinquish<CG>();
    tc::fence_before_sync();
  }
  SegIter<NP> it(T, worker);
  DenseSeg sg;
  if constexpr (CG == 2) cluster_wait();
  uint32_t tmem = 0;
  if (warp == 1 || warp >= kFirstEpi) {
    asm volatile("bar.sync 1, %0;" ::"n"(32 * (1 + kEpiWarps)) : "memory");
    tc::fence_after_sync();
    tmem = *tmem_slot;
  }

  if (warp < kFirstEpi) {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsRest));
  if (warp == 0) {
    // ---------------- TMA producer -----------------------------------------
    if (!T.early_ab) pdl_wait();   // A and B may be the previous launch's output
    // One thread fills ring stage sj with K slab `slab` of a tile: A (this
    // CTA's 128 rows; rows past the last copy are zero-filled) and its BN / 64
    // chunks of 64 B columns, one 3-D box when N is a multiple of 64
    // (x = column in chunk, y = k, z = chunk), else one 2-D box each.
    const uint32_t full0 = CG == 2 ? cluster_addr(full, 0) : smem_u32(full);
    auto issue_stage = [&](const DenseSeg& sg, bool b3d, int slab, int sj) {
      uint8_t* a_dst = smem + (size_t)sj * kStageBytes;
      uint8_t* b_dst = a_dst + kABytes;
      const int k0 = slab * kTK;
      const int arow = (sg.mt * CG + rank) * kTM;
      const int bcol = sg.nt * TN + rank * BN;
      if constexpr (CG == 2) {
        // both CTAs' bytes are counted by the even CTA's barrier
        const uint32_t bar = full0 + (uint32_t)sj * 8u;
        if (rank == 0) mbar_arrive_expect_tx(&full[sj], 2 * kStageBytes);
        tma_load_2d_pair(a_dst, &T.tmA[sg.q], k0, arow, bar);
        if (b3d) {
          tma_load_3d_pair(b_dst, &T.tmB[sg.q], 0, k0, bcol / 64, bar);
        } else {
#pragma unroll
          for (int jj = 0; jj < BN / 64; ++jj)
            tma_load_2d_pair(b_dst + jj * (kTK * 128), &T.tmB[sg.q], bcol + 64 * jj, k0, bar);
        }
      } else {
        mbar_arrive_expect_tx(&full[sj], kStageBytes);
        tma_load_2d(a_dst, &T.tmA[sg.q], k0, arow, &full[sj]);
        if (b3d) {
          tma_load_3d(b_dst, &T.tmB[sg.q], 0, k0, bcol / 64, &full[sj]);
        } else {
#pragma unroll
          for (int jj = 0; jj < BN / 64; ++jj)
            tma_load_2d(b_dst + jj * (kTK * 128), &T.tmB[sg.q], bcol + 64 * jj, k0, &full[sj]);
        }
      }
    };
    int st = 0;
    uint32_t ph = 1;   // parity of the stage's last release (fresh: passes)
    bool ok = true;
    while (ok && it.next(sg)) {
      const bool b3d = T.p[sg.q].b3d != 0;
      for (int s = sg.s0; s < sg.s1; ++s) {
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(&empty[st], ph, T.status))) {
          ok = false;
          break;
        }
        if (elect_one()) issue_stage(sg, b3d, s, st);
        __syncwarp();
        if (++st == S) {
          st = 0;
          ph ^= 1u;
        }
      }
    }
    // every copy has landed and every commit on this CTA's barriers has
    // arrived once each stage is released (bounded; a stage that was never
    // filled passes at once)
    for (int j = 0; j < S; ++j) {
      if (!mbar_wait_bounded(&empty[st], ph, T.status)) break;
      if (++st == S) {
        st = 0;
        ph ^= 1u;
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer --------------------------------------------
    // The warp waits together; an elected lane issues the MMAs and the commits.  The
    // smem descriptors of stage 0 are built once; stage s and K step kk only
    // move the start address (a 14-bit field in 16-byte units: shared memory
    // is below 256 KB, so the sum never carries out of it).
    constexpr uint32_t idesc = tc::idesc_bf16_f32(CG * kTM, TN, false, true);
    const uint32_t sbase = smem_u32(smem);
    // A: K-major, 128-byte swizzle, 8-row groups 1024 B apart; a K step of
    // 16 BF16 is 32 bytes inside the swizzle row.  B: N-major (row k of B =
    // 128 bytes of 64 N values), 128-byte swizzle; 64-wide N chunks are
    // 64 rows x 128 B = 8 KB apart (LBO), 8-row K groups 1024 B apart (SBO);
    // a K step of 16 rows = 2 KB.
    const uint64_t a_desc0 = tc::smem_desc(sbase, 16, 1024, 2) & ~uint64_t(0x3FFF);
    const uint64_t b_desc0 = tc::smem_desc(sbase + kABytes, kTK * 128, 1024, 2) & ~uint64_t(0x3FFF);
    int st = 0;
    uint32_t ph = 0;
    bool ok = true;
    int grp = kParts - 1 ? 0 : 1;        // whose tile the current segment is
    uint32_t used0 = 0, used1 = 0;       // chunks given to each group so far
    while (rank == 0 && ok && it.next(sg)) {
      if (kParts == 1) grp ^= 1;
      const int slabs = chunk_slabs<I8>(sg.s1 - sg.s0, sg.whole, NP > 1 || T.batch);
      for (int c0 = sg.s0; ok && c0 < sg.s1;) {
        // slabs [c0, c1) sum in one accumulator
        const int c1 = min(sg.s1, c0 + slabs);
        const uint32_t u = grp ? used1++ : used0++;
        const int b = 2 * grp + (int)(u & 1u);
        // the epilogue (of both CTAs) must have drained this accumulator
        // (parity of its last release; fresh: passes)
        if (!__all_sync(0xffffffffu, mbar_wait_bounded<CG == 2>(&acc_empty[b], ((u >> 1) & 1u) ^ 1u,
                                                                T.status))) {
          ok = false;
          break;
        }
        tc::fence_after_sync();
        const uint32_t d_tmem = tmem + (uint32_t)(b * TN);
        for (int s = c0; s < c1; ++s) {
          if (!__all_sync(0xffffffffu, mbar_wait_bounded(&full[st], ph, T.status))) {
            ok = false;
            break;
          }
          tc::fence_after_sync();
          if (elect_one()) {
            const uint32_t sa = sbase + (uint32_t)st * kStageBytes;
#pragma unroll
            for (int kk = 0; kk < kTK / 16; ++kk) {
              const uint64_t ad = a_desc0 | (uint64_t)((sa + kk * 32) >> 4);
              const uint64_t bd = b_desc0 | (uint64_t)((sa + kABytes + kk * 16 * 128) >> 4);
              tc::mma_bf16<CG>(d_tmem, ad, bd, idesc, (s > c0 || kk > 0) ? 1u : 0u);
            }
            tc::mma_commit<CG>(&empty[st]);                   // stage free once these finish
            if (s + 1 == c1) tc::mma_commit<CG>(&acc_full[b]);   // accumulator complete
          }
          __syncwarp();
          if (++st == S) {
            st = 0;
            ph ^= 1u;
          }
        }
        c0 = c1;
      }
    }
    if (!ok && lane == 0) {
      // make the epilogue's waits end: release every accumulator it expects
      for (int j = 0; j < NBUF; ++j) tc::mma_commit<CG>(&acc_full[j]);
    }
    __syncwarp();
  }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsEpi));
    // ---------------- epilogue: TMEM -> registers -> C -----------------------
    // C may still be being zero-filled by the kernel this launch depends on
    // (programmatic dependent launch): wait for it before any write to C.
    // Without such a dependency the wait returns at once.
    pdl_wait();
    const int quarter = warp & 3;                  // TMEM lanes 32 quarter .. + 31
    constexpr int kChunks = TN / 32 / kParts;      // 32-column chunks of a warp
    const int group = (warp - kFirstEpi) >> 2;     // this warp's warpgroup
    const int part = kParts == 2 ? group : 0;      // its column part of a tile
    int turn = 0;                                  // whose tile comes next (kParts = 1)
    constexpr int NS = kStagePerWarp<TN>;
    uint8_t* my_stage = stage_c + (size_t)(warp - kFirstEpi) * NS * kStageC;
    int chunk = 0;   // staging tiles alternate per chunk
    const uint32_t drained = CG == 2 ? cluster_addr(acc_empty, 0) : 0u;
    uint32_t used = 0;             // chunks of this group so far
    int b = 0;                     // accumulator of the current one
    const bool i32 = I8 && !T.row_scale;
    WaitGate gate;   // (warp-uniform)
    auto wait_acc = [&]() -> bool {
      b = (kParts == 1 ? 2 * group : 0) + (int)(used & 1u);
      const bool ok = gate([&] {
        return __all_sync(0xffffffffu,
                          mbar_wait_bounded(&acc_full[b], (used >> 1) & 1u, T.status)) != 0;
      });
      ++used;
      tc::fence_after_sync();
      return ok;
    };
    const uint32_t my_tmem = tmem + ((uint32_t)(quarter * 32) << 16);
    auto release_acc = [&]() {
      // accumulator drained: hand it back to the MMA issuer
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) {
        if constexpr (CG == 2) mbar_arrive_cluster(drained + (uint32_t)b * 8u);
        else mbar_arrive(&acc_empty[b]);
      }
    };
    while (gate.open && it.next(sg)) {
      if (kParts == 1 && (turn++ & 1) != group) continue;   // the other group's tile
      const int copy = sg.mt * CG + rank;
      // the tile's C rows, fetched while the MMAs run (what else the stores
      // need is read after the sums: registers are short until then)
      const int trow = copy < T.p[sg.q].n_copy ? __ldg(&T.p[sg.q].tile_order[copy]) : -1;
      // the range's sums (FP32 or INT32 bits); at the end, in place, the bits
      // that go to C
      uint32_t sum[kChunks][32];
#pragma unroll
      for (int cc = 0; cc < kChunks; ++cc)
#pragma unroll
        for (int j = 0; j < 32; ++j) sum[cc][j] = 0;
      const int slabs = chunk_slabs<I8>(sg.s1 - sg.s0, sg.whole, NP > 1 || T.batch);
      for (int c0 = sg.s0; c0 < sg.s1; c0 += slabs) {
        if (!wait_acc()) break;
#pragma unroll
        for (int h = 0; h < 2 * kChunks; ++h) {
          uint32_t r[16];
          tc::tmem_ld_32x32b_x16(my_tmem + (uint32_t)(b * TN + part * kChunks * 32 + h * 16), r);
          tc::tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            uint32_t& t = sum[h / 2][(h & 1) * 16 + j];
            // (INT8: an exact integer in FP32, |partial| < 2^24)
            if constexpr (I8) t += (uint32_t)__float2int_rn(__uint_as_float(r[j]));
            else t = __float_as_uint(__uint_as_float(t) + __uint_as_float(r[j]));
          }
        }
        release_acc();
      }
      if (!gate.open) break;   // a wait ran out: nothing more is waited for or written
      const DenseProb& P = T.p[sg.q];
      const int q = sg.q;
      const int PM = P.M, PN = P.N;
      const int row0 = trow * kTM + quarter * 32;
      const bool rows_ok = trow >= 0 && row0 < PM;
      const int tma_c = P.tma_c;
      const bool add = !sg.whole || P.accumulate;
      const int n0 = sg.nt * TN;
      const int64_t ldc = P.ldc;
      float* c_row0 = P.C + (int64_t)row0 * ldc + lane;   // this lane's column of a chunk
      // write (or add) the 32 x 32 chunk at column col0: r[j] of lane i is
      // the value (FP32 or INT32 bits) of row row0 + i, column col0 + j
      auto put_chunk = [&](const uint32_t (&r)[32], int col0) {
        // row `lane` of the 32 x 32 chunk into a staging tile, 16-byte chunk j at
        // (j ^ (lane % 8)): the 128-byte swizzle.  The tile is free once the
        // copy issued NS chunks ago has read it.
        uint8_t* buf = my_stage + (size_t)(chunk % NS) * kStageC;
        if (lane == 0) bulk_wait_read<NS - 1>();
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 8; ++j)
          *reinterpret_cast<uint4*>(buf + lane * 128 + ((j ^ (lane & 7)) << 4)) =
              make_uint4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
        if (tma_c) {
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            // rows past M and columns past N are clipped by the tensor map
            if (add) tma_reduce_add_2d(&T.tmC[q], col0, row0, buf);
            else tma_store_2d(&T.tmC[q], col0, row0, buf);
            bulk_commit();
          }
          ++chunk;
          return;
        }
        // C rows not 16-byte aligned (no tensor map): read back row by row, so
        // that each store instruction writes 32 consecutive columns of one row
        __syncwarp();
        const int rows = PM - row0 < 32 ? PM - row0 : 32;
        if (col0 + lane < PN) {
          // some rows at a time: their shared-memory reads, then their stores
          constexpr int RB = I8 ? 8 : 16;
          float* dst = c_row0 + col0;
          const uint8_t* src = buf + (lane & 3) * 4;
          const int ch = lane >> 2;
#pragma unroll 1
          for (int r0 = 0; r0 < rows; r0 += RB, dst += RB * ldc) {
            uint32_t v[RB];
#pragma unroll
            for (int i = 0; i < RB; ++i)
              v[i] = *reinterpret_cast<const uint32_t*>(src + (r0 + i) * 128 + ((ch ^ (i & 7)) << 4));
            float* d = dst;
#pragma unroll
            for (int i = 0; i < RB; ++i, d += ldc) {
              if (r0 + i >= rows) break;
              if (!add) {
                *reinterpret_cast<uint32_t*>(d) = v[i];
              } else if (i32) {
                atomicAdd(reinterpret_cast<int*>(d), (int)v[i]);
              } else {
                atomicAdd(d, __uint_as_float(v[i]));   // a cut tile, or C += A.B
              }
            }
          }
        }
        __syncwarp();
      };
      float rs = 0.0f;
      if (I8 && !i32 && rows_ok && row0 + lane < PM) rs = __ldg(&T.row_scale[row0 + lane]);
#pragma unroll
      for (int cc = 0; cc < kChunks; ++cc) {
        const int col0 = n0 + (part * kChunks + cc) * 32;
        if (rows_ok && col0 < PN) {   // warp-uniform
          if (I8 && !i32) {
            const float cs = col0 + lane < PN ? __ldg(&T.col_scale[col0 + lane]) : 0.0f;
#pragma unroll
            for (int j = 0; j < 32; ++j)
              sum[cc][j] = __float_as_uint(((float)(int32_t)sum[cc][j] * rs) *
                                           __shfl_sync(0xffffffffu, cs, j));
          }
          put_chunk(sum[cc], col0);
        }
      }
    }
    // the staging tiles must not be released (CTA exit) while TMA reads
    // them, and C must be complete when the kernel ends
    if (lane == 0) bulk_wait_all();
    __syncwarp();
  }
  tc::fence_before_sync();
  // no CTA of a pair leaves (or frees TMEM) while the other may still signal
  // its barriers or read its shared memory
  if constexpr (CG == 2) cluster_sync_all();
  else __syncthreads();
  if (warp == 1) {
    tc::fence_after_sync();
    tc::tmem_dealloc<CG>(tmem, NBUF * TN);
  }
}

// Zero the C tiles that the split cuts (their pieces are added): block
// (b - 1, part of kFillParts) looks at the start of worker b's share, and
// zeroes its part of the tile when that is the tile's first cut.
constexpr int kFillParts = 8;
constexpr int kFillThreads = 128;   // few registers a block: see kRegsLaunch
__device__ __forceinline__ void fill_cut_tile(const DenseTable<1>& T, int CG, int TN, int b,
                                              int part) {
  const DensePos c = T.start[b + 1];
  if (c.q >= T.split.count || c.slab == 0) return;
  const DensePos prev = T.start[b];
  if (prev.q == c.q && prev.tile == c.tile && prev.slab > 0) return;
  const DenseProb& P = T.p[c.q];
  if (P.accumulate) return;
  int mt, nt;
  dense_tile_at(P, c.tile, &mt, &nt);
  const int64_t n0 = (int64_t)nt * TN;
  const int64_t cols = P.N - n0 < TN ? P.N - n0 : TN;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (int)blockDim.x >> 5;
  const bool vec = P.tma_c && cols % 4 == 0;
  for (int r = part * nw + warp; r < CG * kTM; r += kFillParts * nw) {
    const int copy = mt * CG + r / kTM;
    if (copy >= P.n_copy) continue;
    const int64_t row = (int64_t)__ldg(&P.tile_order[copy]) * kTM + r % kTM;
    if (row >= P.M) continue;
    float* dst = P.C + row * P.ldc + n0;
    if (vec) {
      for (int64_t i = lane; i < cols / 4; i += 32)
        reinterpret_cast<uint4*>(dst)[i] = make_uint4(0, 0, 0, 0);
    } else {
      for (int64_t i = lane; i < cols; i += 32) dst[i] = 0.0f;
    }
  }
}

// A programmatic dependent of the launch before it that lets the tensor-core
// launch start once that one has completed: its A and B are then final and
// only its writes of C wait for this fill.
__global__ void __launch_bounds__(kFillThreads)
    dense_cut_fill_kernel(const __grid_constant__ DenseTable<1> T, int CG, int TN) {
  pdl_wait();
  pdl_trigger();
  fill_cut_tile(T, CG, TN, (int)blockIdx.x / kFillParts, (int)blockIdx.x % kFillParts);
}

// INT8 -> BF16 (exact: |code| <= 127), K rows of N, into rows of ldo (a
// multiple of 8), by blocks [0, gx * gy); the blocks after them zero the cut
// tiles of C, so that an INT8 product has one launch ahead of the tensor-core
// one.  Bound by its 3 bytes per value of memory traffic: a lane takes 8
// consecutive codes (one 8-byte load: rows of B are 16-byte aligned; the last
// group of a row is read code by code, since nothing past N may be), writes
// 16 bytes, and has four rows in flight.  Code-by-code loads took 23 us for
// 11008 x 2048, this 9.5.
constexpr int kCvtRows = 4;
struct Convert {
  const int8_t* B;
  __nv_bfloat16* out;
  int64_t K, N, ldb, ldo;
  int gx, gy;
};
__global__ void __launch_bounds__(256)
    i8_prepare_kernel(const Convert c, const __grid_constant__ DenseTable<1> T, int CG, int TN) {
  pdl_wait();
  pdl_trigger();   // the launch after it waits in its own
  const int bid = (int)blockIdx.x - c.gx * c.gy;
  if (bid >= 0) {
    fill_cut_tile(T, CG, TN, bid / kFillParts, bid % kFillParts);
    return;
  }
  const int by = (int)blockIdx.x / c.gx, bx = (int)blockIdx.x - by * c.gx;
  const int64_t c0 = ((int64_t)bx * 32 + (threadIdx.x & 31)) * 8;
  if (c0 >= c.ldo) return;
  const bool whole = c0 + 8 <= c.N;
  for (int64_t k0 = ((int64_t)by * 8 + (threadIdx.x >> 5)) * kCvtRows; k0 < c.K;
       k0 += (int64_t)c.gy * 8 * kCvtRows) {
    uint2 v[kCvtRows];
#pragma unroll
    for (int i = 0; i < kCvtRows; ++i) {
      v[i] = make_uint2(0u, 0u);
      if (k0 + i >= c.K) break;
      const int8_t* src = c.B + (k0 + i) * c.ldb + c0;
      if (whole) {
        v[i] = __ldg(reinterpret_cast<const uint2*>(src));
      } else {
        for (int j = 0; c0 + j < c.N; ++j) {
          const uint32_t byte = (uint32_t)(uint8_t)src[j] << (8 * (j & 3));
          if (j < 4) v[i].x |= byte;
          else v[i].y |= byte;
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kCvtRows; ++i) {
      if (k0 + i >= c.K) break;
      __nv_bfloat162 o[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t w = j < 2 ? v[i].x : v[i].y;
        const int sh = 16 * (j & 1);
        o[j] = __floats2bfloat162_rn((float)(int8_t)(w >> sh), (float)(int8_t)(w >> (sh + 8)));
      }
      *reinterpret_cast<uint4*>(c.out + (k0 + i) * c.ldo + c0) = *reinterpret_cast<const uint4*>(o);
    }
  }
}

template <int TN, int CG>
constexpr int dense_stages() {
  constexpr int n = (224 * 1024 - (int)kEpiBytes<TN>) / ((int)kABytes + TN / CG * kTK * 2);
  return n > 8 ? 8 : n;
}

template <int TN, int CG>
size_t dense_smem_bytes() {
  return 1024 + (size_t)dense_stages<TN, CG>() * (kABytes + (size_t)TN / CG * kTK * 2) + kEpiBytes<TN> +
         256;
}

int64_t slabs_of(int64_t K) { return (K + kTK - 1) / kTK; }

template <int TN, int NP, int CG, bool I8>
rosko_status launch_table(const DenseTable<NP>& T, cudaStream_t st) {
  constexpr int stages = dense_stages<TN, CG>();
  const size_t smem = dense_smem_bytes<TN, CG>();
  static SmemLimit limit;
  auto fn = dense_panel_kernel<TN, NP, CG, I8>;
  if (!allow_smem(limit, fn, smem)) return ROSKO_ERR_CUDA;
  if (launch_dependent(fn, dim3((unsigned)(T.split.workers * CG)), dim3(kThreads), smem, st, T,
                       stages) != cudaSuccess)
    return ROSKO_ERR_CUDA;
  count_launches(1);
  return cudaGetLastError() == cudaSuccess ? ROSKO_OK : ROSKO_ERR_CUDA;
}

// Persistent workers: one per SM (or pair of SMs) at most, and no share below
// kMinPiece slabs unless it is a tile of its own.
int64_t split_workers(int64_t tiles, int64_t slabs, int ctas, int cg) {
  const int64_t G = std::max(1, std::min(std::min(ctas, num_sms()), kMaxWorkers) / cg);
  return std::max<int64_t>(1, std::min<int64_t>(G, std::max(tiles, slabs / kMinPiece)));
}

// What cutting tiles costs a single product, in K slabs: the zero fill of the
// cut tiles is a launch of its own (~4 us; fused with INT8's conversion; none
// when C is accumulated into).
int cut_cost(int TN, bool i8, bool accumulate) {
  return accumulate ? 0 : (i8 ? 2 : (TN == 256 ? 14 : 20));
}
// Whether to cut the `rest` tiles that do not fill a round of G workers along
// K, or deal them whole (2019x986x3352: 21.4 us cut, 18.5 whole;
// 1024x4096x4096: 32 cut, 26 whole; 512x4608x3136: 22 cut, 28 whole).
bool cut_rest(int64_t rest, int64_t cost, int64_t G, int extra) {
  return rest > 0 && rest * cost / G + extra < cost;
}

// The scalars of the problems and the split over `ctas` CTAs in workers of
// cg; false when the cost space does not fit 31 bits.
bool plan_split(const DenseJob* jobs, int count, int TN, int ctas, int cg, DenseProb* p,
                DenseSplit* S) {
  int64_t units = 0, tiles = 0, slabs_all = 0;
  int n = 0;
  for (int i = 0; i < count; ++i) {
    const DenseJob& j = jobs[i];
    if (j.n_tiles <= 0 || j.N <= 0) continue;
    DenseProb& P = p[n++];
    P.n_copy = (int)j.n_tiles;
    P.mtiles = (P.n_copy + cg - 1) / cg;
    P.ntn = (int)((j.N + TN - 1) / TN);
    P.slabs = (int)slabs_of(j.K);
    P.cost = std::max(P.slabs, kEpiCost);
    const int64_t t = (int64_t)P.mtiles * P.ntn;
    if (units >= (int64_t(1) << 31) || t >= (int64_t(1) << 31)) return false;
    P.tiles = (int)t;
    P.cost0 = (int)units;
    P.accumulate = j.accumulate;
    units += t * P.cost;
    tiles += t;
    slabs_all += t * P.slabs;
  }
  if (units >= (int64_t(1) << 31)) return false;
  S->count = n;
  const int64_t G = split_workers(tiles, slabs_all, ctas, cg);
  S->workers = (int)G;
  S->rounds = n == 1 ? (int)(tiles / G) : 0;
  S->tile0 = (int)(S->rounds * G);
  S->units = (int)(n == 1 ? (tiles - S->tile0) * p[0].cost : units);
  S->cut = tiles < 2 * G ? 1 : 0;
  if (n == 1)
    S->cut = cut_rest(tiles - S->tile0, p[0].cost, G,
                      cut_cost(TN, jobs[0].i8 != 0, p[0].accumulate != 0))
                 ? 1
                 : 0;
  return true;
}

// Which of the (active) problems has a tile cut by the split.
void cut_problems(const DenseSplit& S, const DenseProb* p, std::vector<char>* cut) {
  cut->assign((size_t)S.count, 0);
  for (int b = 1; b < S.workers; ++b) {
    const DensePos c = dense_pos(S, p, b);
    if (c.q < S.count && c.slab > 0) (*cut)[(size_t)c.q] = 1;
  }
}

// Tensor maps of one problem: A, B (bn = columns one CTA loads per slab), C.
rosko_status encode_dense_maps(const DenseJob& j, CUtensorMap* mA, CUtensorMap* mB,
                               CUtensorMap* mC, bool c_ok, int bn, bool* b3d) {
  if (c_ok) {
    const cuuint64_t dims[2] = {(cuuint64_t)j.N, (cuuint64_t)j.M};
    const cuuint64_t strides[1] = {(cuuint64_t)j.ldc * 4};
    const cuuint32_t box[2] = {32, 32};
    const cuuint32_t es[2] = {1, 1};
    const bool i32 = j.i8 && !j.row_scale;
    if (encode_tiled(mC, i32 ? CU_TENSOR_MAP_DATA_TYPE_INT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                     2, j.C, dims, strides, box, es,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                     CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) !=
        CUDA_SUCCESS)
      return ROSKO_ERR_INVALID_ARG;
  }
  {
    const cuuint64_t dims[2] = {(cuuint64_t)j.Kpad, (cuuint64_t)j.dense_rows};
    const cuuint64_t strides[1] = {(cuuint64_t)j.Kpad * 2};
    const cuuint32_t box[2] = {(cuuint32_t)kTK, (cuuint32_t)kTM};
    const cuuint32_t es[2] = {1, 1};
    if (encode_tiled(mA, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(j.dense_A), dims,
                     strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return ROSKO_ERR_INVALID_ARG;
  }
  *b3d = false;
  if (j.N % 64 == 0) {
    // B viewed as [N / 64][K][64]: chunk z starts 128 bytes after chunk z-1
    const cuuint64_t dims[3] = {64, (cuuint64_t)j.K, (cuuint64_t)(j.N / 64)};
    const cuuint64_t strides[2] = {(cuuint64_t)j.ldb * 2, 128};
    const cuuint32_t box[3] = {64, (cuuint32_t)kTK, (cuuint32_t)(bn / 64)};
    const cuuint32_t es[3] = {1, 1, 1};
    *b3d = encode_tiled(mB, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(j.B), dims,
                        strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  }
  if (!*b3d) {
    const cuuint64_t dims[2] = {(cuuint64_t)j.N, (cuuint64_t)j.K};
    const cuuint64_t strides[1] = {(cuuint64_t)j.ldb * 2};
    const cuuint32_t box[2] = {64, (cuuint32_t)kTK};
    const cuuint32_t es[2] = {1, 1};
    if (encode_tiled(mB, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(j.B), dims,
                     strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                     CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return ROSKO_ERR_INVALID_ARG;
  }
  return ROSKO_OK;
}

template <int TN, int NP, int CG, bool I8>
rosko_status run_jobs(const DenseJob* jobs, int count, int ctas, bool zero_cut, bool after_fill,
                      bool batch, cudaStream_t st) {
  static_assert(sizeof(DenseTable<NP>) <= 32 * 1024 - 256, "kernel parameter table too large");
  DenseTable<NP> T;
  std::memset(static_cast<void*>(&T), 0, sizeof(T));
  if (!plan_split(jobs, count, TN, ctas, CG, T.p, &T.split)) return ROSKO_ERR_UNSUPPORTED;
  if (T.split.count == 0) return ROSKO_OK;
  int n = 0;
  for (int i = 0; i < count; ++i) {
    const DenseJob& j = jobs[i];
    if (j.n_tiles <= 0 || j.N <= 0) continue;
    const bool c_ok = ((reinterpret_cast<uintptr_t>(j.C) % 16) == 0) && ((j.ldc * 4) % 16 == 0);
    bool b3d = false;
    rosko_status s =
        encode_dense_maps(j, &T.tmA[n], &T.tmB[n], &T.tmC[n], c_ok, TN / CG, &b3d);
    if (s != ROSKO_OK) return s;
    DenseProb& P = T.p[n];
    P.tma_c = c_ok ? 1 : 0;
    P.b3d = b3d ? 1 : 0;
    P.tile_order = j.tile_order_dev;
    P.C = j.C;
    P.ldc = j.ldc;
    P.M = (int)j.M;
    P.N = (int)j.N;
    ++n;
  }
  for (int b = 0; b <= T.split.workers; ++b) T.start[b] = dense_pos(T.split, T.p, b);
  T.row_scale = jobs[0].row_scale;
  T.col_scale = jobs[0].col_scale;
  T.batch = batch ? 1 : 0;
  T.early_ab = !I8 && (zero_cut || after_fill) ? 1 : 0;
  T.status = device_status_word();
  if (!T.status) return ROSKO_ERR_CUDA;
  const int fill_blocks = zero_cut ? std::max(1, T.split.workers - 1) * kFillParts : 0;
  if constexpr (I8) {
    // B to BF16, and the fill
    const DenseJob& j = jobs[0];
    Convert c;
    c.B = j.src_i8;
    c.out = static_cast<__nv_bfloat16*>(const_cast<void*>(j.B));
    c.K = j.K;
    c.N = j.N;
    c.ldb = j.src_ld;
    c.ldo = j.ldb;
    c.gx = (int)((c.ldo / 8 + 31) / 32);
    c.gy = (int)std::min<int64_t>((c.K + 8 * kCvtRows - 1) / (8 * kCvtRows), 4096);
    if (launch_dependent(i8_prepare_kernel, dim3((unsigned)(c.gx * c.gy + fill_blocks)), dim3(256),
                         0, st, c, T, CG, TN) != cudaSuccess)
      return ROSKO_ERR_CUDA;
    count_launches(1);
  } else if constexpr (NP == 1) {   // (a batch's caller zero-fills before the launch)
    if (fill_blocks > 0) {
      if (launch_dependent(dense_cut_fill_kernel, dim3((unsigned)fill_blocks), dim3(kFillThreads),
                           0, st, T, CG, TN) != cudaSuccess)
        return ROSKO_ERR_CUDA;
      count_launches(1);
    }
  }
  return launch_table<TN, NP, CG, I8>(T, st);
}

// CTAs per worker: pairs as soon as there are two row tiles to share and two
// CTAs to run them (a pair over a single row tile would leave half of it idle).
int group_of(int64_t n_tiles, int ctas) { return n_tiles >= 2 && ctas >= 2 ? 2 : 1; }

template <int TN, int NP, bool I8>
rosko_status dispatch_group(const DenseJob* jobs, int count, int cg, int ctas, bool zero_cut,
                            bool after_fill, bool batch, cudaStream_t st) {
  return cg == 2 ? run_jobs<TN, NP, 2, I8>(jobs, count, ctas, zero_cut, after_fill, batch, st)
                 : run_jobs<TN, NP, 1, I8>(jobs, count, ctas, zero_cut, after_fill, batch, st);
}

rosko_status dispatch_jobs(const DenseJob* jobs, int count, int TN, int cg, int ctas,
                           bool zero_cut, bool after_fill, bool batch, cudaStream_t st) {
  if (count <= 0) return ROSKO_OK;
  if ((TN != 128 && TN != 256) || count > 64) return ROSKO_ERR_INVALID_ARG;
  if (count == 1 && jobs[0].i8)
    return TN == 256
               ? dispatch_group<256, 1, true>(jobs, 1, cg, ctas, zero_cut, after_fill, batch, st)
               : dispatch_group<128, 1, true>(jobs, 1, cg, ctas, zero_cut, after_fill, batch, st);
  if (count == 1)
    return TN == 256
               ? dispatch_group<256, 1, false>(jobs, 1, cg, ctas, zero_cut, after_fill, batch, st)
               : dispatch_group<128, 1, false>(jobs, 1, cg, ctas, zero_cut, after_fill, batch, st);
  return TN == 256
             ? dispatch_group<256, 64, false>(jobs, count, cg, ctas, zero_cut, after_fill, batch, st)
             : dispatch_group<128, 64, false>(jobs, count, cg, ctas, zero_cut, after_fill, batch, st);
}

}  // namespace

bool dense_needs_zero(int64_t n_tiles, int64_t N, int64_t K, int TN, int ctas, bool i8) {
  if (n_tiles <= 0 || N <= 0) return false;
  if (ctas <= 0) ctas = num_sms();
  DenseJob j{};
  j.n_tiles = n_tiles;
  j.N = N;
  j.K = K;
  j.i8 = i8;
  DenseProb p{};
  DenseSplit S{};
  if (!plan_split(&j, 1, TN, ctas, group_of(n_tiles, ctas), &p, &S)) return false;
  std::vector<char> cut;
  cut_problems(S, &p, &cut);
  return !cut.empty() && cut[0];
}

int64_t dense_pieces(int64_t n_tiles, int64_t N, int64_t K, int TN, int ctas) {
  if (n_tiles <= 0 || N <= 0) return 1;
  if (ctas <= 0) ctas = num_sms();
  DenseJob j{};
  j.n_tiles = n_tiles;
  j.N = N;
  j.K = K;
  j.i8 = 1;
  DenseProb p{};
  DenseSplit S{};
  if (!plan_split(&j, 1, TN, ctas, group_of(n_tiles, ctas), &p, &S) || !S.cut) return 1;
  if (S.rounds > 0) return 1;   // most tiles are dealt whole
  const int64_t share = std::max(1, S.units / S.workers);
  return (p.slabs + share - 1) / share;
}

// ~4.6 us around the first and last slabs, the longest share at the measured
// rate per slab (a 256-column slab runs at ~530 cycles of the 512 that the
// pipe needs, a 128-column one at ~350: it moves 96 bytes per pipe cycle into
// each SM), the last tile's epilogue, the zero fill of cut tiles (a launch),
// INT8 into rows of C that are not 16-byte aligned (~4.5 us: dequantised
// 2543x5414x14 / x16 at 96 % 20.1 / 15.6; more where many are added in pieces:
// 1443x3491x907 31 against 28 row-direct), and no less than the memory needs.
// Called on every product: the split's sizes without its positions.
double dense_time_us(int64_t n_tiles, int64_t N, int64_t K, int TN, int ctas, bool i8, bool c16) {
  if (n_tiles <= 0 || N <= 0 || K <= 0) return 0.0;
  if (ctas <= 0) ctas = num_sms();
  const int cg = group_of(n_tiles, ctas);
  const int64_t slabs = slabs_of(K), cost = std::max<int64_t>(slabs, kEpiCost);
  const int64_t tiles = (n_tiles + cg - 1) / cg * ((N + TN - 1) / TN);
  const int64_t G = split_workers(tiles, tiles * slabs, ctas, cg);
  const int64_t rounds = tiles / G, rest = tiles - rounds * G;
  const bool cut = slabs >= 2 * kMinPiece && cut_rest(rest, cost, G, cut_cost(TN, i8, false));
  const double share = (double)rounds * cost +
                       (cut ? (double)rest * cost / G : (rest > 0 ? (double)cost : 0.0));
  const double mem = (2.0 * (double)n_tiles * kTM * K + 2.0 * (double)K * N +
                      4.0 * (double)n_tiles * kTM * N) / 6.5e6;
  return 4.6 + std::max(share * (TN == 256 ? 0.275 : 0.185), mem) + (TN == 256 ? 3.7 : 1.9) +
         (cut && !i8 ? 4.0 : 0.0) +
         (i8 && !c16 ? 4.5 + (cut && rounds == 0 ? 2e-6 * (double)n_tiles * kTM * (double)N : 0.0)
                     : 0.0);
}

rosko_status dense_batch_launch(const DenseJob* jobs, int count, int TN, int cg, cudaStream_t st) {
  return dispatch_jobs(jobs, count, TN, cg, num_sms(), false, false, true, st);
}

// Which jobs of a batch have a tile cut between workers (job order as given;
// the caller zero-fills their C unless they accumulate).
void dense_batch_needs_zero(const DenseJob* jobs, int count, int TN, int cg, bool* out) {
  std::vector<DenseProb> p((size_t)std::max(count, 1));
  DenseSplit S{};
  for (int i = 0; i < count; ++i) out[i] = false;
  if (!plan_split(jobs, count, TN, num_sms(), cg, p.data(), &S)) return;   // the launch refuses it
  std::vector<char> cut;
  cut_problems(S, p.data(), &cut);
  for (int i = 0, n = 0; i < count; ++i)
    if (jobs[i].n_tiles > 0 && jobs[i].N > 0) out[i] = cut[(size_t)n++] != 0;
}

int dense_group(int64_t n_tiles) { return group_of(n_tiles, num_sms()); }

namespace {
// Zero rows x row_bytes of C (pitch bytes apart), one CTA per row at a time.
// As dense_cut_fill_kernel, a link of the programmatic chain.
__global__ void zero_fill_kernel(char* __restrict__ C, int64_t pitch, int64_t row_bytes,
                                 int64_t rows, int vec16) {
  pdl_wait();
  pdl_trigger();   // the tensor-core launch after it starts now
  for (int64_t r = blockIdx.x; r < rows; r += gridDim.x) {
    char* row = C + r * pitch;
    if (vec16) {
      uint4* p = reinterpret_cast<uint4*>(row);
      for (int64_t i = threadIdx.x; i < row_bytes / 16; i += blockDim.x) p[i] = make_uint4(0, 0, 0, 0);
    } else {
      uint32_t* p = reinterpret_cast<uint32_t*>(row);
      for (int64_t i = threadIdx.x; i < row_bytes / 4; i += blockDim.x) p[i] = 0u;
    }
  }
}

}  // namespace

rosko_status zero_fill_launch(const ZeroFill& z, cudaStream_t st) {
  if (z.rows <= 0 || z.row_bytes <= 0) return ROSKO_OK;
  // every C element type is a multiple of 4 bytes
  if ((reinterpret_cast<uintptr_t>(z.C) % 4) != 0 || z.pitch % 4 != 0 || z.row_bytes % 4 != 0)
    return ROSKO_ERR_INVALID_ARG;
  const int vec16 = (reinterpret_cast<uintptr_t>(z.C) % 16 == 0 && z.pitch % 16 == 0 &&
                     z.row_bytes % 16 == 0)
                        ? 1
                        : 0;
  // a grid that is resident at once, so that every CTA has signalled its
  // dependents before the tensor-core launch needs an SM
  const int64_t grid = std::min<int64_t>(z.rows, (int64_t)num_sms() * 4);
  if (launch_dependent(zero_fill_kernel, dim3((unsigned)grid), dim3(256), 0, st,
                       static_cast<char*>(z.C), z.pitch, z.row_bytes, z.rows, vec16) !=
      cudaSuccess)
    return ROSKO_ERR_CUDA;
  count_launches(1);
  return cudaGetLastError() == cudaSuccess ? ROSKO_OK : ROSKO_ERR_CUDA;
}

rosko_status dense_spmm_i8_launch(const rosko_packed_s* h, int64_t n_tiles, const int8_t* B,
                                  int64_t N, int64_t ldb, const float* col_scale, void* C,
                                  int64_t ldc, int accumulate, int TN, int ctas, bool zero_cut,
                                  const ZeroFill* zf, cudaStream_t st) {
  if (n_tiles <= 0 || N <= 0) return ROSKO_OK;
  if (ctas <= 0) ctas = num_sms();
  const int64_t K = h->K;
  const int64_t ldo = (N + 7) / 8 * 8;   // 16-byte rows for the tensor map
  void* scratch = nullptr;
  // stream-ordered (and capturable) from the library's pool, which keeps
  // freed memory mapped: released after the launch that reads it
  if (pool_malloc(&scratch, (size_t)std::max<int64_t>(K * ldo, 1) * 2, st) != cudaSuccess)
    return ROSKO_ERR_OOM;
  // the zero fill of all of C when the sparse panels need it too
  rosko_status s = zf ? zero_fill_launch(*zf, st) : ROSKO_OK;
  if (s == ROSKO_OK) {
    DenseJob j;
    j.dense_A = h->dense_A;
    j.dense_rows = h->n_copy * kTM;
    j.Kpad = h->Kpad;
    j.tile_order_dev = h->tile_order_dev;
    j.n_tiles = n_tiles;
    j.K = K;
    j.B = scratch;
    j.N = N;
    j.ldb = ldo;
    j.C = static_cast<float*>(C);
    j.ldc = ldc;
    j.M = h->M;
    j.accumulate = accumulate;
    j.i8 = 1;
    j.src_i8 = B;
    j.src_ld = ldb;
    j.row_scale = col_scale ? h->row_scale : nullptr;
    j.col_scale = col_scale;
    s = dispatch_jobs(&j, 1, TN, group_of(n_tiles, ctas), ctas, zero_cut, zf != nullptr, false, st);
  }
  pool_free(scratch, st);
  return s;
}

rosko_status dense_spmm_launch(const rosko_packed_s* h, int64_t n_tiles, const void* B, int64_t N,
                               int64_t ldb, float* C, int64_t ldc, int accumulate, int TN,
                               int ctas, bool zero_cut, const ZeroFill* zf, cudaStream_t st) {
  if (n_tiles <= 0 || N <= 0) return ROSKO_OK;
  if (ctas <= 0) ctas = num_sms();
  // the whole of C (the sparse panels need it too), or only the cut tiles
  if (zf) {
    rosko_status s = zero_fill_launch(*zf, st);
    if (s != ROSKO_OK) return s;
  }
  DenseJob j;
  j.dense_A = h->dense_A;
  j.dense_rows = h->n_copy * kTM;
  j.Kpad = h->Kpad;
  j.tile_order_dev = h->tile_order_dev;
  j.n_tiles = n_tiles;
  j.K = h->K;
  j.B = B;
  j.N = N;
  j.ldb = ldb;
  j.C = C;
  j.ldc = ldc;
  j.M = h->M;
  j.accumulate = accumulate;
  // (after its zero fill the launch reads A and B before any wait: the fill
  // started after every earlier launch had completed)
  return dispatch_jobs(&j, 1, TN, group_of(n_tiles, ctas), ctas, zero_cut, zf != nullptr, false, st);
}

}  // namespace rosko
