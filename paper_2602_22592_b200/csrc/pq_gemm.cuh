// Persistent, warp-specialised tcgen05 GEMM engine for sm_100a.
//
// Warp 0 = TMA producer, warp 1 = MMA issuer (also owns the TMEM allocation), the others = epilogue (kEpiWarps / 4 per
// TMEM lane quadrant, which share the column chunks of the tile).  Operands travel global -> shared by TMA into a ring
// of 128-byte-swizzled stages; tcgen05.mma accumulates in TMEM; the epilogue reads the accumulators with tcgen05.ld.
//
// Two forms, chosen by the problem (P::CG):
//   CG = 2  a pair of CTAs (cluster of two, one CTA per SM) works on a tile of 256 rows x (<= 256) columns: each CTA
//           loads its 128 rows of A and its half of B's columns, one thread of the first CTA issues the MMAs for both,
//           and each CTA's TMEM receives its own 128 rows of the result.  This is the form of the large products: a step
//           of 64 (bf16) or 128 (int8) contraction values of a 128 x 256 tile is 512 MMA cycles, but 48 KB of operands for
//           one CTA alone -- 768 cycles of the 64 bytes per clock that an SM takes in from L2 -- and 32 KB, 512 cycles,
//           for a CTA of a pair.
//   CG = 1  one CTA, tiles of 128 rows: the small grouped products of the HP branch, whose rows belong to one expert
//           per 128-row item.
//
// A tile's contraction is a list of SEGMENTS.  Each segment names its operand
// form (int8 or bf16; each operand either contraction-contiguous "K" or
// output-dimension-contiguous "MN"), its tensor maps and start coordinates,
// the number of 128-byte k-blocks, and which of the tile's accumulators it
// adds into.  This lets one kernel chain, e.g., the int8 1-bit product, the
// bf16 expert product and the router product of one output tile.
//
// A "Problem" type supplies the tile list, the segments and the epilogue.  Tiles go to the CTAs (or pairs) in turn or, where
// their lengths differ (P::kTickets, pairs only), by a counter in global memory: whoever is free takes the next one.
#pragma once
#include <cuda.h>

#include <type_traits>

#include "pq_common.cuh"

namespace pq {

constexpr int kMaxStages = 12;            // barrier pairs reserved for the operand ring
constexpr int kTileM = 128;
constexpr int kOperandBytes = 128 * 128;  // 128 rows x 128 B, or two 64x64 bf16 MN boxes: one stage of one operand of a CTA
constexpr int kRingBytes = 12 * kOperandBytes;
constexpr int kMnBoxBytes = 64 * 128;    // one MN-major box: 64 k-rows of 64 bf16
constexpr int kTmemCols = 512;
constexpr int kAccCols = 256;            // TMEM columns of one accumulator
constexpr int kStagingBytes = 32 * 1024; // epilogue warps: transposing buffers (kStagingBytes / kEpiWarps each)
constexpr int kBarrierBytes = 384;
constexpr int kGemmSmemBytes = kRingBytes + 1024 /*alignment slack*/ + kBarrierBytes + kStagingBytes;
static_assert(kGemmSmemBytes <= 227 * 1024, "shared memory of one CTA");

enum OpMode : int {
  MODE_I8_KK = 0,  // int8, A[M,K] and B[N,K] K-contiguous
  MODE_BF_KK = 1,  // bf16, both K-contiguous
  MODE_BF_KM = 2,  // bf16, A K-contiguous, B N-contiguous
  MODE_BF_MM = 3   // bf16, A M-contiguous, B N-contiguous
};

// What one CTA contributes to a step of 128 contraction bytes (64 rows of an MN-major operand) of a tile: 128 rows of A
// and its share of B -- all of it (CG = 1) or one half of its columns (CG = 2).  Coordinates are this CTA's own.  Both CTAs
// of a pair describe the same number of steps and bytes; a CTA without rows of its own in a segment gives coordinates
// outside the tensor (TMA then fills with zeros).
struct Segment {
  int mode;                 // OpMode
  int acc;                  // accumulator of the tile this segment adds into
  int nkb;                  // k-blocks (128 bytes of K each: 128 int8 / 64 bf16)
  int bn;                   // UMMA N for this segment (multiple of 16 (CG = 1) or 32 (CG = 2), <= 256)
  int ksteps;               // UMMA k-steps issued per k-block: 4, or fewer (MODE_BF_KM only)
  const CUtensorMap* ta;
  const CUtensorMap* tb;
  int a_x, a_y, a_z;        // K operand: (k0, row0, z);  MN operand: (mn0, k0, z)
  int b_x, b_y, b_z;
  int a_rank, b_rank;       // tensor-map rank (2 or 3)
  int a_blk;                // MN-major A: > 0 = read through a "blocked" tensor map (64-wide column blocks as an extra
                            // dimension, both blocks in one load), else one 64 x 64 box per load
  int b_blk;                // MN-major B: > 0 = blocked map delivering that many blocks in one load; < 0 = -b_blk plain boxes
  int b_bytes;              // bytes of B this CTA loads per k-block (K-major: the box of tb)
};

// Output tiles are P::CG * 128 rows x `bn` columns, the cells of an (mt x nt) grid walked row by row.
struct TileGrid {
  int mt, nt, bn, total;
};
__host__ inline TileGrid make_tile_grid(int mt, int nt, int bn) { return TileGrid{mt, nt, bn, mt * nt}; }
struct TileCoord { int m, n0, bn; };   // m: this CTA's 128-row tile
template <int CG>
__device__ __forceinline__ TileCoord tile_coord(const TileGrid& g, int i, int rank) {
  return TileCoord{(i / g.nt) * CG + rank, (i % g.nt) * g.bn, g.bn};
}

__device__ __forceinline__ bool a_is_mn(int mode) { return mode == MODE_BF_MM; }
__device__ __forceinline__ bool b_is_mn(int mode) { return mode >= MODE_BF_KM; }

template <int CG>
__device__ __forceinline__ void tma_fetch(uint32_t dst, const CUtensorMap* t, uint32_t bar, int rank, int x, int y, int z) {
  if (rank == 3) {
    if (CG == 2) tma_pair_load_3d(dst, t, bar, x, y, z); else tma_load_3d(dst, t, bar, x, y, z);
  } else {
    if (CG == 2) tma_pair_load_2d(dst, t, bar, x, y); else tma_load_2d(dst, t, bar, x, y);
  }
}
// Blocked view of an MN-major operand: dimensions (64 columns of a block, k row, block index[, batch]).
template <int CG>
__device__ __forceinline__ void tma_fetch_blocked(uint32_t dst, const CUtensorMap* t, uint32_t bar, int base_rank, int k, int blk, int z) {
  if (base_rank == 3) {
    if (CG == 2) tma_pair_load_4d(dst, t, bar, 0, k, blk, z); else tma_load_4d(dst, t, bar, 0, k, blk, z);
  } else {
    if (CG == 2) tma_pair_load_3d(dst, t, bar, 0, k, blk); else tma_load_3d(dst, t, bar, 0, k, blk);
  }
}

struct PipeState {
  int stage = 0;
  uint32_t phase = 0;
  __device__ __forceinline__ void advance(int n) {
    if (++stage == n) { stage = 0; phase ^= 1; }
  }
};

// Bounded wait that also gives up when another role of this CTA has failed.
__device__ __forceinline__ bool pipe_wait(uint32_t bar, uint32_t parity, int where, volatile int* abort_flag) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (*abort_flag) return false;
    if (clock64() - t0 > c_spin_cycles) {
      report_timeout(where);
      *abort_flag = 1;
      return false;
    }
  }
  return true;
}

// Coalescing store for epilogues.  Each lane holds PIECES * 16 contiguous bytes of ITS OWN output row, and rows may live
// anywhere in global memory (row_ptr = 0 skips the row).  The warp transposes through its staging buffer (32 rows x
// PIECES * 16 bytes) so that a store instruction writes whole runs of PIECES * 16 contiguous bytes instead of 32 rows x 16
// bytes.  Only the first valid_bytes of each row are written.  The 16-byte piece j of row r sits at position
// j ^ (r & 7) (eight pieces) or j ^ ((r >> 1) & 3) (four), which keeps both passes free of bank conflicts.
template <int PIECES>
__device__ __forceinline__ void warp_store_rows(uint8_t* stage, const uint4 (&v)[PIECES], void* row_ptr, int valid_bytes, int lane) {
  static_assert(PIECES == 8 || PIECES == 4, "row pieces");
  auto spot = [](int r, int j) { return PIECES == 8 ? (j ^ (r & 7)) : (j ^ ((r >> 1) & 3)); };
  uint4* mine = reinterpret_cast<uint4*>(stage + lane * (PIECES * 16));
#pragma unroll
  for (int j = 0; j < PIECES; ++j) mine[spot(lane, j)] = v[j];
  __syncwarp();
  const unsigned long long my = reinterpret_cast<unsigned long long>(row_ptr);
  const int c = lane % PIECES;
#pragma unroll
  for (int i = 0; i < PIECES; ++i) {
    const int row = (32 / PIECES) * i + lane / PIECES;
    const unsigned long long dst = __shfl_sync(0xffffffffu, my, row);
    const uint4 val = *reinterpret_cast<const uint4*>(stage + row * (PIECES * 16) + (spot(row, c) << 4));
    if (dst != 0ull && c * 16 < valid_bytes) *reinterpret_cast<uint4*>(dst + c * 16) = val;
  }
  __syncwarp();
}

// The same wait, where what it guards was written by the other CTA of the pair
__device__ __forceinline__ bool mbar_try_wait_cluster(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool pipe_wait_cluster(uint32_t bar, uint32_t parity, int where, volatile int* abort_flag) {
  if (mbar_try_wait_cluster(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait_cluster(bar, parity)) {
    if (*abort_flag) return false;
    if (clock64() - t0 > c_spin_cycles) {
      report_timeout(where);
      *abort_flag = 1;
      return false;
    }
  }
  return true;
}

// Problems whose epilogue needs nothing fetched ahead of the accumulator
struct NoPre {};

// Widest B operand of a CTA, in rows of 128 bytes (columns of the tile, or half of them for a pair): the ring holds as
// many stages as fit, so a launch of narrow tiles keeps more k-blocks in flight.  Problems without `stage_rows` use
// 256 (CG = 1) or 128 (CG = 2).
template <class P, class = void>
struct stage_rows_of {
  __device__ static int get(const typename P::Params&) { return 256 / P::CG; }
};
template <class P>
struct stage_rows_of<P, std::void_t<decltype(&P::stage_rows)>> {
  __device__ static int get(const typename P::Params& p) { return P::stage_rows(p); }
};

// Accumulators in TMEM.
//   AccDouble : one accumulator per tile, two stages of 256 columns: the epilogue of a tile overlaps the next tile's
//               contraction.
//   AccSplit  : two accumulators of 256 columns per tile (all of TMEM), each with barriers of its own.  The segments of
//               accumulator 1 come first and are short; the epilogue takes accumulator 1 into registers while
//               accumulator 0 is still being computed, so that the next tile's accumulator-1 segments run while the
//               epilogue empties accumulator 0.
struct AccDouble { static constexpr bool kSplit = false; };
struct AccSplit { static constexpr bool kSplit = true; };

// Problems that hand out their tiles by ticket name the counter (cleared before the launch) and may hold a segment back until what
// it reads has been written: `ready`, called by the producers before each, returns false if it gave up.
template <class P, class = void>
struct tickets_of : std::false_type {};
template <class P>
struct tickets_of<P, std::void_t<decltype(&P::tickets)>> : std::true_type {};

template <class P>
__device__ __forceinline__ void gemm_body(const typename P::Params& p) {
  extern __shared__ uint8_t smem_raw[];
  constexpr int CG = P::CG;
  constexpr int kEpiWarps = P::kEpiWarps;
  constexpr bool kSplit = P::Acc::kSplit;
  constexpr bool kTickets = tickets_of<P>::value;
  static_assert(!kTickets || CG == 2, "tickets are handed out by the first CTA of a pair");
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t kStageBytes = kOperandBytes + (uint32_t)stage_rows_of<P>::get(p) * 128u;   // a multiple of 1024
  const int kStages = min(kMaxStages, (int)(kRingBytes / kStageBytes));
  const uint32_t bar_base = smem_base + kRingBytes;
  // barrier block: full[12] empty[12] tfull[2] tempty[2] kfull[4] kempty[4] (8 B each), tile numbers of the tickets [4],
  // tmem ptr, abort flag
  constexpr int kSlots = 4;
  auto full_bar = [&](int s) { return bar_base + 8u * s; };
  auto empty_bar = [&](int s) { return bar_base + 8u * (kMaxStages + s); };
  auto tfull_bar = [&](int s) { return bar_base + 8u * (2 * kMaxStages + s); };
  auto tempty_bar = [&](int s) { return bar_base + 8u * (2 * kMaxStages + 2 + s); };
  auto kfull_bar = [&](int s) { return bar_base + 8u * (2 * kMaxStages + 4 + s); };
  auto kempty_bar = [&](int s) { return bar_base + 8u * (2 * kMaxStages + 4 + kSlots + s); };
  constexpr int kWords = 8 * (2 * kMaxStages + 4 + 2 * kSlots);
  uint8_t* bar_generic = smem_raw + (bar_base - smem_u32(smem_raw));
  volatile int* slots = reinterpret_cast<volatile int*>(bar_generic + kWords);
  volatile uint32_t* tmem_holder = reinterpret_cast<volatile uint32_t*>(bar_generic + kWords + 4 * kSlots);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bar_generic + kWords + 4 * kSlots + 4);
  uint8_t* epi_stage = bar_generic + kBarrierBytes;
  static_assert(kWords + 4 * kSlots + 8 <= kBarrierBytes, "barrier block");

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int rank = CG == 2 ? (int)cluster_rank() : 0;   // which CTA of the pair
  const int group = blockIdx.x / CG, ngroups = gridDim.x / CG;

  if (threadIdx.x == 0) {
    // the operand barriers complete when every CTA's bytes have arrived at the issuing CTA; an accumulator is empty
    // when the epilogue warps of every CTA have read it
    for (int s = 0; s < kStages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(tfull_bar(s), 1); mbar_init(tempty_bar(s), CG * kEpiWarps); }
    // a ticket's slot is free when every reader of both CTAs has it: the epilogue warps, the MMA warp, the second producer
    if (kTickets)
      for (int s = 0; s < kSlots; ++s) { mbar_init(kfull_bar(s), 1); mbar_init(kempty_bar(s), CG * (kEpiWarps + 1)); }
    *abort_flag = 0;
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc<CG>(smem_u32(const_cast<uint32_t*>(tmem_holder)), kTmemCols);
    tmem_relinquish<CG>();
  }
  // Launched with programmatic stream serialisation: the next kernel's CTAs may start (and do their own set-up)
  // while this one's last tiles run; nothing of global memory is touched before the previous kernel has finished.
  pdl_launch_dependents();
  tc_fence_before();
  __syncthreads();
  if (CG == 2) cluster_sync_all();
  tc_fence_after();
  pdl_wait();
  const uint32_t tmem_base = *tmem_holder;
  const int ntiles = P::num_tiles(p);

  // The next tile of a role (`ntiles` or more: none left).  whole: a warp asks, else one lane does.
  auto next_tile = [&](PipeState& ks, int prev, bool whole, int where) -> int {
    if constexpr (!kTickets) return prev < 0 ? group : prev + ngroups;
    else {
      const bool got = pipe_wait_cluster(kfull_bar(ks.stage), ks.phase, where, abort_flag);
      if (whole ? !__all_sync(0xffffffffu, got) : !got) return ntiles;
      const int tile = slots[ks.stage];
      if (whole) __syncwarp();
      if (!whole || lane == 0) mbar_arrive_cluster(cluster_map(kempty_bar(ks.stage), 0));
      ks.advance(kSlots);
      return tile;
    }
  };

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      PipeState st, ks;
      bool ok = true;
      // the first CTA's producer draws the tickets and hands each to every role of both CTAs
      int drawn = 0;
      auto draw = [&] {
        if constexpr (kTickets) { if (rank == 0) drawn = (int)atomicAdd(P::tickets(p), 1u); }
      };
      draw();
      auto next = [&](int prev) -> int {
        if constexpr (kTickets) {
          if (rank == 0) {
            const int tile = drawn;
            if (!pipe_wait_cluster(kempty_bar(ks.stage), ks.phase ^ 1, WHERE_PRODUCER, abort_flag)) return ntiles;
            const uint32_t slot = smem_u32(const_cast<int*>(slots + ks.stage));
            for (int c = 0; c < 2; ++c) {
              asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_map(slot, c)), "r"(tile) : "memory");
              mbar_arrive_cluster(cluster_map(kfull_bar(ks.stage), c));
            }
            ks.advance(kSlots);
            return tile;
          }
        }
        return next_tile(ks, prev, false, WHERE_PRODUCER);
      };
      for (int tile = next(-1); ok && tile < ntiles; tile = next(tile)) {
        typename P::Tile t;
        P::tile_init(p, tile, rank, t);
        const int nseg = P::num_segments(p, t);
        if (nseg == 0) draw();
        for (int s = 0; ok && s < nseg; ++s) {
          if constexpr (kTickets) { if (!P::ready(p, t, s, abort_flag)) { ok = false; break; } }
          Segment sg;
          P::segment(p, t, s, sg);
          // LOADS: how a step's operands come, chosen once per segment -- 0: both K-major, 1: B MN-major through a blocked map,
          // 2: both MN-major through blocked maps, 3: as the segment says.  With these tests inside the loop, a step of a problem
          // whose segments differ (the backward) cost the one issuing lane more than the 512 cycles that its MMAs take: one 256 x 256
          // tile of dW over 8192 and 16384 tokens 60 and 103 us; as it is now 52 and 87 (537 cycles a step).
          auto produce = [&](auto loads, int lo, int hi) {
            constexpr int LOADS = decltype(loads)::value;
            const int a_step = (sg.mode == MODE_I8_KK) ? 128 : 64;
            const uint32_t bytes = CG * (kOperandBytes + sg.b_bytes);
            for (int kb = lo; kb < hi; ++kb) {
              if (!pipe_wait(empty_bar(st.stage), st.phase ^ 1, WHERE_PRODUCER, abort_flag)) { ok = false; break; }
              // the barrier of the issuing CTA counts the bytes of both
              uint32_t bar = full_bar(st.stage);
              if (rank == 0) mbar_expect_tx(bar, bytes);
              if (CG == 2) bar = cluster_map(bar, 0);
              const uint32_t sa = smem_base + st.stage * kStageBytes, sb = sa + kOperandBytes;
              if (LOADS == 2 || (LOADS == 3 && a_is_mn(sg.mode))) {
                if (LOADS == 2 || sg.a_blk > 0) {
                  tma_fetch_blocked<CG>(sa, sg.ta, bar, LOADS == 2 ? 2 : sg.a_rank, sg.a_y + kb * 64, sg.a_x >> 6, sg.a_z);
                } else {
                  tma_fetch<CG>(sa, sg.ta, bar, sg.a_rank, sg.a_x, sg.a_y + kb * 64, sg.a_z);
                  tma_fetch<CG>(sa + kMnBoxBytes, sg.ta, bar, sg.a_rank, sg.a_x + 64, sg.a_y + kb * 64, sg.a_z);
                }
              } else {
                tma_fetch<CG>(sa, sg.ta, bar, sg.a_rank, sg.a_x + kb * a_step, sg.a_y, sg.a_z);
              }
              if (LOADS == 1 || LOADS == 2 || (LOADS == 3 && b_is_mn(sg.mode))) {
                if (LOADS != 3 || sg.b_blk > 0) {
                  tma_fetch_blocked<CG>(sb, sg.tb, bar, sg.b_rank, sg.b_y + kb * 64, sg.b_x >> 6, sg.b_z);
                } else {
                  for (int b = 0; b < -sg.b_blk; ++b)
                    tma_fetch<CG>(sb + b * kMnBoxBytes, sg.tb, bar, sg.b_rank, sg.b_x + 64 * b, sg.b_y + kb * 64, sg.b_z);
                }
              } else {
                tma_fetch<CG>(sb, sg.tb, bar, sg.b_rank, sg.b_x + kb * a_step, sg.b_y, sg.b_z);
              }
              st.advance(kStages);
            }
          };
          // The next ticket is drawn as late as its trip to memory allows, a ring's worth of steps before the end of the tile: drawn
          // with this one, it would keep a tile from a free pair for as long as this one lasts.  1024 x 1024 over 4096 tokens, sixteen long
          // tiles and 64 short ones: backward 43.6 -> 35.6 us.  What the ring holds whole draws with its first step: drawn in the last quarter, two steps
          // at least, training steps of 200 and 300 tokens, 4096 -> 4096, took 193.8 and 149.7 us instead of 190.9 and 148.2, others from
          // 1.7 % less (448, 2048 -> 2048, eight experts) to 0.8 % more (640, 2048 -> 2048, four).
          for (int lo = 0, hi; ok && lo < sg.nkb; lo = hi) {
            hi = kTickets && s + 1 == nseg && lo < sg.nkb - kStages ? sg.nkb - kStages : sg.nkb;
            if (s + 1 == nseg && hi == sg.nkb) draw();
            if (sg.mode <= MODE_BF_KK) produce(std::integral_constant<int, 0>{}, lo, hi);
            else if (sg.mode == MODE_BF_KM && sg.b_blk > 0) produce(std::integral_constant<int, 1>{}, lo, hi);
            else if (sg.mode == MODE_BF_MM && sg.a_blk > 0 && sg.b_blk > 0 && sg.a_rank == 2) produce(std::integral_constant<int, 2>{}, lo, hi);
            else produce(std::integral_constant<int, 3>{}, lo, hi);
          }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (first CTA of the pair)
    // The whole warp walks the loops, one elected thread issues.  What a tcgen05.mma costs to issue decides the rate: with
    // the descriptors put together per instruction in 64-bit arithmetic, the operand form tested inside the loop and a loop
    // over the k-steps the kernels ran at 190-230 cycles per MMA whatever the operands did (8192^3 int8: 2.7 POP/s with the
    // loads taken out); with the loop below, unrolled and specialised on the operand form, at the 128 cycles of the tensor
    // pipe (4.5 POP/s int8, 2.2 PFLOP/s bf16, loads taken out).
    if (rank == 0) {
      PipeState st, ac, ks;
      bool ok = true;
      auto all_wait = [&](uint32_t bar, uint32_t parity) {
        const bool got = __all_sync(0xffffffffu, pipe_wait(bar, parity, WHERE_MMA, abort_flag));
        tc_fence_after();
        return got;
      };
      auto commit = [&](uint32_t bar) { if (elect_one()) umma_commit<CG>(bar); };
      for (int tile = next_tile(ks, -1, true, WHERE_MMA); ok && tile < ntiles; tile = next_tile(ks, tile, true, WHERE_MMA)) {
        typename P::Tile t;
        P::tile_init(p, tile, rank, t);
        const int nseg = P::num_segments(p, t);
        if (!kSplit && !all_wait(tempty_bar(ac.stage), ac.phase ^ 1)) { ok = false; break; }
        int open = -1;                   // accumulator whose segments are being issued
        for (int s = 0; ok && s < nseg; ++s) {
          Segment sg;
          P::segment(p, t, s, sg);
          uint32_t started = open == sg.acc;
          if (!started) {
            if (kSplit) {
              if (open >= 0) commit(tfull_bar(open));
              if (!all_wait(tempty_bar(sg.acc), ac.phase ^ 1)) { ok = false; break; }
            }
            open = sg.acc;
          }
          const uint32_t d_tmem = tmem_base + (kSplit ? sg.acc : ac.stage) * kAccCols;
          // OP: operand form, STEPS: k-steps per k-block (0: as the segment says)
          auto contract = [&](auto op, auto steps) {
            constexpr int OP = decltype(op)::value, STEPS = decltype(steps)::value;
            constexpr bool amn = OP == MODE_BF_MM, bmn = OP >= MODE_BF_KM;
            constexpr uint32_t astep = amn ? 2048 >> 4 : 32 >> 4, bstep = bmn ? 2048 >> 4 : 32 >> 4;
            const uint32_t idesc = OP == MODE_I8_KK ? umma_idesc(2, 1, 0, 0, sg.bn, CG * 128)
                                                    : umma_idesc(1, 1, amn ? 1 : 0, bmn ? 1 : 0, sg.bn, CG * 128);
            const uint64_t a0 = umma_smem_desc(smem_base, amn ? kMnBoxBytes : 16, 1024);
            const uint64_t b0 = umma_smem_desc(smem_base + kOperandBytes, bmn ? kMnBoxBytes : 16, 1024);
            const uint32_t ahi = (uint32_t)(a0 >> 32), bhi = (uint32_t)(b0 >> 32);
            for (int kb = 0; kb < sg.nkb; ++kb) {
              if (!all_wait(full_bar(st.stage), st.phase)) { ok = false; break; }
              const uint32_t off = (st.stage * kStageBytes) >> 4;   // addresses stay below 2^18: no carry out of the field
              const uint32_t alo = (uint32_t)a0 + off, blo = (uint32_t)b0 + off;
              auto step = [&](int k) {
                const uint64_t ad = ((uint64_t)ahi << 32) | (alo + k * astep), bd = ((uint64_t)bhi << 32) | (blo + k * bstep);
                if (OP == MODE_I8_KK) umma_i8<CG>(d_tmem, ad, bd, idesc, k ? 1u : started);
                else umma_f16<CG>(d_tmem, ad, bd, idesc, k ? 1u : started);
              };
              if (elect_one()) {
                if (STEPS > 0) {
#pragma unroll
                  for (int k = 0; k < STEPS; ++k) step(k);
                } else {
                  for (int k = 0; k < sg.ksteps; ++k) step(k);
                }
                umma_commit<CG>(empty_bar(st.stage));  // frees the smem stage (of both CTAs) once these MMAs retire
              }
              started = 1u;
              st.advance(kStages);
            }
          };
          if (sg.ksteps != 4) contract(std::integral_constant<int, MODE_BF_KM>{}, std::integral_constant<int, 0>{});   // the router's one step
          else if (sg.mode == MODE_I8_KK) contract(std::integral_constant<int, MODE_I8_KK>{}, std::integral_constant<int, 4>{});
          else if (sg.mode == MODE_BF_KK) contract(std::integral_constant<int, MODE_BF_KK>{}, std::integral_constant<int, 4>{});
          else if (sg.mode == MODE_BF_KM) contract(std::integral_constant<int, MODE_BF_KM>{}, std::integral_constant<int, 4>{});
          else contract(std::integral_constant<int, MODE_BF_MM>{}, std::integral_constant<int, 4>{});
        }
        if (ok) commit(tfull_bar(kSplit ? 0 : ac.stage));
        if (kSplit) ac.phase ^= 1;
        else ac.advance(2);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue warps
    PipeState ac, ks;
    const int quad = warp & 3;          // TMEM lanes [32*quad, 32*quad+32) are this warp's
    const int part = (warp - 2) >> 2;   // which of the quadrant's warps: it takes column chunks part, part + kEpiWarps / 4, ...
    uint8_t* stage = epi_stage + (warp - 2) * (kStagingBytes / kEpiWarps);
    const uint32_t tlane = tmem_base + (static_cast<uint32_t>(quad * 32) << 16);
    const uint32_t tempty0 = CG == 2 ? cluster_map(tempty_bar(0), 0) : tempty_bar(0);   // at the issuing CTA
    auto release = [&](int a) {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (CG == 2) mbar_arrive_cluster(tempty0 + 8u * a);
        else mbar_arrive(tempty0 + 8u * a);
      }
    };
    // Every lane watches the barrier itself, but the warp takes ONE decision: what follows is full of
    // warp-collective instructions (tcgen05.ld, shuffles), so a lane that gave up must take the others along.
    auto await = [&](int a, uint32_t phase) {
      const bool got = __all_sync(0xffffffffu, pipe_wait(tfull_bar(a), phase, WHERE_EPILOGUE, abort_flag));
      tc_fence_after();
      return got;
    };
    for (int tile = next_tile(ks, -1, true, WHERE_EPILOGUE); tile < ntiles; tile = next_tile(ks, tile, true, WHERE_EPILOGUE)) {
      typename P::Tile t;
      P::tile_init(p, tile, rank, t);
      // per-row factors and addresses are fetched while the contraction is still running
      const typename P::Pre pre = P::prepare(p, t, quad, lane);
      if constexpr (kSplit) {
        typename P::Regs regs;
        if (!await(1, ac.phase)) break;
        P::take_first(p, t, pre, tlane + kAccCols, part, regs);
        release(1);
        P::scale_first(p, t, pre, part, regs);
        if (!await(0, ac.phase)) break;
        P::combine(p, t, pre, tlane, part, regs);
        release(0);
        P::store(p, t, pre, part, lane, stage, regs);
        ac.phase ^= 1;
      } else {
        if (!await(ac.stage, ac.phase)) break;
        P::epilogue(p, t, pre, tlane + ac.stage * kAccCols, quad, part, lane, stage);
        release(ac.stage);
        ac.advance(2);
      }
    }
  }

  __syncthreads();
  if (*abort_flag) {
    // a wait ran out: give copies and MMAs already in flight time to land before the
    // shared memory and TMEM of this CTA are released
    for (int i = 0; i < 200; ++i) __nanosleep(1000);
  }
  __syncthreads();
  if (CG == 2) cluster_sync_all();   // neither CTA leaves while the other may still signal its barriers or read its operands
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc<CG>(tmem_base, kTmemCols);
  }
}

// One named kernel per problem, so that profiler listings show which product ran.
template <class P>
constexpr int gemm_threads = 64 + 32 * P::kEpiWarps;
#define PQ_DEFINE_GEMM_KERNEL(name, Problem)                                                                           \
  __global__ void __cluster_dims__(Problem::CG, 1, 1) __launch_bounds__(gemm_threads<Problem>, 1)                       \
      name(const __grid_constant__ typename Problem::Params p) {                                                       \
    gemm_body<Problem>(p);                                                                                             \
  }

}  // namespace pq
