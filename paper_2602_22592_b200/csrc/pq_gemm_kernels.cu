// Tensor-core kernels of the pQuant layer, built on the engine in pq_gemm.cuh:
//   forward  : H = X A_e^T (grouped by expert), then the fused output tile
//              Y = alpha g (H B_e^T) + beta (lam/gamma) (q S^T)      (Eq. 10, 11)
//   backward : dH, dX, dW, dB, dA of the straight-through estimator  (App. B.1)
//   debug    : raw accumulators of one contraction, for bit-exact tests
#include <algorithm>
#include <type_traits>

#include "pq_gemm.cuh"
#include "pq_kernels.cuh"

namespace pq {

// ---------------------------------------------------------------------------
// tensor maps
// ---------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = []() -> EncodeTiledFn {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess) return nullptr;
    if (q != cudaDriverEntryPointSuccess) return nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

// Row-major tensor of `rank` dims (dims[0] innermost), 128-byte swizzle, zero fill outside.
// box[0] * elem_bytes must be 128.  Returns false on any violated precondition.
static bool make_map(CUtensorMap* m, bool is_i8, const void* base, int rank, const uint64_t* dims, const uint64_t* strides_bytes,
                     const uint32_t* box) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const int eb = is_i8 ? 1 : 2;
  if ((reinterpret_cast<uintptr_t>(base) & 15) != 0) return false;
  if (box[0] * eb != 128) return false;
  cuuint64_t gd[4];
  cuuint64_t gs[3];
  cuuint32_t bx[4], es[4];
  for (int i = 0; i < rank; ++i) {
    gd[i] = dims[i];
    bx[i] = box[i];
    es[i] = 1;
    if (box[i] > 256 || dims[i] == 0) return false;
  }
  for (int i = 0; i + 1 < rank; ++i) {
    gs[i] = strides_bytes[i];
    if (gs[i] % 16) return false;
  }
  CUresult r = fn(m, is_i8 ? CU_TENSOR_MAP_DATA_TYPE_UINT8 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), gd,
                  gs, bx, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

static bool map2d(CUtensorMap* m, bool is_i8, const void* base, uint64_t inner, uint64_t outer, uint32_t box_inner, uint32_t box_outer) {
  const uint64_t dims[2] = {inner, outer};
  const uint64_t strides[1] = {inner * (is_i8 ? 1 : 2)};
  const uint32_t box[2] = {box_inner, box_outer};
  return make_map(m, is_i8, base, 2, dims, strides, box);
}
static bool map3d(CUtensorMap* m, const void* base, uint64_t inner, uint64_t mid, uint64_t outer, uint32_t box_inner, uint32_t box_mid) {
  const uint64_t dims[3] = {inner, mid, outer};
  const uint64_t strides[2] = {inner * 2, inner * mid * 2};
  const uint32_t box[3] = {box_inner, box_mid, 1};
  return make_map(m, false, base, 3, dims, strides, box);
}

// int8 [outer][mid][inner] with the contraction index innermost: boxes of 128 bytes x box_mid rows of one batch entry;
// `pitch` is the row stride in bytes (a multiple of 16, at least `inner`)
static bool map3d_i8(CUtensorMap* m, const void* base, uint64_t inner, uint64_t pitch, uint64_t mid, uint64_t outer, uint32_t box_mid) {
  const uint64_t dims[3] = {inner, mid, outer};
  const uint64_t strides[2] = {pitch, pitch * mid};
  const uint32_t box[3] = {128, box_mid, 1};
  return make_map(m, true, base, 3, dims, strides, box);
}

// MN-major operand: matrix [batch][k_total][mn_total] with mn contiguous, read in 64 (mn) x 64 (k) boxes.
// When mn_total is a multiple of 64 the map views the 64-wide column blocks as a dimension of their own,
// (64, k_total, mn_total / 64[, batch]) -- base_rank 2 or 3 says whether the operand has the batch dimension --, so that ONE load delivers `nblk` boxes back to back; *blk = nblk.
// Otherwise (a narrower last block would alias the next row) a plain map with one box per load; *blk = -nblk.
static bool map_mn(CUtensorMap* m, int* blk, const void* base, uint64_t mn_total, uint64_t k_total, int base_rank, uint64_t batch, int nblk) {
  if (mn_total % 64 == 0) {
    *blk = nblk;
    const uint64_t dims[4] = {64, k_total, mn_total / 64, batch};
    const uint64_t strides[3] = {mn_total * 2, 128, mn_total * k_total * 2};
    const uint32_t box[4] = {64, 64, (uint32_t)nblk, 1};
    return make_map(m, false, base, base_rank + 1, dims, strides, box);
  }
  *blk = -nblk;
  return base_rank == 3 ? map3d(m, base, mn_total, k_total, batch, 64, 64) : map2d(m, false, base, mn_total, k_total, 64, 64);
}

// max_tiles: tiles of the launch, at most; one CTA (or CTA pair) each, as many as the SMs hold
template <class P>
static int launch_gemm(int kernel_id, void (*kernel)(typename P::Params), const typename P::Params& p, int max_tiles, cudaStream_t st) {
  // (cudaFuncSetAttribute is cheap and idempotent; calling it per launch keeps this free of static state per kernel)
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGemmSmemBytes) != cudaSuccess) return PQ_ERR_CUDA;
  const int grid = P::CG * std::max(1, std::min(max_tiles, sm_count() / P::CG));
  LaunchScope ls(kernel_id, st);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid, 1, 1); cfg.blockDim = dim3(gemm_threads<P>, 1, 1); cfg.dynamicSmemBytes = kGemmSmemBytes;
  cfg.stream = st; cfg.attrs = attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, p) == cudaSuccess ? PQ_OK : PQ_ERR_CUDA;
}

__device__ __forceinline__ int round_up(int x, int m) { return (x + m - 1) / m * m; }
// width actually contracted for a tile that starts at n0: the tile's width, cut at the matrix edge
__device__ __forceinline__ int clip_bn(int bn, int n0, int n_total, int granule) {
  const int left = round_up(n_total - n0, granule);
  return left < bn ? (left > 0 ? left : granule) : bn;
}

// Intermediates that feed a second tensor-core product (H, g H, dH / c) are kept
// as TWO bf16 planes, v ~= hi + lo with hi = bf16(v), lo = bf16(v - hi): about 16
// significand bits, so their rounding does not show in the results.  The planes
// are stacked along the row axis ([2][item_rows][r]); a product against such an
// operand simply runs its contraction over both planes.
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo) {
  hi = pack_bf16x2(a, b);
  lo = pack_bf16x2(a - bf16lo(hi), b - bf16hi(hi));
}
static inline int h_round_up(int x, int m) { return (x + m - 1) / m * m; }

// ---------------------------------------------------------------------------
// debug: D[M,N] = contraction of A and B in one of the four operand forms
// ---------------------------------------------------------------------------
template <int CG_>
struct DebugProblem {
  static constexpr int CG = CG_, kEpiWarps = 8;
  using Acc = AccDouble;
  struct Params {
    CUtensorMap ta, tb;
    TileGrid g;
    int mode, M, N, K, a_blk, b_blk, b_bytes;
    void* D;
  };
  struct Tile { TileCoord c; int rank; };
  __device__ static int num_tiles(const Params& p) { return p.g.total; }
  __device__ static void tile_init(const Params& p, int i, int rank, Tile& t) { t.c = tile_coord<CG>(p.g, i, rank); t.rank = rank; }
  __device__ static int num_segments(const Params&, const Tile&) { return 1; }
  __device__ static void segment(const Params& p, const Tile& t, int, Segment& s) {
    s.mode = p.mode; s.acc = 0; s.ksteps = 4; s.a_blk = p.a_blk; s.b_blk = p.b_blk; s.b_bytes = p.b_bytes;
    s.bn = clip_bn(t.c.bn, t.c.n0, p.N, p.mode >= MODE_BF_KM ? 64 * CG : 32);
    const int bk = p.mode == MODE_I8_KK ? 128 : 64;
    s.nkb = (p.K + bk - 1) / bk;
    s.ta = &p.ta; s.tb = &p.tb; s.a_rank = 2; s.b_rank = 2; s.a_z = 0; s.b_z = 0;
    const int n0 = t.c.n0 + t.rank * (s.bn / CG);
    if (p.mode == MODE_BF_MM) { s.a_x = t.c.m * 128; s.a_y = 0; } else { s.a_x = 0; s.a_y = t.c.m * 128; }
    if (p.mode >= MODE_BF_KM) { s.b_x = n0; s.b_y = 0; } else { s.b_x = 0; s.b_y = n0; }
  }
  using Pre = NoPre;
  __device__ static Pre prepare(const Params&, const Tile&, int, int) { return Pre{}; }
  __device__ static void epilogue(const Params& p, const Tile& t, const Pre& pre, uint32_t tacc, int quad, int part, int lane, uint8_t* stage) {
    const int row = t.c.m * 128 + quad * 32 + lane;
    uint32_t* D = reinterpret_cast<uint32_t*>(p.D);
    for (int c = part; c * 32 < t.c.bn; c += kEpiWarps / 4) {
      const int n0 = t.c.n0 + c * 32;
      if (n0 >= p.N) break;
      uint32_t v[32];
      tmem_ld32(tacc + c * 32, v);
      tmem_ld_wait();
      uint4 o[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) o[j] = make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
      const int valid = min(32, p.N - n0) * 4;   // N is a multiple of 8 -> whole 16-byte pieces
      warp_store_rows<8>(stage, o, row < p.M ? D + (long long)row * p.N + n0 : nullptr, valid, lane);
    }
  }
};
PQ_DEFINE_GEMM_KERNEL(k_gemm_debug, DebugProblem<2>)
PQ_DEFINE_GEMM_KERNEL(k_gemm_debug_single, DebugProblem<1>)

template <class P>
static int run_debug(void (*kernel)(typename P::Params), int mode, int M, int N, int K, const void* A, const void* B, void* D, int tile_n, cudaStream_t st) {
  typename P::Params p;
  p.mode = mode; p.M = M; p.N = N; p.K = K; p.D = D; p.a_blk = 0; p.b_blk = 0;
  const int share = tile_n / P::CG;                  // columns of a tile that one CTA loads
  p.b_bytes = share * 128;
  p.g = make_tile_grid((M + 128 * P::CG - 1) / (128 * P::CG), (N + tile_n - 1) / tile_n, tile_n);
  bool ok = true;
  switch (mode) {
    case MODE_I8_KK:
      ok = map2d(&p.ta, true, A, K, M, 128, 128) && map2d(&p.tb, true, B, K, N, 128, share);
      break;
    case MODE_BF_KK:
      ok = map2d(&p.ta, false, A, K, M, 64, 128) && map2d(&p.tb, false, B, K, N, 64, share);
      break;
    case MODE_BF_KM:
      ok = map2d(&p.ta, false, A, K, M, 64, 128) && map_mn(&p.tb, &p.b_blk, B, N, K, 2, 1, share / 64);
      break;
    case MODE_BF_MM:
      ok = map_mn(&p.ta, &p.a_blk, A, M, K, 2, 1, 2) && map_mn(&p.tb, &p.b_blk, B, N, K, 2, 1, share / 64);
      break;
    default:
      return PQ_ERR_UNSUPPORTED;
  }
  if (!ok) return PQ_ERR_CUDA;
  return launch_gemm<P>(KID_DEBUG, kernel, p, p.g.total, st);
}

int gemm_debug(int mode, int M, int N, int K, const void* A, const void* B, void* D, int tile_n, cudaStream_t st) {
  const int granule = mode >= MODE_BF_KM ? 64 : 32;
  if (tile_n <= 0) tile_n = 256;
  if (tile_n > 256 || tile_n % granule) return PQ_ERR_SHAPE;
  // a pair's CTA loads whole 64-column boxes of an MN-major operand; widths that do not split that way run on one CTA
  if (granule == 64 && tile_n % 128) return run_debug<DebugProblem<1>>(k_gemm_debug_single, mode, M, N, K, A, B, D, tile_n, st);
  return run_debug<DebugProblem<2>>(k_gemm_debug, mode, M, N, K, A, B, D, tile_n, st);
}

// ---------------------------------------------------------------------------
// F1: hidden activations of the HP branch, H = X_sorted A_e^T, one tile per item
// ---------------------------------------------------------------------------
struct HpUpProblem {
  static constexpr int CG = 1, kEpiWarps = 8;
  using Acc = AccDouble;
  struct Params {
    CUtensorMap tx, ta;  // X sorted [T,K]; A [E,r,K]
    RoutingTables rt;
    uint16_t* H;
    int K, r, bn, item_rows;
  };
  struct Tile { int item; int4 it; };
  __device__ static int stage_rows(const Params& p) { return p.bn <= 128 ? 128 : 256; }
  __device__ static int num_tiles(const Params& p) { return p.rt.n_items[0]; }
  __device__ static void tile_init(const Params& p, int i, int, Tile& t) { t.item = i; t.it = p.rt.items[i]; }
  __device__ static int num_segments(const Params&, const Tile&) { return 1; }
  __device__ static void segment(const Params& p, const Tile& t, int, Segment& s) {
    s.mode = MODE_BF_KK; s.acc = 0; s.bn = p.bn; s.ksteps = 4; s.nkb = (p.K + 63) / 64;
    s.ta = &p.tx; s.a_rank = 2; s.a_x = 0; s.a_y = t.it.x * 128; s.a_z = 0;
    s.tb = &p.ta; s.b_rank = 3; s.b_x = 0; s.b_y = 0; s.b_z = t.it.y;
    s.b_bytes = p.bn * 128; s.a_blk = 0; s.b_blk = 0;
  }
  using Pre = NoPre;
  __device__ static Pre prepare(const Params&, const Tile&, int, int) { return Pre{}; }
  __device__ static void epilogue(const Params& p, const Tile& t, const Pre& pre, uint32_t taddr, int quad, int half, int lane, uint8_t* stage) {
    const int row = quad * 32 + lane;
    const bool live = row >= t.it.z && row < t.it.w;
    uint4* out_hi = reinterpret_cast<uint4*>(p.H + ((long long)t.item * 128 + row) * p.r);
    uint4* out_lo = reinterpret_cast<uint4*>(p.H + ((long long)p.item_rows + t.item * 128 + row) * p.r);
    for (int c = half; c * 32 < p.r; c += 2) {
      uint32_t v[32];
      tmem_ld32(taddr + c * 32, v);
      tmem_ld_wait();
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        if (c * 32 + g * 8 < p.r) {
          uint32_t hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};
          if (live) {
#pragma unroll
            for (int j = 0; j < 4; ++j) split2(__uint_as_float(v[8 * g + 2 * j]), __uint_as_float(v[8 * g + 2 * j + 1]), hi[j], lo[j]);
          }
          out_hi[c * 4 + g] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
          out_lo[c * 4 + g] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
      }
    }
  }
};

PQ_DEFINE_GEMM_KERNEL(k_gemm_hp_up, HpUpProblem)

// ---------------------------------------------------------------------------
// F1 in INT8 (Sec. 3.2): h_int = q_sorted A8_e^T, exact in int32, one tile per item; the epilogue quantises each
// row of h per token the way activations are (Eq. 7-9, taken from the integers: gamma_h = 128 / max |h_int|) and
// writes the codes qh [items*128, rp] (row pitch rp = r rounded up to 16, padding zero) and gamma_h [items*128].
// ---------------------------------------------------------------------------
struct HpUp8Problem {
  static constexpr int CG = 1, kEpiWarps = 8;
  using Acc = AccDouble;
  struct Params {
    CUtensorMap tq, ta, tb;  // q sorted [T,K] s8; A8 [E,r,K] s8, twice
    RoutingTables rt;
    int8_t* qh;
    float* gamma_h;
    int* raw;            // not null: write the exact sums h_int [items*128, r] instead of codes (the caller quantises later)
    int* rawb;           // sums of the second matrix (an FFN's gate and up projections in one launch), or null
    int K, r, rp, bn;
  };
  struct Tile { int item, second; int4 it; };
  __device__ static int stage_rows(const Params& p) { return p.bn <= 128 ? 128 : 256; }
  __device__ static int num_tiles(const Params& p) { return p.rt.n_items[0] * (p.rawb ? 2 : 1); }
  __device__ static void tile_init(const Params& p, int i, int, Tile& t) {
    const int n = p.rt.n_items[0];
    t.second = i >= n; t.item = t.second ? i - n : i; t.it = p.rt.items[t.item];
  }
  __device__ static int num_segments(const Params&, const Tile&) { return 1; }
  __device__ static void segment(const Params& p, const Tile& t, int, Segment& s) {
    s.mode = MODE_I8_KK; s.acc = 0; s.bn = p.bn; s.ksteps = 4; s.nkb = (p.K + 127) / 128;
    s.ta = &p.tq; s.a_rank = 2; s.a_x = 0; s.a_y = t.it.x * 128; s.a_z = 0;
    s.tb = t.second ? &p.tb : &p.ta; s.b_rank = 3; s.b_x = 0; s.b_y = 0; s.b_z = t.it.y;
    s.b_bytes = p.bn * 128; s.a_blk = 0; s.b_blk = 0;
  }
  using Pre = NoPre;
  __device__ static Pre prepare(const Params&, const Tile&, int, int) { return Pre{}; }
  __device__ static void epilogue(const Params& p, const Tile& t, const Pre& pre, uint32_t taddr, int quad, int half, int lane, uint8_t* stage) {
    if (p.raw) {
      int* out = (t.second ? p.rawb : p.raw) + ((long long)t.item * 128 + quad * 32 + lane) * p.r;
      for (int c = half; c * 32 < p.r; c += 2) {
        uint32_t v[32];
        tmem_ld32(taddr + c * 32, v);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (c * 32 + 4 * j < p.r) reinterpret_cast<uint4*>(out + c * 32)[j] = make_uint4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
      }
      return;
    }
    if (half) return;   // the maximum over a row's r columns stays in one thread
    const int row = quad * 32 + lane;
    const bool live = row >= t.it.z && row < t.it.w;
    int amax = 0;
    for (int c = 0; c * 32 < p.r; ++c) {
      uint32_t v[32];
      tmem_ld32(taddr + c * 32, v);
      tmem_ld_wait();
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (c * 32 + j < p.r) amax = max(amax, abs((int)v[j]));
    }
    const float gamma_h = __fdiv_rn(kActQmax, fmaxf(__int2float_rn(amax), kActAmaxFloor));
    const long long grow = (long long)t.item * 128 + row;
    p.gamma_h[grow] = live ? gamma_h : 0.f;
    uint4* out = reinterpret_cast<uint4*>(p.qh + grow * p.rp);
    for (int c = 0; c * 32 < p.rp; ++c) {
      uint32_t v[32];
      tmem_ld32(taddr + c * 32, v);
      tmem_ld_wait();
      uint32_t w[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        uint32_t word = 0u;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int col = c * 32 + 4 * j + b;
          int code = 0;
          if (live && col < p.r) code = max(-128, min(127, __float2int_rn(__fmul_rn(__int2float_rn((int)v[4 * j + b]), gamma_h))));
          word |= (uint32_t)(code & 0xFF) << (8 * b);
        }
        w[j] = word;
      }
      if (c * 32 < p.rp) out[2 * c] = make_uint4(w[0], w[1], w[2], w[3]);
      if (c * 32 + 16 < p.rp) out[2 * c + 1] = make_uint4(w[4], w[5], w[6], w[7]);
    }
  }
};
PQ_DEFINE_GEMM_KERNEL(k_gemm_hp_up8, HpUp8Problem)

// ---------------------------------------------------------------------------
// F2: fused output tile.  Accumulator 0 (int32): q S^T over K.  Accumulator 1
// (fp32): H B_e^T over r, once per item of the tile (masked H rows are zero).
// Epilogue: Y[token, n] = alpha_n g z + beta_n (lam / gamma) acc, rounded once.
// ---------------------------------------------------------------------------
// GEN = false: scalar feature scales and K < 32768; GEN = true: anything (the extra addresses and branches cost registers the
// common form does not have to spare).
// CG_: a pair of CTAs per 256 rows, or one CTA per 128 (see gemm_forward).
template <bool HP, bool GEN, int CG_>
struct FwdProblem {
  // With the HP branch a tile holds an int32 and an fp32 accumulator of 256 columns each, all of TMEM.  Sixteen epilogue
  // warps, 64 columns of a row per thread: the fp32 accumulator waits in 64 registers while the int8 contraction runs, and
  // what the next tile's int8 contraction has to wait for is only the read of the int32 accumulator, which the next tile's
  // HP segments cover.
  static constexpr int CG = CG_, kEpiWarps = HP ? 16 : 8;
  using Acc = typename std::conditional<HP, AccSplit, AccDouble>::type;
  struct Params {
    CUtensorMap tq, ts, ts2, th, tb;  // q [T,K] s8; S [N,K] s8, of a second matrix too; H [items*128,r]; B [E,N,r]
    RoutingTables rt;
    TileGrid g;
    const int* perm;
    const float* gamma;
    const float* gate;
    const float* w_scales;
    const float* alpha;
    const float* beta;
    uint16_t* Y;
    // INT8 HP branch (Sec. 3.2): th / tb then map the int8 codes of h and of B_e, the second accumulator is int32, and
    // its de-quantisation factor 1 / (gamma_B gamma_h gamma_A gamma_t) is folded into the row's HP factor
    const float* gamma_h;    // [items*128], null for the bf16 branch
    const float* hp_scales;  // [E][2] = {gamma_A, gamma_B}
    int hp_ext;              // the codes of h and gamma_h were written by the caller
    // without an HP branch: a second matrix of the same sizes, whose column tiles follow those of the first (`tiles1` of them)
    const float* w_scales2;
    uint16_t* Y2;
    int T, N, K, r, sstride, item_rows, tiles1;
  };
  struct Tile { TileCoord c; int bn, pb, pe, rank, second; };
  __device__ static int num_tiles(const Params& p) { return p.g.total; }
  __device__ static void tile_init(const Params& p, int i, int rank, Tile& t) {
    t.c = tile_coord<CG>(p.g, i, rank);
    t.rank = rank;
    t.second = !HP && t.c.n0 >= p.tiles1 * p.g.bn;
    if (t.second) t.c.n0 -= p.tiles1 * p.g.bn;
    t.bn = clip_bn(t.c.bn, t.c.n0, p.N, 32);
    const int* begin = CG == 2 ? p.rt.pair_begin : p.rt.tile_item_begin;   // entries of the pair of row tiles, or items of the row tile
    if (HP) { t.pb = begin[t.c.m / CG]; t.pe = begin[t.c.m / CG + 1]; } else { t.pb = t.pe = 0; }
  }
  // The HP product uses the leading bf16 plane of H only: its 2^-9 relative rounding is of the size of the
  // output's own rounding to bf16; the second plane serves the backward pass, whose sums are longer.
  __device__ static int num_segments(const Params&, const Tile& t) { return (t.pe - t.pb) + 1; }
  __device__ static void segment(const Params& p, const Tile& t, int i, Segment& s) {
    s.bn = t.bn; s.ksteps = 4; s.a_z = 0; s.b_z = 0; s.a_blk = 0; s.b_blk = 0; s.b_bytes = kOperandBytes * (2 / CG);
    s.b_x = 0; s.b_y = t.c.n0 + t.rank * (t.bn / CG);
    if (i == t.pe - t.pb) {
      s.mode = MODE_I8_KK; s.acc = 0; s.nkb = (p.K + 127) / 128;
      s.ta = &p.tq; s.a_rank = 2; s.a_x = 0; s.a_y = t.c.m * 128;
      s.tb = t.second ? &p.ts2 : &p.ts; s.b_rank = 2;
    } else {
      int item, expert;
      if (CG == 2) {
        const int4 pi = p.rt.pair_items[t.pb + i];
        item = t.rank ? pi.z : pi.y; expert = pi.x;
      } else {
        item = t.pb + i; expert = p.rt.items[item].y;
      }
      if (p.gamma_h) { s.mode = MODE_I8_KK; s.nkb = (p.r + 127) / 128; }
      else { s.mode = MODE_BF_KK; s.nkb = (p.r + 63) / 64; }
      s.acc = 1;
      s.ta = &p.th; s.a_rank = p.gamma_h ? 3 : 2; s.a_x = 0;
      s.a_y = item >= 0 ? item * 128 : 2 * p.item_rows;    // no rows of this expert here: beyond both planes of H, read as zeros
      s.tb = &p.tb; s.b_rank = 3; s.b_z = expert;
    }
  }
  // float of an accumulator of the 1-bit product, exactly.  |acc| <= 128 K: below K = 32768 the integer fits the mantissa of
  // 1.5 * 2^23, so that an integer add and a float subtract do what the slower conversion instruction does.
  __device__ static __forceinline__ float acc_float(uint32_t a) {
    return GEN ? (float)(int)a : __int_as_float((int)a + 0x4B400000) - 12582912.0f;
  }
  // y = beta_n cb * acc + z for 16 consecutive columns starting at n (z: the HP term, factors applied), as 8 bf16 pairs
  __device__ static __forceinline__ void combine16(const Params& p, int n, float cb, const uint32_t (&a)[16], const uint32_t* z, uint32_t* w) {
#pragma unroll
    for (int q4 = 0; q4 < 4; ++q4) {
      float b4[4] = {cb, cb, cb, cb};
      if (GEN && p.sstride) {
        const float4 bv = __ldg(reinterpret_cast<const float4*>(p.beta + n) + q4);
        b4[0] *= bv.x; b4[1] *= bv.y; b4[2] *= bv.z; b4[3] *= bv.w;
      }
      float y[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float f = acc_float(a[4 * q4 + u]);
        y[u] = HP ? fmaf(b4[u], f, __uint_as_float(z[4 * q4 + u])) : b4[u] * f;
      }
      w[2 * q4] = pack_bf16x2(y[0], y[1]);
      w[2 * q4 + 1] = pack_bf16x2(y[2], y[3]);
    }
  }
  // per-row factors: 1-bit branch lam / gamma_t (Eq. 10), HP branch g_t; scalar feature scales folded in
  struct Pre { uint16_t* yrow; float cb, ca; };
  __device__ static Pre prepare(const Params& p, const Tile& t, int quad, int lane) {
    const int pos = t.c.m * 128 + quad * 32 + lane;
    Pre r{nullptr, 0.f, 0.f};
    if (pos < p.T) {
      const int token = p.perm ? p.perm[pos] : pos;
      r.yrow = (t.second ? p.Y2 : p.Y) + (long long)token * p.N;
      r.cb = __fdiv_rn((t.second ? p.w_scales2 : p.w_scales)[0], p.gamma[pos]);
      if (HP) r.ca = p.gate[pos];
      if (HP && p.gamma_h) {
        // the item of this row: its expert's weight scales and the row's own hidden scale
        const int rel = quad * 32 + lane;
        float deq = 0.f;
        for (int it = p.rt.tile_item_begin[t.c.m]; it < p.rt.tile_item_begin[t.c.m + 1]; ++it) {
          const int4 d = p.rt.items[it];
          if (rel >= d.z && rel < d.w) {
            const float gh = p.gamma_h[(long long)it * 128 + rel];
            // hidden codes made by the library from h_int = A8 q carry gamma_A gamma_t; codes handed in from outside
            // (the FFN-level form, whose hidden activation went through its non-linearity first) carry gamma_h alone
            deq = p.hp_ext ? 1.0f / (p.hp_scales[2 * d.y + 1] * gh) : 1.0f / (p.hp_scales[2 * d.y + 1] * gh * p.hp_scales[2 * d.y] * p.gamma[pos]);
          }
        }
        r.ca *= deq;
      }
      if (!p.sstride) { r.cb *= p.beta[0]; if (HP) r.ca *= p.alpha[0]; }
    }
    return r;
  }
  // pure 1-bit tile
  __device__ static void epilogue(const Params& p, const Tile& t, const Pre& pre, uint32_t tacc, int quad, int part, int lane, uint8_t* stage) {
    for (int c = part; c * 64 < t.bn; c += kEpiWarps / 4) {     // 64 output columns = 128 bytes of the row per pass
      const int n0 = t.c.n0 + c * 64;
      if (n0 >= p.N) break;
      uint32_t w[32];
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const int nb = n0 + h * 16;
        if (c * 64 + h * 16 < t.bn && nb < p.N) {
          uint32_t a[16];
          tmem_ld16(tacc + c * 64 + h * 16, a);
          tmem_ld_wait();
          combine16(p, nb, pre.cb, a, a, w + 8 * h);
        }
      }
      uint4 o[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) o[j] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
      warp_store_rows<8>(stage, o, pre.yrow ? pre.yrow + n0 : nullptr, min(64, min(t.bn - c * 64, p.N - n0)) * 2, lane);
    }
  }
  // Tile with an HP branch: thread = row, columns [64 part, 64 part + 64).  The HP term is finished (alpha, gate, INT8 scales)
  // while the int8 contraction runs; between that contraction and the next one stand only the read of the int32
  // accumulator, one multiply-add per value and the rounding.
  struct Regs { uint32_t z[64]; };
  __device__ static __forceinline__ void take_first(const Params& p, const Tile& t, const Pre& pre, uint32_t tz, int part, Regs& r) {
    if (part * 64 < t.bn) {
      tmem_ld32(tz + part * 64, *reinterpret_cast<uint32_t(*)[32]>(r.z));
      tmem_ld32(tz + part * 64 + 32, *reinterpret_cast<uint32_t(*)[32]>(r.z + 32));
      tmem_ld_wait();
    }
  }
  __device__ static __forceinline__ void scale_first(const Params& p, const Tile& t, const Pre& pre, int part, Regs& r) {
    const bool is_int = p.gamma_h != nullptr;
#pragma unroll
    for (int q4 = 0; q4 < 16; ++q4) {
      const int n = t.c.n0 + part * 64 + q4 * 4;
      float a4[4] = {pre.ca, pre.ca, pre.ca, pre.ca};
      if (GEN && p.sstride && n < p.N) {             // N is a multiple of 32: whole groups of four
        const float4 av = __ldg(reinterpret_cast<const float4*>(p.alpha + n));
        a4[0] *= av.x; a4[1] *= av.y; a4[2] *= av.z; a4[3] *= av.w;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t v = r.z[4 * q4 + u];
        r.z[4 * q4 + u] = __float_as_uint(a4[u] * (is_int ? (float)(int)v : __uint_as_float(v)));
      }
    }
  }
  // the results take the place of the z values they are made from: pair j of the row's 64 columns ends up in z[j]
  __device__ static __forceinline__ void combine(const Params& p, const Tile& t, const Pre& pre, uint32_t tacc, int part, Regs& r) {
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const int n0 = t.c.n0 + part * 64 + h * 16;
      if (part * 64 + h * 16 < t.bn && n0 < p.N) {
        uint32_t a[16], w[8];
        tmem_ld16(tacc + part * 64 + h * 16, a);
        tmem_ld_wait();
        combine16(p, n0, pre.cb, a, r.z + 16 * h, w);
#pragma unroll
        for (int j = 0; j < 8; ++j) r.z[8 * h + j] = w[j];
      }
    }
  }
  __device__ static __forceinline__ void store(const Params& p, const Tile& t, const Pre& pre, int part, int lane, uint8_t* stage, const Regs& r) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int n0 = t.c.n0 + part * 64 + h * 32;
      if (part * 64 + h * 32 >= t.bn || n0 >= p.N) break;
      uint4 o[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) o[j] = make_uint4(r.z[16 * h + 4 * j], r.z[16 * h + 4 * j + 1], r.z[16 * h + 4 * j + 2], r.z[16 * h + 4 * j + 3]);
      warp_store_rows<4>(stage, o, pre.yrow ? pre.yrow + n0 : nullptr, min(32, p.N - n0) * 2, lane);
    }
  }
};
// (the macro takes one name per problem)
using FwdHp = FwdProblem<true, false, 2>;
using FwdHpGen = FwdProblem<true, true, 2>;
using Fwd1 = FwdProblem<false, false, 2>;
using Fwd1Gen = FwdProblem<false, true, 2>;
using FwdHpSingle = FwdProblem<true, false, 1>;
using FwdHpGenSingle = FwdProblem<true, true, 1>;
using Fwd1Single = FwdProblem<false, false, 1>;
using Fwd1GenSingle = FwdProblem<false, true, 1>;
PQ_DEFINE_GEMM_KERNEL(k_gemm_fwd_hp, FwdHp)
PQ_DEFINE_GEMM_KERNEL(k_gemm_fwd_hp_general, FwdHpGen)
PQ_DEFINE_GEMM_KERNEL(k_gemm_fwd_1bit, Fwd1)
PQ_DEFINE_GEMM_KERNEL(k_gemm_fwd_1bit_general, Fwd1Gen)
PQ_DEFINE_GEMM_KERNEL(k_gemm_fwd_hp_single, FwdHpSingle)
PQ_DEFINE_GEMM_KERNEL(k_gemm_fwd_hp_general_single, FwdHpGenSingle)
PQ_DEFINE_GEMM_KERNEL(k_gemm_fwd_1bit_single, Fwd1Single)
PQ_DEFINE_GEMM_KERNEL(k_gemm_fwd_1bit_general_single, Fwd1GenSingle)

// INT8 branch: the saved h region holds the codes qh [items*128, r] and, behind them, gamma_h [items*128]
static inline float* hp8_gamma_h(const SavedPtrs& sv, int r) {
  const size_t codes = ((size_t)sv.max_items * 128 * r + 255) / 256 * 256;
  return reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(sv.h) + codes);
}

// the fused output tile of a layer, with or without an HP branch
template <class P>
static int launch_forward(const LayerArgs& a, const int8_t* w_s8, const SavedPtrs& sv, uint16_t* Y, void (*kernel)(typename P::Params), bool HP,
                          cudaStream_t st, const SecondWeight& second) {
  constexpr int rows_b = 256 / P::CG;                // features of a tile that one CTA loads
  typename P::Params f;
  if (!map2d(&f.tq, true, sv.q, a.K, a.T, 128, 128)) return PQ_ERR_CUDA;
  if (!map2d(&f.ts, true, w_s8, a.K, a.N, 128, rows_b)) return PQ_ERR_CUDA;
  f.ts2 = f.ts; f.w_scales2 = second.w_scales; f.Y2 = second.Y;
  if (second.w_s8 && !map2d(&f.ts2, true, second.w_s8, a.K, a.N, 128, rows_b)) return PQ_ERR_CUDA;
  f.th = f.tq; f.tb = f.tq;
  f.gamma_h = nullptr; f.hp_scales = a.hp_scales; f.hp_ext = a.hp_ext ? 1 : 0;
  if (HP && a.hp_scales) {
    // INT8 branch: codes of h [items*128, r] and of B_e [E, N, r], one byte per value
    const uint64_t rows = (uint64_t)sv.max_items * 128;
    if (!map3d_i8(&f.th, sv.h, a.r, a.r, rows, 1, 128)) return PQ_ERR_CUDA;
    if (!map3d_i8(&f.tb, a.B, a.r, a.r, a.N, a.E, rows_b)) return PQ_ERR_CUDA;
    f.gamma_h = hp8_gamma_h(sv, a.r);
  } else if (HP) {
    if (!map2d(&f.th, false, sv.h, a.r, (uint64_t)sv.max_items * 256, 64, 128)) return PQ_ERR_CUDA;
    if (!map3d(&f.tb, a.B, a.r, a.N, a.E, 64, rows_b)) return PQ_ERR_CUDA;
  }
  f.rt = sv.rt; f.perm = (HP && a.E > 1) ? sv.perm : nullptr; f.gamma = sv.gamma; f.gate = sv.gate; f.w_scales = a.w_scales;
  f.alpha = a.alpha; f.beta = a.beta; f.Y = Y; f.T = a.T; f.N = a.N; f.K = a.K; f.r = a.r; f.sstride = a.scale_stride;
  f.item_rows = sv.max_items * 128;
  f.tiles1 = (a.N + 255) / 256;
  f.g = make_tile_grid((a.T + 128 * P::CG - 1) / (128 * P::CG), f.tiles1 * (second.w_s8 ? 2 : 1), 256);
  return launch_gemm<P>(KID_FWD, kernel, f, f.g.total, st);
}

// h_int = q A8_e^T per item.  raw == nullptr: codes and scales of h into the saved h region; otherwise the exact sums
// [items*128, r] into `raw` (A8 [E, r, K] int8).
int gemm_hp_up8(const LayerArgs& a, const SavedPtrs& sv, const void* A8, int* raw, cudaStream_t st, const void* A8b, int* rawb) {
  HpUp8Problem::Params p;
  p.rt = sv.rt; p.qh = reinterpret_cast<int8_t*>(sv.h); p.gamma_h = raw ? nullptr : hp8_gamma_h(sv, a.r); p.raw = raw; p.rawb = rawb;
  p.K = a.K; p.r = a.r; p.rp = a.r; p.bn = h_round_up(a.r, 16);
  if (!map2d(&p.tq, true, sv.q, a.K, a.T, 128, 128)) return PQ_ERR_CUDA;
  if (!map3d_i8(&p.ta, A8, a.K, a.K, a.r, a.E, p.bn)) return PQ_ERR_CUDA;
  p.tb = p.ta;
  if (rawb && !map3d_i8(&p.tb, A8b, a.K, a.K, a.r, a.E, p.bn)) return PQ_ERR_CUDA;
  return launch_gemm<HpUp8Problem>(KID_HP_UP, k_gemm_hp_up8, p, sv.max_items * (rawb ? 2 : 1), st);
}

int gemm_forward(const LayerArgs& a, const int8_t* w_s8, const SavedPtrs& sv, const uint16_t* xs, uint16_t* Y, cudaStream_t st,
                 cudaEvent_t before_main, const SecondWeight& second) {
  if (a.r > 0 && a.hp_scales) {
    if (!a.hp_ext) {
      const int rc = gemm_hp_up8(a, sv, a.A, nullptr, st);
      if (rc) return rc;
    }
  } else if (a.r > 0) {
    HpUpProblem::Params p;
    p.rt = sv.rt; p.H = sv.h; p.K = a.K; p.r = a.r; p.bn = h_round_up(a.r, 16); p.item_rows = sv.max_items * 128;
    if (!map2d(&p.tx, false, xs, a.K, a.T, 64, 128)) return PQ_ERR_CUDA;
    if (!map3d(&p.ta, a.A, a.K, a.r, a.E, 64, p.bn)) return PQ_ERR_CUDA;
    const int rc = launch_gemm<HpUpProblem>(KID_HP_UP, k_gemm_hp_up, p, sv.max_items, st);
    if (rc) return rc;
  }
  if (before_main && cudaStreamWaitEvent(st, before_main, 0) != cudaSuccess) return PQ_ERR_CUDA;
  const bool general = a.scale_stride != 0 || a.K >= 32768;
  // A pair takes half of the operand bytes per MMA, but its two CTAs go through launch, accumulators and epilogue in step: worth it from
  // a contraction of more than eight steps on.  Forward, single / pairs: 8192 tokens, 512 -> 2048, dense 33.9 / 39.5 us, 1024 -> 1024
  // 31.1 / 33.2, 256 tokens, 512 -> 512 20.8 / 22.4; without experts 8192, 2048 -> 2048 50.5 / 47.0, 2048, 3200 -> 8640 54.7 / 50.1.
  const bool pairs = a.K > 1024;
  if (a.r > 0 && pairs)
    return general ? launch_forward<FwdHpGen>(a, w_s8, sv, Y, k_gemm_fwd_hp_general, true, st, second) : launch_forward<FwdHp>(a, w_s8, sv, Y, k_gemm_fwd_hp, true, st, second);
  if (a.r > 0)
    return general ? launch_forward<FwdHpGenSingle>(a, w_s8, sv, Y, k_gemm_fwd_hp_general_single, true, st, second)
                   : launch_forward<FwdHpSingle>(a, w_s8, sv, Y, k_gemm_fwd_hp_single, true, st, second);
  if (pairs)
    return general ? launch_forward<Fwd1Gen>(a, w_s8, sv, Y, k_gemm_fwd_1bit_general, false, st, second) : launch_forward<Fwd1>(a, w_s8, sv, Y, k_gemm_fwd_1bit, false, st, second);
  return general ? launch_forward<Fwd1GenSingle>(a, w_s8, sv, Y, k_gemm_fwd_1bit_general_single, false, st, second)
                 : launch_forward<Fwd1Single>(a, w_s8, sv, Y, k_gemm_fwd_1bit_single, false, st, second);
}


// ===========================================================================
// backward (straight-through estimator, App. B.1)
// ===========================================================================
// The scale of the 1-bit input gradient: dX1 = c * (dYs . Sb) with
//   scalar beta:  Sb = S,            c = lam * beta
//   vector beta:  Sb = bf16(beta_n) S, c = lam
// The HP and router contributions are accumulated in the same tile, so they
// are pre-divided by c (and the whole tile multiplied by c in the epilogue).
// c == 0 switches the 1-bit term off instead.
__device__ __forceinline__ float dx_scale(const float* w_scales, const float* beta, int sstride) {
  return sstride ? w_scales[0] : w_scales[0] * beta[0];
}

// ---------------------------------------------------------------------------
// The whole backward in one launch.  Tiles of a pair of CTAs, in the order of their tickets:
//   dH   (one per pair of 128-row tiles and expert with rows there): dHraw = dYs . (alpha B_e); the epilogue forms
//          dg_t = alpha * sum_j H dHraw,  dH = g dHraw  ->  dhc = dH / c  (bf16, masked)
//          gh = g H (bf16, masked),  dl[t,j] = dg g (delta_je - p_tj),  dlc = dl / c
//   dW   (256 output features x 256 columns of K): G = dYs^T . xt; dW = beta_n G; per-tile partial of
//          dbeta_n = lam * sum_k S[n,k] G[n,k].
//   dWr  (256 columns of K): dWr^T = c * Xs^T . (dl / c), the logit gradient in the bf16 form the dX tile also uses
//          (Sec. 3.3, "trained end-to-end").
//   dX   (256 tokens x 256 columns of K) = c * ( dYs . Sb  +  sum_items dhc . A_e  +  dlc . Wr ), rows scattered back to
//          token order.
//   dB   (one per expert and 256 output features): dBraw_e = dYs^T . (g H) over the expert's items, the hi and lo
//          planes of g H side by side as the two halves of the tile's columns (one half per CTA of the pair);
//          dB = alpha_n dBraw, and the partial of dalpha_n = sum_j B[e,n,j] dBraw[n,j].
//   dA   (one per expert and 256 columns of K): dA_e^T = c * Xs^T . (dH / c) over the expert's items, with the
//          leading bf16 plane of dH / c (its 2^-9 rounding averages out over the tokens of the sum).
// dWr and dA have K as the rows of the tile, 256 of them for the pair, and the short dimension (E or r) as columns: the
// other way round half of a pair's rows would be empty.
//
// Bound by the tensor pipe, at the rate that a library's product reaches too: it is active 77 and 65 % of the time (2048 -> 5632 dense,
// 5632 -> 2048 with eight experts; 32 KB per CTA and 512 MMA cycles from L2, and tiles that take a quarter less gained nothing).  The tiles'
// contractions run over T, N, the tokens of an expert or a few hundred values, so what was left on the table was the last
// waves: as three launches (dH, dX, the rest, on two streams) with tiles handed out in turn, pairs with an extra dW tile also
// got the experts' tiles, and dH kept 64 SMs busy.  Here the longest tiles come first and whoever is free takes the next
// one.  dH has the first tickets and its readers (dWr, dX, dB, dA) wait for a counter of finished dH tiles: a ticket is
// drawn by a running pair only, a dH tile waits for nothing, so the counter gets there.  dW needs none of it and fills the
// time.  Measured, whole training step, three GEMM launches on two streams -> this: 256 tokens, 512 -> 512 54.6 -> 51.8 us;
// 8192 tokens, eight experts, 2048 -> 2048 329 -> 301 us, 5632 -> 2048 663 -> 671 us.
// ---------------------------------------------------------------------------
struct BwdProblem {
  static constexpr int CG = 2, kEpiWarps = 8;
  using Acc = AccDouble;
  enum Kind : int { KIND_DH = 0, KIND_DW, KIND_DWR, KIND_DX, KIND_DB, KIND_DA };
  struct Params {
    CUtensorMap tdy, tba, tsb, tdh, ta3, tdl, twr;   // dYs [T,N]; (alpha) B [E,N,r]; Sb [N,K]; dhc; A; dlc; Wr
    CUtensorMap tdyT, txt, tgh, tdlT, txs, tdhT;     // the same and q / gamma, g H, Xs, contracted over tokens
    RoutingTables rt;
    const uint16_t* H;
    const float* gate;
    const float* probs;
    const int8_t* s8;
    const float* beta;
    const float* alpha;
    const float* w_scales;
    const uint16_t* B;       // [E, N, r]
    const int* perm;
    const int* offsets;      // [E + 1] first row of each expert
    uint16_t* dhc;
    uint16_t* gh;
    float* dl;
    uint16_t* dlc;
    uint16_t* dX;
    float* dWr;              // [E, K]
    float* dA;               // [E, r, K]
    float* dW;
    float* dB;               // [E, N, r]
    float* dbeta_partial;    // [2 * ceil(K/256), N]
    float* dalpha_partial;   // [2 * E, N]
    unsigned* sync;          // {.., tickets, finished warps of dH tiles}
    TileGrid gx, gw;
    int T, N, K, r, r64, E, sstride, item_rows, ntn, ntk, mpairs, hp, long_experts, early_dx;
    int ba_blk, sb_blk, a3_blk, wr_blk, dy_blk, xt_blk, gh_blk, xs_blk, dh_blk;
  };
  // nt: this CTA's block of 128 rows (tokens, features, or columns of K); [ib, ie): items (dB, dA), pair entries (dX); item: this
  // CTA's item of a dH tile or -1, with its rows [lo, hi); lo: of a dB or dA tile, the 128-row tile of its first item
  struct Tile { int kind, rank, nt, n0, bn, e, ib, ie, item, lo, hi, skip1; };
  __device__ static unsigned* tickets(const Params& p) { return p.sync + 1; }
  __device__ static int dh_tiles(const Params& p) { return p.hp ? p.rt.pair_begin[p.mpairs] : 0; }
  __device__ static int num_tiles(const Params& p) {
    return dh_tiles(p) + p.gw.total + p.gx.total + (p.hp ? p.E * (p.ntn + p.ntk) + (p.E > 1 ? p.ntk : 0) : 0);
  }
  __device__ static void tile_init(const Params& p, int i, int rank, Tile& t) {
    t.ib = t.ie = 0; t.e = 0; t.n0 = 0; t.rank = rank; t.item = -1; t.lo = t.hi = 0; t.skip1 = 0;
    const int dh = dh_tiles(p);
    if (i < dh) {
      const int4 pi = p.rt.pair_items[i];
      t.kind = KIND_DH; t.e = pi.x; t.item = rank ? pi.z : pi.y; t.nt = 2 * pi.w + rank; t.bn = round_up(p.r, 128);
      if (t.item >= 0) { const int4 it = p.rt.items[t.item]; t.lo = it.z; t.hi = it.w; }
      return;
    }
    i -= dh;
    if (i < p.gw.total) {
      t.kind = KIND_DW;
      // along the shorter side of the grid first: the tiles under way at a time then read the fewest different panels
      const bool tall = p.gw.mt > p.gw.nt;
      const int m = tall ? i / p.gw.nt : i % p.gw.mt, n = tall ? i % p.gw.nt : i / p.gw.mt;
      t.nt = CG * m + rank; t.n0 = n * p.gw.bn;
      t.bn = clip_bn(p.gw.bn, t.n0, p.K, 128);
      return;
    }
    i -= p.gw.total;
    if (p.hp && p.E > 1) {
      if (i < p.ntk) {
        t.kind = KIND_DWR; t.nt = 2 * i + rank; t.bn = 128;
        return;
      }
      i -= p.ntk;
    }
    // the experts' tiles before dX where their contraction (all tokens, with one expert) is the longer one, else after it
    const int experts = p.hp ? p.E * (p.ntn + p.ntk) : 0;
    int x = p.long_experts ? i - experts : i;
    if (x >= 0 && x < p.gx.total) {
      t.kind = KIND_DX;
      const TileCoord c = tile_coord<CG>(p.gx, x, rank);
      t.nt = c.m; t.n0 = c.n0;
      t.bn = clip_bn(c.bn, c.n0, p.K, 128);
      if (p.hp) { t.ib = p.rt.pair_begin[t.nt >> 1]; t.ie = p.rt.pair_begin[(t.nt >> 1) + 1]; }
      t.skip1 = dx_scale(p.w_scales, p.beta, p.sstride) == 0.f;
      return;
    }
    x = p.long_experts ? i : i - p.gx.total;
    t.e = x / (p.ntn + p.ntk);
    x -= t.e * (p.ntn + p.ntk);
    t.ib = p.rt.expert_item_begin[t.e]; t.ie = p.rt.expert_item_begin[t.e + 1];
    t.lo = p.offsets[t.e] >> 7;
    if (x < p.ntn) { t.kind = KIND_DB; t.nt = 2 * x + rank; t.bn = 2 * p.r64; }
    else { t.kind = KIND_DA; t.nt = 2 * (x - p.ntn) + rank; t.bn = 128; }
  }
  // What reads the results of the dH tiles waits for them; they were written through the generic proxy.  In a dX tile that is every
  // segment but the first, the product with Sb; where it is long and the tiles are few (see early_dx) the wait comes after it.
  __device__ static bool ready(const Params& p, const Tile& t, int i, volatile int* abort_flag) {
    if (!p.hp || t.kind == KIND_DH || t.kind == KIND_DW || i != (t.kind == KIND_DX && !t.skip1 && p.early_dx ? 1 : 0)) return true;
    const unsigned want = 8u * dh_tiles(p);                // four warps in each CTA of a pair
    const long long t0 = clock64();
    unsigned v;
    for (;;) {
      asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(p.sync + 2) : "memory");
      if (v >= want) break;
      if (*abort_flag) return false;
      if (clock64() - t0 > c_spin_cycles) {
        report_timeout(WHERE_PRODUCER);
        *abort_flag = 1;
        return false;
      }
    }
    asm volatile("fence.proxy.async;" ::: "memory");
    return true;
  }
  __device__ static int num_segments(const Params& p, const Tile& t) {
    if (t.kind == KIND_DX) return (t.skip1 ? 0 : 1) + 2 * (t.ie - t.ib) + (p.hp && p.E > 1 ? 1 : 0);
    return t.kind == KIND_DB || t.kind == KIND_DA ? t.ie > t.ib : 1;
  }
  __device__ static void segment(const Params& p, const Tile& t, int i, Segment& s) {
    s.acc = 0; s.bn = t.bn; s.ksteps = 4; s.b_bytes = kOperandBytes;
    s.a_rank = 2; s.a_z = 0; s.b_rank = 2; s.b_z = 0;
    if (t.kind == KIND_DX) {
      s.mode = MODE_BF_KM; s.a_x = 0; s.a_blk = 0;
      s.b_x = t.n0 + t.rank * (t.bn >> 1); s.b_y = 0;
      if (!t.skip1) {
        if (i == 0) {
          s.nkb = (p.N + 63) / 64;
          s.ta = &p.tdy; s.a_y = t.nt * 128;
          s.tb = &p.tsb; s.b_rank = 2; s.b_blk = p.sb_blk;
          return;
        }
        --i;
      }
      if (i < 2 * (t.ie - t.ib)) {
        const int4 pi = p.rt.pair_items[t.ib + (i >> 1)];
        const int item = t.rank ? pi.z : pi.y, plane = i & 1;
        s.nkb = (p.r + 63) / 64;
        s.ta = &p.tdh; s.a_y = item >= 0 ? plane * p.item_rows + item * 128 : 2 * p.item_rows;   // beyond both planes: zeros
        s.tb = &p.ta3; s.b_rank = 3; s.b_z = pi.x; s.b_blk = p.a3_blk;
        return;
      }
      s.nkb = 1; s.ksteps = 1;
      s.ta = &p.tdl; s.a_y = t.nt * 128;
      s.tb = &p.twr; s.b_rank = 2; s.b_blk = p.wr_blk;
      return;
    }
    if (t.kind == KIND_DH) {
      s.mode = MODE_BF_KM; s.nkb = (p.N + 63) / 64; s.a_x = 0; s.a_blk = 0;
      s.ta = &p.tdy; s.a_y = t.item >= 0 ? t.nt * 128 : p.T;     // no rows of this expert in the CTA's tile: zeros
      s.tb = &p.tba; s.b_rank = 3; s.b_x = t.rank * (t.bn >> 1); s.b_y = 0; s.b_z = t.e; s.b_blk = p.ba_blk; s.b_bytes = t.bn * 64;
      return;
    }
    s.mode = MODE_BF_MM; s.a_x = t.nt * 128;
    switch (t.kind) {
      case KIND_DW:
        s.nkb = (p.T + 63) / 64;
        s.ta = &p.tdyT; s.a_y = 0; s.a_blk = p.dy_blk;
        s.tb = &p.txt; s.b_x = t.n0 + t.rank * (t.bn >> 1); s.b_y = 0; s.b_blk = p.xt_blk;
        break;
      case KIND_DB:
        // The 128 tokens of every item's tile (rows outside the item are zero in g H).  An expert's items lie behind one another, in tiles
        // behind one another, so that its contraction is one run on both sides.  As a segment per item, looked up each time, a step of
        // these tiles took 1170 cycles, 310 or 512 of them the tensor pipe's.  Training step, dense: 8192 tokens, 2048 -> 5632 518 -> 504 us, 4096,
        // 2048 -> 1024 121 -> 110; with eight experts 1 % (8192 tokens, 5632 -> 2048 649 -> 642, 2048 -> 2048 285 -> 282), what runs differ by.
        s.nkb = 2 * (t.ie - t.ib);
        s.ta = &p.tdyT; s.a_y = t.lo * 128; s.a_blk = p.dy_blk;
        s.tb = &p.tgh; s.b_x = 0; s.b_y = t.rank * p.item_rows + t.ib * 128; s.b_blk = p.gh_blk; s.b_bytes = p.r64 * 128;
        break;
      case KIND_DWR:
        s.nkb = (p.T + 63) / 64;
        s.ta = &p.txs; s.a_y = 0; s.a_blk = p.xs_blk;
        s.tb = &p.tdlT; s.b_x = t.rank * 64; s.b_y = 0; s.b_blk = -1; s.b_bytes = kMnBoxBytes;   // 16 columns, zeros beyond
        break;
      default:                                            // KIND_DA
        s.nkb = 2 * (t.ie - t.ib);
        s.ta = &p.txs; s.a_y = t.lo * 128; s.a_blk = p.xs_blk;
        s.tb = &p.tdhT; s.b_x = t.rank * 64; s.b_y = t.ib * 128; s.b_blk = p.dh_blk; s.b_bytes = kMnBoxBytes;
        break;
    }
  }
  struct Pre { uint16_t* xrow; float cc; };
  __device__ static Pre prepare(const Params& p, const Tile& t, int quad, int lane) {
    Pre r{nullptr, 1.0f};
    if (t.kind == KIND_DH && t.item >= 0) {
      const long long row = ((long long)t.item * 128 + quad * 32 + lane) * p.r, plane = (long long)p.item_rows * p.r;
      for (int j = 0; j < p.r; j += 64) {
        asm volatile("prefetch.global.L1 [%0];" ::"l"(p.H + row + j));
        asm volatile("prefetch.global.L1 [%0];" ::"l"(p.H + plane + row + j));
      }
    }
    if (t.kind != KIND_DX) return r;
    const int pos = t.nt * 128 + quad * 32 + lane;
    const float c = dx_scale(p.w_scales, p.beta, p.sstride);
    if (c != 0.f) r.cc = c;
    if (pos < p.T) r.xrow = p.dX + (long long)(p.perm ? p.perm[pos] : pos) * p.K;
    return r;
  }
  __device__ static void epilogue(const Params& p, const Tile& t, const Pre& pre, uint32_t taddr, int quad, int part, int lane, uint8_t* stage) {
    if (t.kind == KIND_DX) epilogue_dx(p, t, pre, taddr, part, lane, stage);
    else if (t.kind != KIND_DH) epilogue_tokens(p, t, taddr, quad, part, lane, stage);
    else if (part == 0) {                          // each row's sum over all r columns stays in one thread
      if (t.item >= 0) epilogue_dh(p, t, taddr, quad, lane);
      // this warp's rows are written: visible to every later TMA load, then counted
      __threadfence();
      asm volatile("fence.proxy.async;" ::: "memory");
      __syncwarp();
      if (lane == 0) atomicAdd(p.sync + 2, 1u);
    }
  }
  __device__ static void epilogue_dh(const Params& p, const Tile& t, uint32_t taddr, int quad, int lane) {
    const int row = quad * 32 + lane;
    const bool live = row >= t.lo && row < t.hi;
    const int pos = t.nt * 128 + row;
    const float c = dx_scale(p.w_scales, p.beta, p.sstride);
    const float inv_cc = c != 0.f ? 1.0f / c : 1.0f;
    const float ca = p.sstride ? 1.0f : p.alpha[0];
    const float g = live ? p.gate[pos] : 0.f;
    const long long hrow = ((long long)t.item * 128 + row) * p.r;
    const long long plane = (long long)p.item_rows * p.r;
    const uint4* hin = reinterpret_cast<const uint4*>(p.H + hrow);
    const uint4* hin_lo = reinterpret_cast<const uint4*>(p.H + plane + hrow);
    uint4* dhc = reinterpret_cast<uint4*>(p.dhc + hrow);
    uint4* dhc_lo = reinterpret_cast<uint4*>(p.dhc + plane + hrow);
    uint4* gh = reinterpret_cast<uint4*>(p.gh + hrow);
    uint4* gh_lo = reinterpret_cast<uint4*>(p.gh + plane + hrow);
    float dg = 0.f;
    for (int c32 = 0; c32 * 32 < p.r; ++c32) {
      uint32_t v[32];
      tmem_ld32(taddr + c32 * 32, v);
      tmem_ld_wait();
#pragma unroll
      for (int q8 = 0; q8 < 4; ++q8) {
        if (c32 * 32 + q8 * 8 < p.r) {
          uint32_t w1[4] = {0, 0, 0, 0}, w1l[4] = {0, 0, 0, 0}, w2[4] = {0, 0, 0, 0}, w2l[4] = {0, 0, 0, 0};
          if (live) {
            const uint4 hv = hin[c32 * 4 + q8], hl = hin_lo[c32 * 4 + q8];
            const uint32_t hw[4] = {hv.x, hv.y, hv.z, hv.w}, hlw[4] = {hl.x, hl.y, hl.z, hl.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float h0 = bf16lo(hw[j]) + bf16lo(hlw[j]), h1 = bf16hi(hw[j]) + bf16hi(hlw[j]);
              const float d0 = __uint_as_float(v[q8 * 8 + 2 * j]), d1 = __uint_as_float(v[q8 * 8 + 2 * j + 1]);
              dg = fmaf(h0, d0, dg);
              dg = fmaf(h1, d1, dg);
              const float sc = ca * g * inv_cc;
              split2(sc * d0, sc * d1, w1[j], w1l[j]);
              split2(g * h0, g * h1, w2[j], w2l[j]);
            }
          }
          dhc[c32 * 4 + q8] = make_uint4(w1[0], w1[1], w1[2], w1[3]);
          dhc_lo[c32 * 4 + q8] = make_uint4(w1l[0], w1l[1], w1l[2], w1l[3]);
          gh[c32 * 4 + q8] = make_uint4(w2[0], w2[1], w2[2], w2[3]);
          gh_lo[c32 * 4 + q8] = make_uint4(w2l[0], w2l[1], w2l[2], w2l[3]);
        }
      }
    }
    if (p.E > 1 && live) {
      dg *= ca;
      uint32_t packed[8];
      float prev = 0.f;
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        float d = 0.f;
        if (e < p.E) {
          d = dg * g * ((e == t.e ? 1.0f : 0.0f) - p.probs[(long long)pos * p.E + e]);
          p.dl[(long long)pos * p.E + e] = d;
        }
        if (e & 1) packed[e >> 1] = pack_bf16x2(prev * inv_cc, d * inv_cc);
        prev = d;
      }
      uint4* o = reinterpret_cast<uint4*>(p.dlc + (long long)pos * 16);
      o[0] = make_uint4(packed[0], packed[1], packed[2], packed[3]);
      o[1] = make_uint4(packed[4], packed[5], packed[6], packed[7]);
    }
  }
  __device__ static void epilogue_dx(const Params& p, const Tile& t, const Pre& pre, uint32_t taddr, int part, int lane, uint8_t* stage) {
    const float cc = pre.cc;
    const bool has = num_segments(p, t) > 0;
    for (int c64 = part; c64 * 64 < t.bn; c64 += kEpiWarps / 4) {
      const int k0 = t.n0 + c64 * 64;
      if (k0 >= p.K) break;
      uint32_t v0[32], v1[32];
      tmem_ld32(taddr + c64 * 64, v0);
      tmem_ld32(taddr + c64 * 64 + 32, v1);
      tmem_ld_wait();
      uint4 o[8];
      uint32_t w[32];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        w[j] = has ? pack_bf16x2(cc * __uint_as_float(v0[2 * j]), cc * __uint_as_float(v0[2 * j + 1])) : 0u;
        w[16 + j] = has ? pack_bf16x2(cc * __uint_as_float(v1[2 * j]), cc * __uint_as_float(v1[2 * j + 1])) : 0u;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) o[j] = make_uint4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
      warp_store_rows<8>(stage, o, pre.xrow ? pre.xrow + k0 : nullptr, min(64, p.K - k0) * 2, lane);
    }
  }
  __device__ static void epilogue_tokens(const Params& p, const Tile& t, uint32_t taddr, int quad, int part, int lane, uint8_t* stage) {
    if (t.kind == KIND_DWR || t.kind == KIND_DA) {
      // ---- row k of the tile, column j: dWr[j, k] / c, or dA[e, j, k] / c.  A warp holds 32 consecutive k of one j: whole lines
      const int k = t.nt * 128 + quad * 32 + lane;
      const float c = dx_scale(p.w_scales, p.beta, p.sstride);
      const float cc = c != 0.f ? c : 1.0f;
      const bool any = t.kind == KIND_DWR || t.ie > t.ib;    // an expert without tokens: exact zeros
      const int cols = t.kind == KIND_DWR ? p.E : p.r;
      float* out = t.kind == KIND_DWR ? p.dWr + k : p.dA + (long long)t.e * p.r * p.K + k;
      for (int c32 = part; c32 * 32 < cols; c32 += kEpiWarps / 4) {
        uint32_t v[32];
        if (any) {
          tmem_ld32(taddr + c32 * 32, v);
          tmem_ld_wait();
        } else {
#pragma unroll
          for (int u = 0; u < 32; ++u) v[u] = 0u;
        }
        if (k < p.K) {
#pragma unroll
          for (int u = 0; u < 32; ++u)
            if (c32 * 32 + u < cols) out[(long long)(c32 * 32 + u) * p.K] = cc * __uint_as_float(v[u]);
        }
      }
      return;
    }
    const int n = t.nt * 128 + quad * 32 + lane;
    const bool live = n < p.N;
    if (t.kind == KIND_DB) {
      // ---- dB tile: columns [0, r64) hold the hi-plane product, [r64, 2 r64) the lo-plane product
      const bool any = t.ie > t.ib;                     // an expert without tokens: exact zeros
      const float al = live ? p.alpha[n * p.sstride] : 0.f;
      const long long row = ((long long)t.e * p.N + (live ? n : 0)) * p.r;
      float psum = 0.f;
      for (int c32 = part; c32 * 32 < p.r; c32 += kEpiWarps / 4) {
        uint32_t vh[32], vl[32];
        if (any) {
          tmem_ld32(taddr + c32 * 32, vh);
          tmem_ld32(taddr + p.r64 + c32 * 32, vl);
          tmem_ld_wait();
        }
        uint4 o[8];
#pragma unroll
        for (int q4 = 0; q4 < 8; ++q4) {
          float gsum[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) gsum[u] = any ? __uint_as_float(vh[4 * q4 + u]) + __uint_as_float(vl[4 * q4 + u]) : 0.f;
          const int j = c32 * 32 + q4 * 4;
          if (live && j < p.r) {
            const uint2 bv = *reinterpret_cast<const uint2*>(p.B + row + j);
            psum = fmaf(bf16lo(bv.x), gsum[0], psum); psum = fmaf(bf16hi(bv.x), gsum[1], psum);
            psum = fmaf(bf16lo(bv.y), gsum[2], psum); psum = fmaf(bf16hi(bv.y), gsum[3], psum);
          }
          o[q4] = make_uint4(__float_as_uint(al * gsum[0]), __float_as_uint(al * gsum[1]), __float_as_uint(al * gsum[2]),
                             __float_as_uint(al * gsum[3]));
        }
        warp_store_rows<8>(stage, o, live ? p.dB + row + c32 * 32 : nullptr, min(32, p.r - c32 * 32) * 4, lane);
      }
      if (live) p.dalpha_partial[(long long)(2 * t.e + part) * p.N + n] = psum;
      return;
    }
    const float be = live ? p.beta[n * p.sstride] : 0.f;
    float* wrow = live ? p.dW + (long long)n * p.K : nullptr;
    const uint4* srow = reinterpret_cast<const uint4*>(p.s8 + (long long)(live ? n : 0) * p.K);
    float psum = 0.f;
    for (int c32 = part; c32 * 32 < t.bn; c32 += kEpiWarps / 4) {
      const int k0 = t.n0 + c32 * 32;
      if (k0 >= p.K) break;
      uint32_t v[32];
      tmem_ld32(taddr + c32 * 32, v);
      tmem_ld_wait();
      uint4 o[8];
      uint32_t sw[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      if (live) {
        const uint4 s0 = __ldg(srow + (k0 >> 4)), s1 = __ldg(srow + (k0 >> 4) + 1);
        sw[0] = s0.x; sw[1] = s0.y; sw[2] = s0.z; sw[3] = s0.w; sw[4] = s1.x; sw[5] = s1.y; sw[6] = s1.z; sw[7] = s1.w;
      }
#pragma unroll
      for (int q4 = 0; q4 < 8; ++q4) {
        const float g0 = __uint_as_float(v[q4 * 4]), g1 = __uint_as_float(v[q4 * 4 + 1]);
        const float g2 = __uint_as_float(v[q4 * 4 + 2]), g3 = __uint_as_float(v[q4 * 4 + 3]);
        const uint32_t sb = sw[q4];  // four +-1 bytes: bit 7 set <-> -1
        psum += (sb & 0x80u) ? -g0 : g0;
        psum += (sb & 0x8000u) ? -g1 : g1;
        psum += (sb & 0x800000u) ? -g2 : g2;
        psum += (sb & 0x80000000u) ? -g3 : g3;
        o[q4] = make_uint4(__float_as_uint(be * g0), __float_as_uint(be * g1), __float_as_uint(be * g2), __float_as_uint(be * g3));
      }
      warp_store_rows<8>(stage, o, wrow ? wrow + k0 : nullptr, 128, lane);
    }
    // one slot per (column tile, warp of the row pair)
    if (live) p.dbeta_partial[(long long)(2 * (t.n0 / 256) + part) * p.N + n] = psum;
  }
};
PQ_DEFINE_GEMM_KERNEL(k_gemm_bwd, BwdProblem)

int gemm_backward(const LayerArgs& a, const int8_t* w_s8, const SavedPtrs& sv, const BwdBuffers& b, uint16_t* dX, float* dW, float* dA,
                  float* dB, float* dWr, cudaStream_t st) {
  const int ntk = (a.K + 255) / 256, ntn = (a.N + 255) / 256;
  const bool hp = a.r > 0, routed = hp && a.E > 1;
  const int r64 = h_round_up(a.r, 64);
  const uint64_t item_rows = (uint64_t)sv.max_items * 128;  // rows of one plane; buffers hold two
  BwdProblem::Params p{};
  if (!map2d(&p.tdy, false, b.dys, a.N, a.T, 64, 128)) return PQ_ERR_CUDA;
  if (!map_mn(&p.tsb, &p.sb_blk, b.sb, a.K, a.N, 2, 1, 2)) return PQ_ERR_CUDA;
  if (!map_mn(&p.tdyT, &p.dy_blk, b.dys, a.N, a.T, 2, 1, 2)) return PQ_ERR_CUDA;
  if (!map_mn(&p.txt, &p.xt_blk, sv.xt, a.K, a.T, 2, 1, 2)) return PQ_ERR_CUDA;
  p.tba = p.tdh = p.ta3 = p.tdl = p.twr = p.tgh = p.tdlT = p.txs = p.tdhT = p.tdy;
  if (hp) {
    if (!map_mn(&p.tba, &p.ba_blk, b.ba, a.r, a.N, 3, a.E, h_round_up(a.r, 128) / 128)) return PQ_ERR_CUDA;
    if (!map2d(&p.tdh, false, b.dhc, a.r, 2 * item_rows, 64, 128)) return PQ_ERR_CUDA;
    if (!map_mn(&p.ta3, &p.a3_blk, a.A, a.K, a.r, 3, a.E, 2)) return PQ_ERR_CUDA;
    if (!map_mn(&p.tgh, &p.gh_blk, b.gh, a.r, 2 * item_rows, 2, 1, r64 / 64)) return PQ_ERR_CUDA;
    if (!map_mn(&p.txs, &p.xs_blk, b.xs, a.K, a.T, 2, 1, 2)) return PQ_ERR_CUDA;
    if (!map_mn(&p.tdhT, &p.dh_blk, b.dhc, a.r, 2 * item_rows, 2, 1, 1)) return PQ_ERR_CUDA;
  }
  if (routed) {
    int one_box = 0;
    if (!map2d(&p.tdl, false, b.dlc, 16, a.T, 64, 128)) return PQ_ERR_CUDA;
    if (!map_mn(&p.twr, &p.wr_blk, a.Wr, a.K, a.E, 2, 1, 2)) return PQ_ERR_CUDA;
    if (!map_mn(&p.tdlT, &one_box, b.dlc, 16, a.T, 2, 1, 1)) return PQ_ERR_CUDA;
  }
  p.rt = sv.rt; p.H = sv.h; p.gate = sv.gate; p.probs = sv.probs; p.s8 = w_s8; p.beta = a.beta; p.alpha = a.alpha; p.w_scales = a.w_scales;
  p.B = a.B; p.perm = routed ? sv.perm : nullptr; p.offsets = sv.offsets;
  p.dhc = b.dhc; p.gh = b.gh; p.dl = b.dl; p.dlc = b.dlc; p.dX = dX; p.dWr = dWr; p.dA = dA; p.dW = dW; p.dB = dB;
  p.dbeta_partial = b.dbeta_partial; p.dalpha_partial = b.dalpha_partial; p.sync = b.sync;
  p.T = a.T; p.N = a.N; p.K = a.K; p.r = a.r; p.r64 = r64; p.E = hp ? a.E : 1; p.sstride = a.scale_stride; p.item_rows = (int)item_rows;
  p.ntn = ntn; p.ntk = ntk; p.mpairs = (a.T + 255) / 256; p.hp = hp; p.long_experts = hp && a.E == 1;
  // A dX tile that has done its first product beside the dH tiles has little left when they are finished; one of many, drawn by pairs
  // that the dH tiles need the L2 of, only slows them.  Backward, waiting before and after: 512 tokens, 1024 -> 4096, one / eight experts
  // 68 / 83 and 56 / 71 us; 1024 tokens, 1024 -> 1024, eight experts 51 and 47; 8192 tokens, 2048 -> 2048, one / eight 134 / 161 and 137 / 166.
  p.early_dx = routed ? a.N >= a.T : a.N > a.T;
  p.gx = make_tile_grid(p.mpairs, ntk, 256);
  p.gw = make_tile_grid(ntn, ntk, 256);
  return launch_gemm<BwdProblem>(KID_BWD_DW, k_gemm_bwd, p, p.gx.total + p.gw.total + (hp ? p.E * (ntn + ntk) : 0), st);
}

}  // namespace pq
