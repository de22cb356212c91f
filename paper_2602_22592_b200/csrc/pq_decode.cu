// Decode path of the pQuant layer (App. A): M <= 16 tokens against weights stored as packed sign bits, three kernels per group
// of independent linears:
//
//   k_decode_prep    a cluster of eight CTAs per (linear, token): RMSNorm (optional), absmax quantisation (Eq. 7-9), router
//                    (Sec. 3.3); every CTA takes its share of the experts' logits and of the codes.
//   k_decode_hidden  a cluster of CTAs per (linear, expert in use, 16 hidden rows): h = A_e x for all tokens of the expert.
//   k_decode_main    one CTA per SM, a contiguous share of the output features of all linears each, in units of 16:
//                    1-bit product on mma.sync (u8 bit masks x s8 codes, exact in int32), expert product z = B_e h on bf16
//                    mma.sync (dp4a for the INT8 branch), epilogue (Eq. 10-11).
//
// A call of one or two linears is a chain of dependent steps, not a stream: its weights take 1-2 us at the memory's rate, a
// dependent trip to memory about 1 us.  So everything off the chain runs beside it.  The kernels are launched with programmatic
// stream serialisation; each lets its successor start once the kernels before it have finished, so that a kernel may read what
// its predecessor's predecessors wrote before it waits for the predecessor itself: k_decode_main has its sign bits multiplied
// with the codes and the experts' rows of B on their way when h arrives.
//
// Measured, two kernels with the hidden rows in the first (INT8 experts: the streaming kernel) -> these three: one 2048 x 2048
// linear, one token 13.8 -> 10.8 us; 26 layers of gate + up, then down of 3200 x 8640, one token 1010 -> 790 us, sixteen 1767 -> 1591
// us; 8 layers, four tokens, INT8 experts 573 -> 278 us.  A dense branch with nine to fourteen tokens loses 1 us a call.
//
// The sum over k of q S is evaluated as 2 * (sum over the set bits of q) - (sum of q): the bit
// words feed the tensor cores as 0/1 masks without expansion to +-1.
#include <algorithm>

#include "pq_kernels.cuh"

namespace pq {

constexpr int kDecodeMaxTokens = 16;
constexpr int kDecodeMaxBatch = 96;       // linears per launch (their descriptors travel as kernel parameters)
constexpr int kPrepThreads = 256;
constexpr int kPrepWarps = kPrepThreads / 32;
constexpr int kPrepCluster = 8;           // CTAs that share a token's router
constexpr int kHiddenSplit = 32;          // shares of the contraction of sixteen hidden rows, added up in order
constexpr int kHiddenThreads = 256;
constexpr int kHiddenWarps = kHiddenThreads / 32;
constexpr int kMainThreads = 512;
constexpr int kMainWarps = kMainThreads / 32;
constexpr int kUnit = 16;                 // output features of a unit of work (the rows of one mma tile)
constexpr int kMaxPassUnits = 8;          // units a CTA works on at once (two warps or more each)
constexpr int kWarpRows = 2;              // tiles of expert rows a warp of k_decode_main has in flight
constexpr int kMaxRows = kWarpRows * kMainWarps;
static_assert(kWarpRows == 2, "the host's choice of places");

struct DecodeTokInfo {  // one per token
  int expert;
  float gate;
  float gamma;
  int rowsum;           // sum over k of q[k]
};

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar) : "memory");
}
// ask `bytes` (a multiple of 16) into L2
__device__ __forceinline__ void bulk_prefetch(const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(reinterpret_cast<uint64_t>(src)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mma_u8s8(int (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.u8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// ---------------------------------------------------------------------------
// Layout of the quantised activations handed from prep to main ("q fragments").
// A chunk is 128 values of k: four 32-bit weight words per feature, word c for the threads of quad index c (lane & 3).  For
// b = 0..3 such a thread takes from its word w the bits b + 8 j (mask 0x01010101 of w >> b) and b + 4 + 8 j (mask 0x10101010,
// i.e. the value 16), j = 0..3: one 4-byte operand register each.  The tokens' side of bit b is the word of codes
// q[128 chunk + 32 c + b + 8 j].  The eight words of (chunk, token, c) are two 16-byte pieces, half h holding b = 4 h .. 4 h + 3;
// only the tokens that exist are stored: with Mg = min(8, M - 8 group) tokens in the group, the piece of (chunk, half h, token
// g, c) sits at uint4 index group * chunks * 64 + ((2 chunk + h) * Mg + g) * 4 + c.
// ---------------------------------------------------------------------------

// One linear of a batch: device pointers and sizes (the workspace pointers are carved by the host).
struct alignas(16) DecodeLinear {
  const uint4* X;           // [M, K] bf16
  const uint4* Wr;          // [E, K] bf16 or null
  const uint16_t* A;        // [E, r, K]
  const uint16_t* B;        // [E, N, r]
  const uint32_t* bits;     // [N, K/32]
  const uint4* bits_il;     // the same bits as laid out by decode_pack, or null
  const float* w_scales;
  const float* alpha;
  const float* beta;
  uint16_t* Y;              // [M, N]
  DecodeTokInfo* info;      // [16]
  uint4* qfrag;             // [2 groups][chunks][2][8 tokens][4] fragments
  uint4* hfrag;             // [2 groups][2 planes (hi, lo)][ceil(r/32)][32] fragments of h = A_e x
  uint16_t* xn;             // [M, K] what k_decode_hidden multiplies: normalised tokens (bf16; X itself without a norm), or int8 codes
  int* acc_dump;            // [M, N] exact 1-bit accumulators (test hook) or null
  const uint4* norm_w;      // [K] bf16 RMSNorm gain or null
  // INT8 high-precision branch (Sec. 3.2), null without it
  const int8_t* A8;         // [E, r, K]
  const uint4* B8_il;       // [E][N / 32 groups, padded to whole 128-feature groups][r / 16][32] pieces of 16 codes
  const float* hp_scales;   // [E][2]
  int* h_int;               // [M, r]
  int* zint_dump;           // [M, N] or null
  float norm_eps;
  int M, K, N, r, E, sstride;
  int hidden0;              // first cluster of this linear in k_decode_hidden (min(E, M) * ceil(r / 16) of them)
  int unit0;                // first unit of work of this linear in the launch
};
static_assert(sizeof(DecodeLinear) % 16 == 0, "copied in 16-byte pieces");
template <int CAP>
struct DecodeBatch {
  int n, units;             // linears; units of 16 features of all of them
  int poll;                 // waits are polled
  int early;                // k_decode_hidden runs in between: k_decode_main may read prep's results before it waits
  int hidden_groups, hidden_cluster;   // k_decode_hidden: clusters of all linears, CTAs of each
  // k_decode_main: buffers of sign bits, their size, the carve-up of shared memory behind them, and how many tiles of expert rows
  // have a place apart (0: they go over used sign bits)
  int nbuf, buf_bytes, off_q, off_h, off_red, off_rows, row_slots;
  int q_chunks;             // chunks of 128 values of k whose codes are in shared memory at once
  int pass_units;           // units of a pass at most
  int rows_early;           // k_decode_hidden brings the experts' rows of B into L2
  int red_tokens;
  int unit0[CAP + 1];
  DecodeLinear lin[CAP];
};

// A record of the batch into shared memory, one 16-byte piece per warp at a time: a piece of the parameters that no thread has
// touched yet is a trip to memory, so all are touched at once and before anything has to be waited for.
template <int CAP>
__device__ __forceinline__ void copy_record(DecodeLinear* dst, const DecodeBatch<CAP>& bp, int l) {
  const uint4* src = reinterpret_cast<const uint4*>(&bp.lin[l]);
  for (int i = threadIdx.x >> 5; i < (int)(sizeof(DecodeLinear) / 16); i += blockDim.x >> 5) {
    const uint4 v = src[i];
    if ((threadIdx.x & 31) == 0) reinterpret_cast<uint4*>(dst)[i] = v;
  }
}

// Wait with a bound.  Once any wait of the CTA has run out, every later wait returns at once, so that
// all threads keep the same control flow and the kernel ends (with an error status and undefined output): no copy is
// issued any more, and the thread whose wait ran out sleeps until those in flight have landed, before the CTA's shared memory passes to
// another.  (Here, and plain barriers behind it: a look at `fail` at the end of each kernel and barriers that vote on it were 0.3 us a call.)
// A copy takes a microsecond or two, less than the hardware may suspend a waiting thread for: a limit as short as that is polled
// (`poll`, from the host: to look the limit up here is a trip to memory that no wait hides, 0.35 us a call).
__device__ __forceinline__ void decode_wait(uint32_t bar, uint32_t parity, volatile int* fail, bool poll) {
  auto done = [&] { return poll ? mbar_test_wait(bar, parity) : mbar_try_wait(bar, parity); };
  if (done() || *fail) return;
  const long long t0 = clock64();
  while (!done()) {
    if (*fail) return;
    if (clock64() - t0 > c_spin_cycles) {
      report_timeout(WHERE_OTHER);
      *fail = 1;
      for (int i = 0; i < 200; ++i) __nanosleep(1000);
      return;
    }
  }
}

__device__ __forceinline__ int quant_code(float x, float gamma) { return max(-128, min(127, __float2int_rn(__fmul_rn(x, gamma)))); }

// codes of eight consecutive values, in order, as two words
__device__ __forceinline__ void quant_codes8(const uint4& v, float gamma, uint32_t (&o)[2]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  o[0] = o[1] = 0u;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int q0 = quant_code(bf16lo(w[u]), gamma), q1 = quant_code(bf16hi(w[u]), gamma);
    o[u >> 1] |= ((uint32_t)(q0 & 0xFF) | ((uint32_t)(q1 & 0xFF) << 8)) << (16 * (u & 1));
  }
}
__device__ __forceinline__ double sum_squares(const uint4& v) {
  const double d0 = bf16lo(v.x), d1 = bf16hi(v.x), d2 = bf16lo(v.y), d3 = bf16hi(v.y);
  const double d4 = bf16lo(v.z), d5 = bf16hi(v.z), d6 = bf16lo(v.w), d7 = bf16hi(v.w);
  return ((d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3)) + ((d4 * d4 + d5 * d5) + (d6 * d6 + d7 * d7));
}

// Element (token m, hidden index j) of the expert product's token-side operand: step j / 32, lane 4 (m % 8) + (j % 32) / 8,
// 16-bit slot j % 8; hi = bf16(a), lo = bf16(a - hi).
__device__ __forceinline__ void store_h(const DecodeLinear& L, int m, int j, float a) {
  const int rsteps = (L.r + 31) >> 5;
  const __nv_bfloat16 hi = __float2bfloat16_rn(a), lo = __float2bfloat16_rn(a - __bfloat162float(hi));
  uint16_t* base = reinterpret_cast<uint16_t*>(L.hfrag);
  const int pos = (((m >> 3) * 2 * rsteps + (j >> 5)) * 32 + (m & 7) * 4 + ((j & 31) >> 3)) * 8 + (j & 7);
  base[pos] = __bfloat16_as_ushort(hi);
  base[pos + rsteps * 32 * 8] = __bfloat16_as_ushort(lo);
}

// Shared memory of k_decode_prep: the token's K bf16 values, the router rows of the CTA's experts, the norm's gains.  Where the three do
// not fit (rows of 25,600 values with more than eight experts and a norm), the gains stay in global memory and a CTA's two
// router rows take turns.
struct PrepPlan { uint32_t row, off_gain; int slots; bool lean; size_t bytes; };
constexpr size_t kDecodePrepSmemLimit = 200 * 1024;
__host__ __device__ inline PrepPlan prep_plan(int K, int E, bool norm) {
  PrepPlan p{};
  p.row = ((uint32_t)K * 2u + 255u) / 256u * 256u;             // the token, and what follows it
  p.slots = E > kPrepCluster ? 2 : E > 1 ? 1 : 0;
  p.off_gain = p.row * (1u + p.slots);
  p.bytes = p.off_gain + (norm ? p.row : 0u);
  p.lean = p.bytes > kDecodePrepSmemLimit;
  if (p.lean) {
    p.slots = E > 1 ? 1 : 0;
    p.bytes = p.row * (size_t)(1 + p.slots);
  }
  return p;
}

// grid (8, M, linears), one cluster per token
template <int CAP>
__global__ void __cluster_dims__(kPrepCluster, 1, 1) __maxnreg__(80) k_decode_prep(const __grid_constant__ DecodeBatch<CAP> bp) {
  extern __shared__ __align__(128) uint8_t prep_smem[];
  __shared__ DecodeLinear L;
  __shared__ __align__(8) uint64_t wr_bar;
  __shared__ double red_d[kPrepWarps];
  __shared__ float red_f[kPrepWarps];
  __shared__ __align__(16) float logit_sh[kMaxExperts];
  __shared__ int sum_sh[kPrepCluster][kPrepWarps];
  __shared__ int fail_sh;
  const int m = blockIdx.y, rank = blockIdx.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  copy_record(&L, bp, blockIdx.z);
  const bool poll = bp.poll;
  if (tid == 0) {
    fail_sh = 0;
    mbar_init(smem_u32(&wr_bar), 1);
    mbar_fence_init();
  }
  __syncthreads();
  if (m >= L.M) return;                                        // whole clusters
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  const int K = L.K, E = L.E, r = L.r;
  const int chunks = K >> 3;
  const uint32_t row_bytes = (uint32_t)K * 2u;
  uint4* xs4 = reinterpret_cast<uint4*>(prep_smem);
  const PrepPlan plan = prep_plan(K, E, L.norm_w != nullptr);
  const uint32_t off_wr = plan.row;
  uint4* gain4 = reinterpret_cast<uint4*>(prep_smem + plan.off_gain);   // unless plan.lean
  const int my_experts = E > 1 && rank < E ? (E - rank + kPrepCluster - 1) / kPrepCluster : 0;   // rank, rank + 8
  const int my_warps = min(my_experts, plan.slots);             // warps that multiply router rows
  // weights start towards L2 while the previous kernel is still running
  if (m == 0) {
    if (tid < my_experts) bulk_prefetch(L.Wr + (long long)(rank + tid * kPrepCluster) * chunks, row_bytes);
    if (L.norm_w && tid == 32 && rank == 0) bulk_prefetch(L.norm_w, row_bytes);
  }
  pdl_wait();                // X may come from the previous kernel; the buffers written here may still be read by it
  pdl_launch_dependents();   // from here on the kernels behind this one may start: what they read early is final
  if (tid == 0 && my_experts > 0) {
    mbar_expect_tx(smem_u32(&wr_bar), (uint32_t)my_warps * row_bytes);
    for (int i = 0; i < my_warps; ++i)
      bulk_load(smem_u32(prep_smem + off_wr) + (uint32_t)i * row_bytes, L.Wr + (long long)(rank + i * kPrepCluster) * chunks, row_bytes, smem_u32(&wr_bar));
  }

  // the token (and the norm's gains): all loads of a thread in flight together
  float amax = 0.f;
  double ss = 0.0;
  auto fold_amax = [&](const uint4& v) {
    amax = fmaxf(amax, fmaxf(fmaxf(fabsf(bf16lo(v.x)), fabsf(bf16hi(v.x))), fmaxf(fabsf(bf16lo(v.y)), fabsf(bf16hi(v.y)))));
    amax = fmaxf(amax, fmaxf(fmaxf(fabsf(bf16lo(v.z)), fabsf(bf16hi(v.z))), fmaxf(fabsf(bf16lo(v.w)), fabsf(bf16hi(v.w)))));
  };
  {
    const uint4* x4 = L.X + (long long)m * chunks;
    for (int c0 = tid; c0 < chunks; c0 += 4 * kPrepThreads) {
      uint4 v[4], g[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool in = c0 + u * kPrepThreads < chunks;
        v[u] = in ? __ldcg(x4 + c0 + u * kPrepThreads) : make_uint4(0u, 0u, 0u, 0u);
        if (L.norm_w && in && !plan.lean) g[u] = __ldcg(L.norm_w + c0 + u * kPrepThreads);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (c0 + u * kPrepThreads < chunks) {
          xs4[c0 + u * kPrepThreads] = v[u];
          if (L.norm_w) {
            if (!plan.lean) gain4[c0 + u * kPrepThreads] = g[u];
            ss += sum_squares(v[u]);
          } else {
            fold_amax(v[u]);
          }
        }
      }
    }
  }
  if (L.norm_w) {
    // RMSNorm fused in front of the quantiser (App. A): mean of squares and its reciprocal root in fp64 (thread sums
    // in ascending chunk order, then a fixed tree), the factor rounded once to fp32; the token in shared memory is
    // replaced by bf16(fp32(fp32(x s) w)), which every later step reads.
    for (int d = 16; d > 0; d >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, d);
    if (lane == 0) red_d[warp] = ss;
    __syncthreads();
    double tot = 0.0;
#pragma unroll
    for (int w = 0; w < kPrepWarps; ++w) tot += red_d[w];
    const float s = (float)(1.0 / sqrt(tot / (double)K + (double)L.norm_eps));
    for (int c = tid; c < chunks; c += kPrepThreads) {   // each thread reads back the chunks it wrote itself
      const uint4 v = rms_apply(xs4[c], s, plan.lean ? __ldcg(L.norm_w + c) : gain4[c]);
      xs4[c] = v;
      fold_amax(v);
    }
  }
  for (int d = 16; d > 0; d >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, d));
  if (lane == 0) red_f[warp] = amax;
  __syncthreads();                                             // the token and the maxima are visible
  amax = red_f[0];
#pragma unroll
  for (int w = 1; w < kPrepWarps; ++w) amax = fmaxf(amax, red_f[w]);
  const float gamma = __fdiv_rn(kActQmax, fmaxf(amax, kActAmaxFloor));

  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");  // every CTA of the cluster is running
  // router: the same pinned fp32 order as the training path (lane j owns the chunks c = j mod 32, ascending,
  // fused multiply-add; butterfly 16, 8, 4, 2, 1), one warp per expert of this CTA; the cluster exchanges the logits
  if (warp < my_warps) {
    const uint4* wrow = reinterpret_cast<const uint4*>(prep_smem + off_wr) + (size_t)warp * chunks;
    for (int k = warp; k < my_experts; k += my_warps) {           // once, unless two rows share a place
      decode_wait(smem_u32(&wr_bar), k == warp ? 0 : 1, &fail_sh, poll);
      float acc = 0.f;
      auto fold = [&](const uint4& xv, const uint4& wv) {
        acc = fmaf(bf16lo(xv.x), bf16lo(wv.x), acc); acc = fmaf(bf16hi(xv.x), bf16hi(wv.x), acc);
        acc = fmaf(bf16lo(xv.y), bf16lo(wv.y), acc); acc = fmaf(bf16hi(xv.y), bf16hi(wv.y), acc);
        acc = fmaf(bf16lo(xv.z), bf16lo(wv.z), acc); acc = fmaf(bf16hi(xv.z), bf16hi(wv.z), acc);
        acc = fmaf(bf16lo(xv.w), bf16lo(wv.w), acc); acc = fmaf(bf16hi(xv.w), bf16hi(wv.w), acc);
      };
      int c = lane;
      for (; c + 96 < chunks; c += 128) {
        uint4 wv[4], xv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) { wv[u] = wrow[c + 32 * u]; xv[u] = xs4[c + 32 * u]; }
#pragma unroll
        for (int u = 0; u < 4; ++u) fold(xv[u], wv[u]);
      }
      for (; c < chunks; c += 32) fold(xs4[c], wrow[c]);
      for (int d = 16; d > 0; d >>= 1) acc = acc + __shfl_xor_sync(0xffffffffu, acc, d);
      if (lane == 0)
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cluster_map(smem_u32(&logit_sh[rank + k * kPrepCluster]), 0)), "f"(acc) : "memory");
      if (k + my_warps < my_experts) {
        __syncwarp();
        if (lane == 0 && !*(volatile int*)&fail_sh) {
          mbar_expect_tx(smem_u32(&wr_bar), row_bytes);
          bulk_load(smem_u32(wrow), L.Wr + (long long)(rank + (k + my_warps) * kPrepCluster) * chunks, row_bytes, smem_u32(&wr_bar));
        }
      }
    }
  } else {
    // meanwhile the other warps: this CTA's eighth of the token's codes (Eq. 7-9), in fragment order -- an item is one 16-byte
    // piece (chunk and half, quad index) -- and, for the INT8 branch, in natural order
    const int nhalves = 2 * ((K + 127) >> 7), first = my_warps * 32, nthr = kPrepThreads - first;
    const int group = m >> 3, g = m & 7, mg = min(8, L.M - 8 * group);
    const int i_lo = nhalves * 4 * rank / kPrepCluster, i_hi = nhalves * 4 * (rank + 1) / kPrepCluster;
    uint4* dst = L.qfrag + (long long)group * nhalves * 32 + g * 4;
    const uint16_t* xs = reinterpret_cast<const uint16_t*>(prep_smem);
    int rowsum = 0;
    for (int i = i_lo + tid - first; i < i_hi; i += nthr) {
      const int ip = i >> 2, c = i & 3;
      uint32_t w[4];
#pragma unroll
      for (int reg = 0; reg < 4; ++reg) {
        const int base = 128 * (ip >> 1) + 32 * c + 4 * (ip & 1) + reg;
        w[reg] = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int q = base + 8 * j < K ? quant_code(bf16_bits_to_float(xs[base + 8 * j]), gamma) : 0;
          w[reg] |= (uint32_t)(q & 0xFF) << (8 * j);
          rowsum += q;
        }
      }
      dst[(long long)ip * mg * 4 + c] = make_uint4(w[0], w[1], w[2], w[3]);
    }
    for (int d = 16; d > 0; d >>= 1) rowsum += __shfl_xor_sync(0xffffffffu, rowsum, d);
    if (lane == 0)
      asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(cluster_map(smem_u32(&sum_sh[rank][warp]), 0)), "r"(rowsum) : "memory");
    if (L.A8) {
      const int c_lo = chunks * rank / kPrepCluster, c_hi = chunks * (rank + 1) / kPrepCluster;
      for (int c = c_lo + tid - first; c < c_hi; c += nthr) {
        uint32_t o[2];
        quant_codes8(xs4[c], gamma, o);
        reinterpret_cast<uint2*>(L.xn)[(long long)m * chunks + c] = make_uint2(o[0], o[1]);
      }
    } else if (L.norm_w && r > 0) {
      const int c_lo = chunks * rank / kPrepCluster, c_hi = chunks * (rank + 1) / kPrepCluster;
      for (int c = c_lo + tid - first; c < c_hi; c += nthr) reinterpret_cast<uint4*>(L.xn)[(long long)m * chunks + c] = xs4[c];
    }
  }
  cluster_sync_all();
  if (rank == 0 && warp == 0) {
    // lane e: expert e (lowest index on ties); the lanes also add up the code sums of the cluster's warps
    int best = 0;
    float gate = 1.0f;
    if (E > 1) {
      const float lg = lane < E ? logit_sh[lane] : -INFINITY;
      float lmax = lg;
      for (int d = 16; d > 0; d >>= 1) lmax = fmaxf(lmax, __shfl_xor_sync(0xffffffffu, lmax, d));
      best = __ffs(__ballot_sync(0xffffffffu, lane < E && lg == lmax)) - 1;
      // as the training path's comparison of one logit after the other has it: expert 0 if its own logit is not a number
      if (best < 0 || isnan(logit_sh[0])) best = 0;
      const float pe = lane < E ? expf(lg - lmax) : 0.f;
      float den = pe;
      for (int d = 16; d > 0; d >>= 1) den += __shfl_xor_sync(0xffffffffu, den, d);
      gate = __shfl_sync(0xffffffffu, pe, best) * (1.0f / den);
    }
    int tot = 0;
#pragma unroll
    for (int i = 0; i < kPrepCluster * kPrepWarps / 32; ++i) {
      const int k = i * 32 + lane, rk = k / kPrepWarps, w = k % kPrepWarps;
      const int routed = E > 1 && rk < E ? (E - rk + kPrepCluster - 1) / kPrepCluster : 0;
      if (w >= min(routed, plan.slots)) tot += sum_sh[rk][w];
    }
    for (int d = 16; d > 0; d >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, d);
    if (lane == 0) L.info[m] = DecodeTokInfo{best, gate, gamma, tot};   // after a failed wait too: an expert that exists
  }
}

// ---------------------------------------------------------------------------
// k_decode_hidden: h = A_e x, expert by expert, so that a row of A_e is read once for all tokens of its expert (eight experts,
// sixteen tokens: about six experts in use).  A cluster of one, two or four CTAs per (linear, k-th expert in use, 16 hidden
// rows), as many as make about one CTA per SM: k_decode_main's has to fit beside it.  K is cut into 32 shares whatever the
// cluster's size; a warp contracts over its shares one after the other on mma.sync (bf16, or s8 for the INT8 branch), rows of A
// as the 16-row operand straight from global memory (a lane takes 16 consecutive bytes: the order of the contraction index is
// the same on both sides), the expert's tokens as columns; the sums meet in the first CTA's shared memory and are added in
// the order of the shares.
// ---------------------------------------------------------------------------
__device__ __forceinline__ void mma_s8s8(int (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// Steps [st_lo, st_hi) of 64 bytes per row.  Rows of `pitch` 16-byte pieces; r0, r1, x0, x1 point at this lane's piece of step 0
// (x0, x1: its columns' tokens, null for columns without one).
// TWO: the expert has more than eight tokens.
template <bool INT8, bool TWO>
__device__ __forceinline__ void hidden_walk(const uint4* r0, const uint4* r1, const uint4* x0, const uint4* x1, int st_lo, int st_hi, int last, int c,
                                            uint32_t (&z0)[4], uint32_t (&z1)[4]) {
  constexpr int U = TWO ? 3 : 4;                               // steps in flight, as many as 80 registers hold
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  auto mma = [](uint32_t (&z)[4], const uint4& a, const uint4& b, const uint4& v) {
    if (INT8) {
      int (&d)[4] = reinterpret_cast<int(&)[4]>(z);
      mma_s8s8(d, a.x, b.x, a.y, b.y, v.x, v.y);
      mma_s8s8(d, a.z, b.z, a.w, b.w, v.z, v.w);
    } else {
      float (&d)[4] = reinterpret_cast<float(&)[4]>(z);
      mma_bf16(d, a.x, b.x, a.y, b.y, v.x, v.y);
      mma_bf16(d, a.z, b.z, a.w, b.w, v.z, v.w);
    }
  };
  for (int st = st_lo; st < st_hi; st += U) {
    uint4 w0[U], w1[U], v[U], v1[TWO ? U : 1];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool in = st + u < st_hi && (st + u) * 4 + c < last;   // a row's last step may be half a step (INT8, K % 64 = 32)
      w0[u] = in ? __ldg(r0 + (st + u) * 4) : zero;
      w1[u] = in ? __ldg(r1 + (st + u) * 4) : zero;
      v[u] = in && x0 ? __ldcg(x0 + (st + u) * 4) : zero;
      if (TWO) v1[u] = in && x1 ? __ldcg(x1 + (st + u) * 4) : zero;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) mma(z0, w0[u], w1[u], v[u]);
    if (TWO) {
#pragma unroll
      for (int u = 0; u < U; ++u) mma(z1, w0[u], w1[u], v1[u]);
    }
  }
}

template <int CAP>
__global__ void __maxnreg__(80) k_decode_hidden(const __grid_constant__ DecodeBatch<CAP> bp) {
  __shared__ DecodeLinear L;
  __shared__ uint32_t red[kHiddenSplit][16][17];               // used in the cluster's first CTA
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cs = bp.hidden_cluster, rank = (int)cluster_rank(), group = (int)blockIdx.x / cs;
  int l = 0;
  for (int i = 1; i < bp.n; ++i)
    if (bp.lin[i].r > 0 && group >= bp.lin[i].hidden0) l = i;
  while (bp.lin[l].r <= 0) ++l;
  copy_record(&L, bp, l);
  __syncthreads();
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  const int K = L.K, r = L.r, M = L.M;
  const bool int8 = L.A8 != nullptr;
  const int pitch = int8 ? K >> 4 : K >> 3, steps = (pitch + 3) >> 2;
  const int tiles = (r + 15) >> 4, local = group - L.hidden0;
  const int slot = local / tiles, tile = local - slot * tiles, j0 = tile * 16;   // the slot-th expert in use
  const int g = lane >> 2, c = lane & 3;
  const long long row0 = (long long)j0 * pitch, expert_pitch = (long long)r * pitch;
  const uint4* base = int8 ? reinterpret_cast<const uint4*>(L.A8) : reinterpret_cast<const uint4*>(L.A);
  // with as many tokens as experts most experts are in use: the rows start towards L2 before it is known which
  if (M >= L.E) {
    const uint32_t bytes = (uint32_t)min(16, r - j0) * (uint32_t)pitch * 16u;
    for (uint32_t at = (rank * kHiddenThreads + tid) * 4096u; at < bytes; at += cs * kHiddenThreads * 4096u)
      bulk_prefetch(reinterpret_cast<const uint8_t*>(base + slot * expert_pitch + row0) + at, min(4096u, bytes - at));
  }
  pdl_wait();
  pdl_launch_dependents();   // k_decode_main may read k_decode_prep's results from here on
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");  // every CTA of the cluster is running
  const int my_e = lane < M ? __ldcg(&L.info[lane].expert) : -1;
  unsigned used = __reduce_or_sync(0xffffffffu, my_e >= 0 ? 1u << (my_e & 15) : 0u);
  for (int k = 0; k < slot; ++k) used &= used - 1;
  if (used == 0u) return;                                      // the whole cluster: fewer experts are in use
  const int e = __ffs(used) - 1;
  const unsigned mine = __ballot_sync(0xffffffffu, my_e == e);
  const int cnt = __popc(mine);
  // up to sixteen tokens: columns 0-7 and 8-15
  unsigned left = mine;
  for (int k = 0; k < g; ++k) left &= left - 1;
  const int t0 = g < cnt ? __ffs(left) - 1 : -1;
  for (int k = 0; k < 8; ++k) left &= left - 1;
  const int t1 = g + 8 < cnt ? __ffs(left) - 1 : -1;
  const uint4* x = (int8 || L.norm_w ? reinterpret_cast<const uint4*>(L.xn) : L.X) + c;
  const uint4* x0 = t0 >= 0 ? x + (long long)t0 * pitch : nullptr;
  const uint4* x1 = t1 >= 0 ? x + (long long)t1 * pitch : nullptr;
  const uint4* rows = base + e * expert_pitch + row0 + c;
  const uint4 *r0 = rows + (long long)g * pitch, *r1 = rows + (long long)(j0 + g + 8 < r ? g + 8 : g) * pitch;
  // where k_decode_main asks for the rows of B_e late, they start towards L2 (512-byte pieces)
  if (bp.rows_early && !int8) {
    const int total = (L.N >> 5) * (r >> 3), per = (total + tiles - 1) / tiles, lo = per * tile, hi = min(total, lo + per);
    const uint8_t* b = reinterpret_cast<const uint8_t*>(L.B) + (long long)e * total * 512;
    for (int at = lo + (rank * kHiddenThreads + tid) * 8; at < hi; at += cs * kHiddenThreads * 8) bulk_prefetch(b + (long long)at * 512, (uint32_t)min(8, hi - at) * 512u);
  }
  const bool two = cnt > 8;
  for (int v = rank * kHiddenWarps + warp; v < kHiddenSplit; v += cs * kHiddenWarps) {
    uint32_t z0[4] = {0u, 0u, 0u, 0u}, z1[4] = {0u, 0u, 0u, 0u};   // fp32 or int32 sums; zero is the same word
    const int st_lo = steps * v / kHiddenSplit, st_hi = steps * (v + 1) / kHiddenSplit;
    if (int8) {
      if (two) hidden_walk<true, true>(r0, r1, x0, x1, st_lo, st_hi, pitch, c, z0, z1);
      else hidden_walk<true, false>(r0, r1, x0, x1, st_lo, st_hi, pitch, c, z0, z1);
    } else {
      if (two) hidden_walk<false, true>(r0, r1, x0, x1, st_lo, st_hi, pitch, c, z0, z1);
      else hidden_walk<false, false>(r0, r1, x0, x1, st_lo, st_hi, pitch, c, z0, z1);
    }
    const uint32_t to = cluster_map(smem_u32(&red[v][0][0]), 0);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t at = to + 4u * ((g + (u >> 1) * 8) * 17 + 2 * c + (u & 1));
      asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(at), "r"(z0[u]) : "memory");
      if (two) asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(at + 32u), "r"(z1[u]) : "memory");
    }
  }
  cluster_sync_all();
  if (rank == 0) {
    const int row = tid & 15, col = tid >> 4;
    if (col < cnt && j0 + row < r) {
      unsigned m = mine;
      for (int k = 0; k < col; ++k) m &= m - 1;
      const int t = __ffs(m) - 1;
      if (int8) {
        int a = 0;
#pragma unroll
        for (int w = 0; w < kHiddenSplit; ++w) a += (int)red[w][row][col];
        L.h_int[(long long)t * r + j0 + row] = a;
      } else {
        float a = 0.f;
#pragma unroll
        for (int w = 0; w < kHiddenSplit; ++w) a += __uint_as_float(red[w][row][col]);
        store_h(L, t, j0 + row, a);
      }
    }
  }
}

// ---------------------------------------------------------------------------
// k_decode_main.  A CTA walks its share of the units in passes of up to kMaxPassUnits units of one linear.  The sign bits
// of a pass sit in shared memory as [chunk of 128 k][feature of the pass][16 bytes]; with the streaming layout they arrive
// by bulk copies, one pass ahead, otherwise through registers.  1-bit product: a warp works on two tiles of 16 features and a
// slice of the contraction; the slices' sums (integers) are added up in shared memory.  Expert product: the rows of B_e of
// one tile are one contiguous piece, fetched by a bulk copy; a warp takes whole (expert, tile) items.
// ---------------------------------------------------------------------------
struct DecodePass { int l, unit, nu; };   // linear; first unit within it; units (0: no pass)

// Chunks [c_lo, c_hi) of the pass's sign bits, tiles of 16 features at row0 and (T = 2) row0 + 16, against the codes; q: fragments
// whose first chunk is q_c0, q_chunks of them per group of eight tokens.  G: groups of eight tokens.  Shared memory bounds this
// loop (a 16-byte load of a warp takes four of the cycles the SM has for all its warps, however few different bytes it reads):
// hence one weight word per lane and two tiles per set of codes.
template <int G, int T>
__device__ __forceinline__ void main_bits(const uint32_t* bits_s, int rows, int row0, const uint4* q, int q_c0, int q_chunks, int M, int c_lo, int c_hi, int lane,
                                          int (&a1)[T][G][4], int (&a16)[T][G][4]) {
  const int g = lane >> 2, c = lane & 3;
  const uint32_t* w = bits_s + ((size_t)c_lo * rows + row0 + g) * 4 + c;
  const int mg0 = min(8, M), mg1 = M - 8;
  const uint4* q0 = q + (size_t)(c_lo - q_c0) * 2 * mg0 * 4 + min(g, mg0 - 1) * 4 + c;
  const uint4* q1 = G > 1 ? q + (size_t)q_chunks * 64 + (size_t)(c_lo - q_c0) * 2 * mg1 * 4 + min(g, mg1 - 1) * 4 + c : q;
#pragma unroll 2
  for (int ch = c_lo; ch < c_hi; ++ch) {
    uint32_t u[T], v[T];
#pragma unroll
    for (int t = 0; t < T; ++t) { u[t] = w[t * 64]; v[t] = w[t * 64 + 32]; }
    w += rows * 4;
    uint4 qq[G][2];
    qq[0][0] = q0[0]; qq[0][1] = q0[mg0 * 4];
    q0 += mg0 * 8;
    if (G > 1) { qq[G - 1][0] = q1[0]; qq[G - 1][1] = q1[mg1 * 4]; q1 += mg1 * 8; }
#pragma unroll
    for (int t = 0; t < T; ++t) {
      uint32_t m1[4][2], m16[4][2];
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        const uint32_t x = u[t] >> b, y = v[t] >> b;
        m1[b][0] = x & 0x01010101u; m1[b][1] = y & 0x01010101u;
        m16[b][0] = x & 0x10101010u; m16[b][1] = y & 0x10101010u;
      }
      const uint32_t A0[4] = {m1[0][0], m1[0][1], m1[1][0], m1[1][1]}, A1[4] = {m1[2][0], m1[2][1], m1[3][0], m1[3][1]};
      const uint32_t B0[4] = {m16[0][0], m16[0][1], m16[1][0], m16[1][1]}, B1[4] = {m16[2][0], m16[2][1], m16[3][0], m16[3][1]};
#pragma unroll
      for (int G_ = 0; G_ < G; ++G_) {
        mma_u8s8(a1[t][G_], A0, qq[G_][0].x, qq[G_][0].y);
        mma_u8s8(a16[t][G_], B0, qq[G_][1].x, qq[G_][1].y);
        mma_u8s8(a1[t][G_], A1, qq[G_][0].z, qq[G_][0].w);
        mma_u8s8(a16[t][G_], B1, qq[G_][1].z, qq[G_][1].w);
      }
    }
  }
}

// One (expert, tile) item of the expert product: b_s = the expert's rows of the tile (16 rows of r values), order[0 .. cnt) =
// its tokens.  The columns of the product are those tokens; up to four of them sit beside one another with the leading halves of
// h in columns 0-3 and the trailing ones in 4-7, more take two products per step.  A token has one expert, so its sums go
// straight to out[token][16 features].
__device__ __forceinline__ void main_expert(const uint4* b_s, int r, const uint8_t* order, int cnt, const uint4* h_s, int lane, float* out) {
  const int g = lane >> 2, c = lane & 3;
  const int steps = (r + 31) >> 5, r8 = r >> 3;
  const bool packed = cnt <= 4;
  const uint4 *r0 = b_s + g * r8 + c, *r1 = b_s + (g + 8) * r8 + c;
  for (int first = 0; first < cnt; first += 8) {
    const int n = min(8, cnt - first), col = packed ? g & 3 : g;
    const bool in = col < n;
    // h of token t, plane: piece ((t / 8) * 2 + plane) * steps * 32 + step * 32 + 4 (t % 8) + c
    const int t = in ? order[first + col] : 0;
    const uint4* h0 = h_s + (((t >> 3) * 2 + (packed ? g >> 2 : 0)) * steps) * 32 + 4 * (t & 7) + c;
    const uint4* h1 = h0 + steps * 32;
    float z0[4] = {0.f, 0.f, 0.f, 0.f}, z1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 2
    for (int st = 0; st < steps; ++st) {
      uint4 w0 = make_uint4(0u, 0u, 0u, 0u), w1 = w0, hh = w0, hl = w0;
      if (4 * st + c < r8) {
        w0 = r0[4 * st]; w1 = r1[4 * st];
        if (in) { hh = h0[st * 32]; if (!packed) hl = h1[st * 32]; }
      }
      mma_bf16(z0, w0.x, w1.x, w0.y, w1.y, hh.x, hh.y);
      mma_bf16(z1, w0.z, w1.z, w0.w, w1.w, hh.z, hh.w);
      if (!packed) {
        mma_bf16(z0, w0.x, w1.x, w0.y, w1.y, hl.x, hl.y);
        mma_bf16(z1, w0.z, w1.z, w0.w, w1.w, hl.z, hl.w);
      }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {                              // columns 2 c and 2 c + 1; features g and g + 8
      float v0 = z0[u] + z1[u], v1 = z0[u + 2] + z1[u + 2];
      if (packed) { v0 += __shfl_xor_sync(0xffffffffu, v0, 2); v1 += __shfl_xor_sync(0xffffffffu, v1, 2); }
      if (2 * c + u < n) {
        float* o = out + order[first + 2 * c + u] * 16 + g;
        o[0] = v0; o[8] = v1;
      }
    }
  }
}

// G: groups of eight tokens the launch's linears have at most; a linear of a single group runs the one-group code
template <int CAP, int G>
__global__ void __maxnreg__(88) k_decode_main(const __grid_constant__ DecodeBatch<CAP> bp) {
  extern __shared__ __align__(128) uint8_t smem[];
  __shared__ DecodeLinear lin_sh[2];       // records of the current linear and the next one (linear l in slot l & 1)
  __shared__ __align__(8) uint64_t bars[2 + kMaxRows];     // sign bits (two buffers), expert rows
  __shared__ DecodeTokInfo tok[kDecodeMaxTokens];
  __shared__ float gh_sh[kDecodeMaxTokens], deq_sh[kDecodeMaxTokens];
  // the linear's experts in use, in ascending order: index, first token in `order_sh`, number of tokens
  __shared__ int used_sh, expert_sh[kDecodeMaxTokens], first_sh[kDecodeMaxTokens], count_sh[kDecodeMaxTokens];
  __shared__ uint8_t order_sh[kDecodeMaxTokens];
  __shared__ float be_sh[kMaxPassUnits * kUnit], al_sh[kMaxPassUnits * kUnit];
  __shared__ int fail_sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int u_lo = (int)((long long)bp.units * blockIdx.x / gridDim.x), u_hi = (int)((long long)bp.units * (blockIdx.x + 1) / gridDim.x);
  int l_at = 0;
  while (bp.unit0[l_at + 1] <= u_lo) ++l_at;
  copy_record(&lin_sh[l_at & 1], bp, l_at);
  if (l_at + 1 < bp.n && bp.unit0[l_at + 1] < u_hi) copy_record(&lin_sh[(l_at + 1) & 1], bp, l_at + 1);
  const int nbuf = bp.nbuf, buf_bytes = bp.buf_bytes, q_chunks = bp.q_chunks, MT = bp.red_tokens, off_h = bp.off_h;
  const bool poll = bp.poll;
  if (tid == 0) fail_sh = 0;
  if (tid < 2 + kMaxRows) {
    mbar_init(smem_u32(&bars[tid]), 1);
    mbar_fence_init();
  }
  __syncthreads();
  pdl_launch_dependents();
  // the pass that begins at launch-wide unit u, known to belong to linear l or a later one
  auto pass_at = [&](int u, int l) {
    DecodePass p{l, 0, 0};
    if (u >= u_hi) return p;
    while (bp.unit0[p.l + 1] <= u) ++p.l;
    const DecodeLinear& L = lin_sh[p.l & 1];
    const int cap = max(1, min(bp.pass_units, buf_bytes / (256 * ((L.K + 127) >> 7))));
    const int rem = min(u_hi, bp.unit0[p.l + 1]) - u, npass = (rem + cap - 1) / cap;
    p.unit = u - bp.unit0[p.l];
    p.nu = (rem + npass - 1) / npass;
    return p;
  };
  // bulk copies of a pass's sign bits, issued by all warps; a pass is one or two runs within 128-feature groups, one copy per
  // chunk and run
  auto fetch_bits = [&](const DecodePass& p, int b) {
    if (p.nu == 0) return;
    const DecodeLinear& L = lin_sh[p.l & 1];
    if (!L.bits_il) return;
    const int C = (L.K + 127) >> 7;
    const uint32_t dst = smem_u32(smem) + (uint32_t)b * buf_bytes, bar = smem_u32(&bars[b]);
    if (tid == 0) mbar_expect_tx(bar, (uint32_t)p.nu * 256u * (uint32_t)C);   // (copies may land before: the phase completes when both agree)
    for (int done = 0; done < p.nu;) {
      const int unit = p.unit + done, run = min(p.nu - done, 8 - (unit & 7));
      const uint4* src = L.bits_il + (long long)(unit >> 3) * C * 128 + (unit & 7) * 16;
      for (int c = warp + kMainWarps * lane; c < C; c += 32 * kMainWarps)
        bulk_load(dst + ((uint32_t)c * p.nu + done) * 256u, src + (long long)c * 128, (uint32_t)run * 256u, bar);
      done += run;
    }
  };
  // per-feature factors of a pass
  auto load_scales = [&](const DecodePass& p) {
    const DecodeLinear& L = lin_sh[p.l & 1];
    if (p.nu == 0) return;
    if (tid < p.nu * kUnit) be_sh[tid] = __ldg(L.beta + (long long)(p.unit * kUnit + tid) * L.sstride);
    else if (tid >= 256 && tid - 256 < p.nu * kUnit && L.r > 0) al_sh[tid - 256] = __ldg(L.alpha + (long long)(p.unit * kUnit + tid - 256) * L.sstride);
  };
  DecodePass cur = pass_at(u_lo, l_at);
  int u_next = u_lo + cur.nu;
  DecodePass nxt = nbuf > 1 ? pass_at(u_next, cur.l) : DecodePass{0, 0, 0};
  fetch_bits(cur, 0);
  if (nbuf > 1) fetch_bits(nxt, 1);
  load_scales(cur);
  bool waited = false;                     // for the kernel before this one
  if (!bp.early) { pdl_wait(); waited = true; }
  const uint4* q_loaded = nullptr;
  uint32_t phase[2] = {0u, 0u}, row_phase = 0u;
  uint4* q_s = reinterpret_cast<uint4*>(smem + bp.off_q);
  uint4* h_s = reinterpret_cast<uint4*>(smem + off_h);
  int8_t* qh_s = reinterpret_cast<int8_t*>(smem + off_h);
  int* red_i = reinterpret_cast<int*>(smem + bp.off_red);        // [tile][token][16 features]
  float* red_z = reinterpret_cast<float*>(red_i + bp.pass_units * MT * 16);   // [tile][token][16]
  int loaded_l = -1;
  for (int b = 0; cur.nu > 0;) {
    const DecodeLinear& L = lin_sh[cur.l & 1];
    const int M = L.M, K = L.K, N = L.N, r = L.r;
    const int C = (K + 127) >> 7, rsteps = (r + 31) >> 5;
    const int rows = cur.nu * kUnit, n0 = cur.unit * kUnit;
    uint8_t* bits_s = smem + (size_t)b * buf_bytes;
    const float lam = __ldg(L.w_scales);
    const bool whole = q_chunks >= C;
    // codes of the chunks [ch0, ch1) into shared memory: group 0 first, group 1 at q_chunks * 64
    auto load_codes = [&](int ch0, int ch1) {
      const int mg0 = min(8, M), n0q = (ch1 - ch0) * mg0 * 8, n1q = (ch1 - ch0) * (M - 8) * 8;
      const uint4 *s0 = L.qfrag + (long long)ch0 * mg0 * 8, *s1 = L.qfrag + (long long)C * 64 + (long long)ch0 * (M - 8) * 8;
      const int n = n0q + (M > 8 ? n1q : 0);
      for (int i0 = tid; i0 < n; i0 += 4 * kMainThreads) {
        uint4 v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * kMainThreads;
          v[u] = i < n0q ? __ldcg(s0 + i) : i < n ? __ldcg(s1 + i - n0q) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * kMainThreads;
          if (i < n) q_s[i < n0q ? i : q_chunks * 64 + i - n0q] = v[u];
        }
      }
    };
    const bool new_linear = cur.l != loaded_l;
    loaded_l = cur.l;
    if (new_linear && warp == kMainWarps - 1) {
      DecodeTokInfo t{-1, 0.f, 1.f, 0};
      if (lane < M) {
        const int4 a = __ldcg(reinterpret_cast<const int4*>(L.info) + lane);
        t = DecodeTokInfo{a.x & 15, __int_as_float(a.y), __int_as_float(a.z), a.w};
        tok[lane] = t;
        deq_sh[lane] = __fdiv_rn(lam, t.gamma);
      }
      // tokens by expert: a token's place is the number of tokens with a lower expert, or the same one and a lower index
      int place = 0;
      const unsigned used = __reduce_or_sync(0xffffffffu, lane < M ? 1u << t.expert : 0u);
      for (int i = 0; i < M; ++i) {
        const int e = __shfl_sync(0xffffffffu, t.expert, i);
        place += e < t.expert || (e == t.expert && i < lane);
      }
      const unsigned same = __match_any_sync(0xffffffffu, t.expert);
      if (lane < M) {
        order_sh[place] = (uint8_t)lane;
        if ((same & ((1u << lane) - 1u)) == 0u) {                // the expert's first token
          const int k = __popc(used & ((1u << t.expert) - 1u));
          expert_sh[k] = t.expert; first_sh[k] = place; count_sh[k] = __popc(same);
        }
      }
      if (lane == 0) used_sh = r > 0 ? __popc(used) : 0;
    }
    if (whole && q_loaded != L.qfrag) { load_codes(0, C); q_loaded = L.qfrag; }
    for (int i = tid; i < cur.nu * MT * 16; i += kMainThreads) red_i[i] = 0;
    if (!L.bits_il) {
      // natural layout [N, K/32]: four lanes take four consecutive chunks of a row
      const int KW = K >> 5;
      for (int i = tid; i < rows * ((C + 3) & ~3); i += kMainThreads) {
        const int ci = i & 3, row = (i >> 2) % rows, c = ((i >> 2) / rows) * 4 + ci;
        if (c < C) {
          const uint32_t* src = L.bits + (long long)(n0 + row) * KW + 4 * c;
          uint32_t w[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) w[u] = 4 * c + u < KW ? __ldg(src + u) : 0u;
          reinterpret_cast<uint4*>(bits_s)[(size_t)c * rows + row] = make_uint4(w[0], w[1], w[2], w[3]);
        }
      }
    }
    __syncthreads();
    // Expert rows: every warp has places of its own and takes every W-th (expert, tile) item.  The places either lie apart, and the
    // rows set out now, beside the 1-bit product; or over what the product has used by then -- this pass's sign bits, and in the CTA's
    // last pass all buffers and the codes.
    const bool rows_now = r > 0 && !L.A8, own = bp.row_slots > 0, last = u_next >= u_hi && (nbuf == 1 || nxt.nu == 0);
    const uint32_t item_bytes = 32u * (uint32_t)max(r, 1);
    const int tiles = cur.nu;
    uint8_t* ring = smem + bp.off_rows;
    int W = 1, per = 1, items = 0;                               // warps that take items, places of each, items
    auto issue = [&](int i, int j) {                             // item i into this warp's place j
      if (lane == 0) {
        const int ei = i / tiles, t = i - ei * tiles;
        const uint32_t bar = smem_u32(&bars[2 + warp * kWarpRows + j]);   // barriers belong to a warp, whatever the places of a pass
        mbar_expect_tx(bar, item_bytes);
        bulk_load(smem_u32(ring) + (uint32_t)(warp * per + j) * item_bytes, L.B + ((long long)expert_sh[ei] * N + n0 + t * 16) * r, item_bytes, bar);
      }
    };
    auto ask = [&](int slots) {
      W = min(kMainWarps, slots); per = slots < kMaxRows ? 1 : kWarpRows; items = warp < W ? used_sh * tiles : 0;
      for (int j = 0; j < per && warp + W * j < items; ++j) issue(warp + W * j, j);
    };
    if (rows_now && own) ask(bp.row_slots);
    // ---- 1-bit product
    const int pairs = (tiles + 1) >> 1, S = kMainWarps / pairs;   // at most 4 pairs of tiles
    const int sl = warp / pairs, tile = 2 * (warp - sl * pairs);
    if (L.bits_il) {
      decode_wait(smem_u32(&bars[b]), phase[b], &fail_sh, poll);
      phase[b] ^= 1u;
    }
    {
      auto bits = [&](auto groups, auto per_warp) {
        constexpr int GG = decltype(groups)::value, T = decltype(per_warp)::value;
        int a1[T][GG][4], a16[T][GG][4];
#pragma unroll
        for (int t = 0; t < T; ++t)
#pragma unroll
          for (int G_ = 0; G_ < GG; ++G_)
#pragma unroll
            for (int u = 0; u < 4; ++u) { a1[t][G_][u] = 0; a16[t][G_][u] = 0; }
        for (int ch0 = 0; ch0 < C; ch0 += q_chunks) {            // once, unless the codes of all of K do not fit
          const int ch1 = min(C, ch0 + q_chunks);
          if (!whole) {
            __syncthreads();
            load_codes(ch0, ch1);
            __syncthreads();
          }
          if (sl < S)
            main_bits<GG, T>(reinterpret_cast<const uint32_t*>(bits_s), rows, tile * 16, q_s, ch0, q_chunks, M, ch0 + (ch1 - ch0) * sl / S,
                             ch0 + (ch1 - ch0) * (sl + 1) / S, lane, a1, a16);
        }
        const int g = lane >> 2, c = lane & 3;
        if (sl < S) {
#pragma unroll
          for (int t = 0; t < T; ++t) {
            if (tile + t < tiles) {
#pragma unroll
              for (int G_ = 0; G_ < GG; ++G_)
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                  const int m = 8 * G_ + 2 * c + (u & 1);
                  // the weight-16 sums are exact multiples of 16; integer sums do not depend on the order of the slices
                  if (m < M) atomicAdd(red_i + ((tile + t) * MT + m) * 16 + g + (u >> 1) * 8, a1[t][G_][u] + (a16[t][G_][u] >> 4));
                }
            }
          }
        }
      };
      using One = std::integral_constant<int, 1>;
      using Two = std::integral_constant<int, 2>;
      if (G > 1 && M > 8) { if (tiles > 1) bits(std::integral_constant<int, G>{}, Two{}); else bits(std::integral_constant<int, G>{}, One{}); }
      else { if (tiles > 1) bits(One{}, Two{}); else bits(One{}, One{}); }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // what plain stores filled may be overwritten by bulk copies
    __syncthreads();                                             // the sign bits of this pass have been used
    // ---- expert product
    if (rows_now && !own && !*(volatile int*)&fail_sh) {         // after a failed wait nothing goes over copies that may be in flight
      ring = last ? smem : bits_s;
      ask(min(kMaxRows, (int)((uint32_t)(last ? off_h : buf_bytes) / item_bytes)));
    }
    if (!waited) { pdl_wait(); waited = true; }                  // h
    if (new_linear) {
      if (rows_now) {
        // only the pieces of tokens that exist
        const int n = ((M + 7) >> 3) * 2 * rsteps * 32;
        for (int i = tid; i < n; i += kMainThreads)
          if (((i & 31) >> 2) + (i >= 2 * rsteps * 32 ? 8 : 0) < M) h_s[i] = __ldcg(L.hfrag + i);
      }
      if (L.A8) {
        // the hidden activation enters the second 8-bit product quantised per token from its exact integers (Eq. 7-9)
        for (int t = warp; t < M; t += kMainWarps) {
          float v[8];
          float amax = 0.f;
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            v[u] = lane + 32 * u < r ? (float)__ldcg(L.h_int + (long long)t * r + lane + 32 * u) : 0.f;
            amax = fmaxf(amax, fabsf(v[u]));
          }
          for (int d = 16; d > 0; d >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, d));
          const float gh = __fdiv_rn(kActQmax, fmaxf(amax, kActAmaxFloor));
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (lane + 32 * u < r) qh_s[t * r + lane + 32 * u] = (int8_t)quant_code(v[u], gh);
          if (lane == 0) gh_sh[t] = gh;
        }
      }
      __syncthreads();                                           // h is visible
    }
    for (int i = warp, j = 0; i < items; i += W) {
      const int ei = i / tiles, t = i - ei * tiles;
      decode_wait(smem_u32(&bars[2 + warp * kWarpRows + j]), (row_phase >> j) & 1u, &fail_sh, poll);
      row_phase ^= 1u << j;
      main_expert(reinterpret_cast<const uint4*>(ring + (size_t)(warp * per + j) * item_bytes), r, order_sh + first_sh[ei], count_sh[ei], h_s, lane, red_z + (size_t)t * MT * 16);
      __syncwarp();
      if (i + W * per < items && !*(volatile int*)&fail_sh) issue(i + W * per, j);
      if (++j == per) j = 0;
    }
    if (last && !own) q_loaded = nullptr;
    if (L.A8) {
      // INT8 branch: z_int = B8_e qh (exact), z = z_int / (gamma_B gamma_h gamma_A gamma_t).  An item is (tile, token): lanes l and
      // l + 16 share feature l of the tile and take alternate pieces of 16 hidden values
      const int r16 = r >> 4, G32 = ((N + 127) >> 7) * 4, half = lane >> 4, f = lane & 15;
      for (int i = warp; i < tiles * M; i += kMainWarps) {
        const int t = i / tiles, un = i - t * tiles, e = tok[t].expert, at = cur.unit + un;
        const uint4* bp8 = L.B8_il + ((long long)e * G32 + (at >> 1)) * r16 * 32 + (at & 1) * 16 + f;
        const uint4* qv = reinterpret_cast<const uint4*>(qh_s + t * r);
        uint4 w[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) w[u] = 2 * u + half < r16 ? __ldg(bp8 + (2 * u + half) * 32) : make_uint4(0u, 0u, 0u, 0u);
        int zi = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (2 * u + half < r16) {
            const uint4 q = qv[2 * u + half];
            zi = __dp4a((int)w[u].x, (int)q.x, zi); zi = __dp4a((int)w[u].y, (int)q.y, zi);
            zi = __dp4a((int)w[u].z, (int)q.z, zi); zi = __dp4a((int)w[u].w, (int)q.w, zi);
          }
        }
        zi += __shfl_xor_sync(0xffffffffu, zi, 16);
        const float den = __fmul_rn(__fmul_rn(__fmul_rn(__ldg(L.hp_scales + 2 * e + 1), gh_sh[t]), __ldg(L.hp_scales + 2 * e)), tok[t].gamma);
        if (half == 0) {
          red_z[(un * MT + t) * 16 + f] = __fdiv_rn((float)zi, den);
          if (L.zint_dump) L.zint_dump[(long long)t * N + n0 + un * 16 + f] = zi;
        }
      }
    }
    __syncthreads();
    // ---- epilogue (Eq. 10-11), two features per thread
    for (int o = tid; o < (rows >> 1) * M; o += kMainThreads) {
      const int t = o / (rows >> 1), f = 2 * (o - t * (rows >> 1));
      const int at = ((f >> 4) * MT + t) * 16 + (f & 15);
      const int2 v = *reinterpret_cast<const int2*>(red_i + at);
      const int a0 = 2 * v.x - tok[t].rowsum, a1 = 2 * v.y - tok[t].rowsum;
      const float deq = deq_sh[t];
      float y0 = be_sh[f] * deq * (float)a0, y1 = be_sh[f + 1] * deq * (float)a1;
      if (r > 0) {
        const float2 z = *reinterpret_cast<const float2*>(red_z + at);
        y0 = fmaf(al_sh[f] * tok[t].gate, z.x, y0); y1 = fmaf(al_sh[f + 1] * tok[t].gate, z.y, y1);
      }
      uint16_t* y = L.Y + (long long)t * N + n0 + f;
      const uint32_t both = pack_bf16x2(y0, y1);
      if ((reinterpret_cast<uintptr_t>(L.Y) & 3) == 0) {         // rows have an even number of features
        *reinterpret_cast<uint32_t*>(y) = both;
      } else {                                                   // an output that starts at an odd element
        y[0] = (uint16_t)both; y[1] = (uint16_t)(both >> 16);
      }
      if (L.acc_dump) { L.acc_dump[(long long)t * N + n0 + f] = a0; L.acc_dump[(long long)t * N + n0 + f + 1] = a1; }
    }
    // ---- the buffer is free: the pass after the next one
    const int was = cur.l;
    cur = nbuf > 1 ? nxt : pass_at(u_next, cur.l);
    u_next += cur.nu;
    if (cur.nu == 0) break;
    __syncthreads();                                             // the sums, factors and records of this pass have been used
    if (*(volatile int*)&fail_sh) break;
    if (cur.l != was && cur.l + 1 < bp.n && bp.unit0[cur.l + 1] < u_hi) {
      copy_record(&lin_sh[(cur.l + 1) & 1], bp, cur.l + 1);
      __syncthreads();
    }
    if (nbuf > 1) {
      nxt = pass_at(u_next, cur.l);
      fetch_bits(nxt, b);
      b ^= 1;
    } else {
      fetch_bits(cur, 0);
    }
    load_scales(cur);
  }
  if (!waited) pdl_wait();
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
static inline size_t up256(size_t x) { return (x + 255) / 256 * 256; }

size_t decode_workspace_bytes(int M, int K, int N, int r, bool dump) {
  const size_t halves = 2 * (((size_t)K + 127) / 128);
  size_t b = up256(sizeof(DecodeTokInfo) * kDecodeMaxTokens);
  b += up256((size_t)(M > 8 ? 2 : 1) * halves * 32 * sizeof(uint4));
  b += up256((size_t)2 * 2 * ((r + 31) / 32 > 0 ? (r + 31) / 32 : 1) * 512);
  if (dump) b += up256(sizeof(int) * (size_t)M * N);
  b += up256((size_t)M * K * 2);                           // normalised tokens, or codes in natural order
  return b;
}

DecodeViewPtrs decode_view(int M, int K, int N, int r, void* ws, bool dump) {
  uint8_t* w = static_cast<uint8_t*>(ws);
  const size_t halves = 2 * (((size_t)K + 127) / 128);
  DecodeViewPtrs v{w, nullptr};
  w += up256(sizeof(DecodeTokInfo) * kDecodeMaxTokens) + up256((size_t)(M > 8 ? 2 : 1) * halves * 32 * sizeof(uint4)) + up256((size_t)2 * 2 * ((r + 31) / 32 > 0 ? (r + 31) / 32 : 1) * 512);
  if (dump) v.acc = reinterpret_cast<int*>(w);
  (void)N;
  return v;
}

// Launch option: programmatic stream serialisation of the two decode kernels (on by default).
static int g_decode_pdl = 1;
void decode_set_pdl(int on) { g_decode_pdl = on ? 1 : 0; }
static int g_decode_poll = 0;
void decode_set_poll(int on) { g_decode_poll = on ? 1 : 0; }

constexpr size_t kDecodeMainSmemLimit = 220 * 1024;   // dynamic shared memory of k_decode_main (it has a few KB of its own)
constexpr size_t kDecodeMainSmemBeside = 185 * 1024;  // ... that leaves room for one CTA of k_decode_hidden on the SM

template <int CAP>
static int decode_launch_as(const DecodeItemArgs* items, int n, cudaStream_t st) {
  const int sms = sm_count();
  DecodeBatch<CAP> bp;
  bp.n = n;
  bp.poll = g_decode_poll;
  size_t h_bytes = 0, smem_prep = 0, slot_bytes = 0;
  int max_m = 1, units = 0, max_c = 1, row_bytes = 0, max_used = 1, min_c = 1 << 30;
  bp.hidden_groups = 0;
  for (int i = 0; i < n; ++i) {
    const DecodeItemArgs& it = items[i];
    const int M = it.a.T, K = it.a.K, N = it.a.N, r = it.a.r;
    DecodeLinear& L = bp.lin[i];
    uint8_t* w = static_cast<uint8_t*>(it.ws);
    const size_t rsteps = std::max(1, (r + 31) / 32);
    L.info = reinterpret_cast<DecodeTokInfo*>(w); w += up256(sizeof(DecodeTokInfo) * kDecodeMaxTokens);
    L.qfrag = reinterpret_cast<uint4*>(w); w += up256((size_t)(M > 8 ? 2 : 1) * (((size_t)K + 127) / 128) * 64 * sizeof(uint4));
    L.hfrag = reinterpret_cast<uint4*>(w); w += up256((size_t)2 * 2 * rsteps * 512);
    L.acc_dump = it.dump ? reinterpret_cast<int*>(w) : nullptr;
    if (it.dump) w += up256(sizeof(int) * (size_t)M * N);
    L.xn = reinterpret_cast<uint16_t*>(w);
    L.X = reinterpret_cast<const uint4*>(it.X); L.Wr = reinterpret_cast<const uint4*>(it.a.Wr); L.A = it.a.A; L.B = it.a.B;
    L.bits = it.bits; L.bits_il = reinterpret_cast<const uint4*>(it.bits_il);
    L.w_scales = it.a.w_scales; L.alpha = it.a.alpha; L.beta = it.a.beta; L.Y = it.Y;
    L.norm_w = reinterpret_cast<const uint4*>(it.norm_weight); L.norm_eps = it.norm_eps;
    L.M = M; L.K = K; L.N = N; L.r = r; L.E = (r > 0 && it.a.E > 1) ? it.a.E : 1; L.sstride = it.a.scale_stride;
    L.A8 = it.A8; L.B8_il = it.A8 ? reinterpret_cast<const uint4*>(it.B_il) : nullptr; L.hp_scales = it.hp_scales;
    L.h_int = L.zint_dump = nullptr;
    if (it.A8) {
      decode_stream_view(M, K, N, r, it.ws, it.dump, &L.h_int, &L.zint_dump);
      h_bytes = std::max(h_bytes, up256((size_t)M * r));
    } else if (r > 0) {
      h_bytes = std::max(h_bytes, up256((size_t)((M + 7) / 8) * 2 * rsteps * 512));
      slot_bytes = std::max(slot_bytes, (size_t)32 * r);
      max_used = std::max(max_used, std::min(L.E, M));
    }
    L.unit0 = units;
    bp.unit0[i] = units;
    units += N / kUnit;
    L.hidden0 = bp.hidden_groups;
    if (r > 0) row_bytes = std::max(row_bytes, it.A8 ? K : 2 * K);
    if (r > 0) bp.hidden_groups += std::min(L.E, M) * ((r + 15) / 16);
    max_m = std::max(max_m, M); max_c = std::max(max_c, (K + 127) / 128); min_c = std::min(min_c, (K + 127) / 128);
    smem_prep = std::max(smem_prep, prep_plan(K, L.E, L.norm_w != nullptr).bytes);
  }
  for (int i = n; i <= CAP; ++i) bp.unit0[i] = units;
  bp.units = units;

  // ---- k_decode_main: one CTA per SM (fewer when there is less than a unit for each)
  const int ctas = std::min(sms, units), share = (units + ctas - 1) / ctas;
  bp.red_tokens = max_m > 8 ? 16 : 8;
  // ---- k_decode_hidden: CTAs of a cluster
  // One CTA per SM; with rows of A_e beyond 4 KB, whose contraction is worth more than room for k_decode_main's CTAs beside it, up to
  // three.  Per call, one CTA per cluster against two where two are more than the SMs hold: M = 11, 1056 x 7552 18.6 / 21.7 us, M = 4,
  // INT8, 3200 x 8640 16.9 / 18.3; M = 13, 2816 x 4960 22.1 / 20.7, M = 16, 3200 x 8640 37.2 / 31.4.
  // Up to four tokens and rows of one length, where pairs would be a few more than the SMs and a CTA of k_decode_main has room beside one
  // of these, one: two linears of 3200 x 8640 (8640 x 3200), four tokens 21.2 (25.9) us, with pairs 24.8 (30.8).
  const bool few_over = max_m <= 4 && 4 * bp.hidden_groups <= 2 * sms + sms / 2 && min_c == max_c;
  const int pairs_to = row_bytes > 4096 ? 3 * sms : sms;
  bp.hidden_cluster = 4 * bp.hidden_groups <= sms ? 4 : 2 * bp.hidden_groups <= pairs_to ? 2 : 1;
  // CTAs of k_decode_main that start beside k_decode_hidden's take room and memory requests from them: with more than eight tokens and rows
  // of A_e beyond 4 KB, where those are more than the SMs but would all be resident without, they start only afterwards.  Beside / after,
  // eight experts, sixteen tokens: 8640 x 3200 29.6 / 28.2 us, 2784 x 4960 21.8 / 20.8, two of 3200 x 8640 31.5 / 30.4.  Eight tokens:
  // 8640 x 3200 20.6 / 22.6; shorter rows: three of 2048 x 2048, sixteen 24.1 / 26.1; more CTAs: twelve of 2048 x 5632, eight 72.4 / 73.5.
  const int hidden_ctas = bp.hidden_groups * bp.hidden_cluster;
  const bool apart = max_m > 8 && row_bytes > 4096 && hidden_ctas > sms && hidden_ctas <= 3 * sms;
  // Shared memory goes to sign bits (units of 16 features in a pass), codes (those of all of K, or of a slice of it), sums, and
  // places for expert rows, apart from the rest or over it.  In microseconds, about: a pass is three of barriers and first trips, a
  // further slice of the codes one, a round of expert rows (as many items as there are places) one, and one more where they set
  // out only after the 1-bit product; a CTA that leaves no room for one of k_decode_hidden's beside it starts one and a half later.  The split
  // with the least of these is taken.  Linears of different K share it: `units` are of the longest row, shorter ones have more in a pass.
  // Places apart against places over used sign bits, us a call with eight experts of 160: 1056 x 7552, four tokens 12.9 / 19.6, sixteen
  // 20.3 / 24.5; 2048 x 5632, twelve linears, eight tokens 74 / 98; two of 3200 x 8640, sixteen tokens 33.7 / 31.2.
  const size_t unit_bytes = (size_t)256 * max_c, chunk_bytes = (size_t)128 * max_m;   // a unit's sign bits; codes of 128 values of k
  struct Split { int nbuf, units, red_units, q_chunks, slots; size_t q_bytes, bytes; double cost; } best{};
  const int most = std::min(share, kMaxPassUnits);
  const bool one_pass = n == 1 && share <= kMaxPassUnits;        // sign bits of a single pass need no second buffer
  auto places = [](size_t bytes, size_t each, int wanted) {      // two for each warp, one, or fewer than there are warps
    const int fit = (int)(bytes / each);
    return wanted > kMainWarps && fit >= kMaxRows ? kMaxRows : std::min({kMainWarps, wanted, fit});
  };
  auto rounds = [](int wanted, int slots) { return std::max(1.0, (double)wanted / slots); };
  for (int nbuf = one_pass ? 1 : 2; nbuf >= 1 && best.units == 0; --nbuf) {
    for (int units = most; units >= 1; --units) {
      if (one_pass && units < share && best.units > 0) break;
      int passes = 1;
      for (int i = 0; i < n; ++i) {
        const int cap = std::min(most, units * max_c / ((items[i].a.K + 127) / 128));
        passes = std::max(passes, (std::min(share, items[i].a.N / kUnit) + cap - 1) / cap);
      }
      for (int slices = 1; slices <= max_c; ++slices) {
        Split c{nbuf, units, nbuf == 1 && !one_pass ? units : most, (max_c + slices - 1) / slices, 0, 0, 0, 0.0};
        c.q_bytes = up256(c.q_chunks * chunk_bytes);
        const size_t red = (size_t)2 * c.red_units * bp.red_tokens * 16 * 4, buf = units * unit_bytes, used = nbuf * buf + c.q_bytes + h_bytes + red;
        if (used > kDecodeMainSmemLimit) continue;
        const int wanted = max_used * units;
        auto offer = [&](int slots, double rows) {               // rows: what the expert rows of all passes cost
          c.slots = slots; c.bytes = used + slots * slot_bytes;
          c.cost = passes * (3.0 + (slices - 1)) + rows + (c.bytes > kDecodeMainSmemBeside && !apart ? 1.5 : 0.0);
          if (best.units == 0 || c.cost < best.cost) best = c;
        };
        if (slot_bytes == 0) {
          offer(0, 0.0);
        } else {
          for (size_t limit : {kDecodeMainSmemBeside, kDecodeMainSmemLimit})
            if (const int s = used < limit ? places(limit - used, slot_bytes, wanted) : 0) offer(s, passes * rounds(wanted, s));
          if (buf >= slot_bytes)
            offer(0, passes + (passes - 1) * rounds(wanted, places(buf, slot_bytes, wanted)) +
                         rounds(wanted, places(nbuf * buf + c.q_bytes, slot_bytes, wanted)));
        }
        if (slices >= 4 && best.units > 0) break;
      }
    }
  }
  if (best.units == 0) return PQ_ERR_UNSUPPORTED;
  bp.nbuf = best.nbuf; bp.pass_units = best.red_units; bp.q_chunks = best.q_chunks; bp.row_slots = best.slots;
  bp.buf_bytes = (int)(best.units * unit_bytes);
  if (few_over && best.bytes <= kDecodeMainSmemBeside && 2 * bp.hidden_groups > sms) bp.hidden_cluster = 1;
  // One or two linears only: of more, the rows take the memory from those of A that k_decode_hidden is waiting for (twelve of 3200 x
  // 8640, sixteen tokens 163 us with, 145 without; two 31.2 / 31.8).
  bp.rows_early = best.slots == 0 && n <= 2;
  size_t off = (size_t)bp.nbuf * bp.buf_bytes;
  bp.off_q = (int)off; off += best.q_bytes;
  bp.off_h = (int)off; off += h_bytes;
  bp.off_red = (int)off; off += (size_t)2 * best.red_units * bp.red_tokens * 16 * 4;
  bp.off_rows = (int)off; off += best.slots * slot_bytes;
  const size_t smem_main = apart ? kDecodeMainSmemLimit : off;

  // ---- k_decode_prep
  bp.early = bp.hidden_groups > 0;
  if (smem_prep > kDecodePrepSmemLimit) return PQ_ERR_UNSUPPORTED;

  using Kern = void (*)(DecodeBatch<CAP>);
  const Kern prep = k_decode_prep<CAP>, hidden = k_decode_hidden<CAP>;
  const Kern main = max_m > 8 ? (Kern)k_decode_main<CAP, 2> : (Kern)k_decode_main<CAP, 1>;
  // The opt-in limits are set once, to the largest request this file can make: a launch recorded in a CUDA graph
  // keeps its own shared-memory size, and a later call with a smaller one must not lower the limit under it.  All kernels ask
  // for the same split of an SM's memory: CTAs that want different splits cannot be resident together.
  static const bool attributes_set = [] {
    const Kern all[4] = {k_decode_prep<CAP>, k_decode_hidden<CAP>, k_decode_main<CAP, 1>, k_decode_main<CAP, 2>};
    const size_t limit[4] = {kDecodePrepSmemLimit, 0, kDecodeMainSmemLimit, kDecodeMainSmemLimit};
    for (int i = 0; i < 4; ++i) {
      if (limit[i] && cudaFuncSetAttribute(all[i], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit[i]) != cudaSuccess) return false;
      if (cudaFuncSetAttribute(all[i], cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) != cudaSuccess) return false;
    }
    return true;
  }();
  if (!attributes_set) return PQ_ERR_CUDA;

  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.stream = st; cfg.attrs = attr; cfg.numAttrs = g_decode_pdl ? 1 : 0;
  {
    cfg.gridDim = dim3(kPrepCluster, max_m, n); cfg.blockDim = dim3(kPrepThreads, 1, 1); cfg.dynamicSmemBytes = smem_prep;
    LaunchScope ls(KID_DECODE_PREP, st);
    if (cudaLaunchKernelEx(&cfg, prep, bp) != cudaSuccess) return PQ_ERR_CUDA;
  }
  if (bp.hidden_groups > 0) {
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = bp.hidden_cluster; attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    if (!g_decode_pdl) attr[0] = attr[1];
    cfg.numAttrs = g_decode_pdl ? 2 : 1;
    cfg.gridDim = dim3(bp.hidden_groups * bp.hidden_cluster, 1, 1); cfg.blockDim = dim3(kHiddenThreads, 1, 1); cfg.dynamicSmemBytes = 0;
    LaunchScope ls(KID_DECODE_PREP, st);
    if (cudaLaunchKernelEx(&cfg, hidden, bp) != cudaSuccess) return PQ_ERR_CUDA;
    cfg.numAttrs = g_decode_pdl ? 1 : 0;
  }
  {
    cfg.gridDim = dim3(ctas, 1, 1); cfg.blockDim = dim3(kMainThreads, 1, 1); cfg.dynamicSmemBytes = smem_main;
    LaunchScope ls(KID_DECODE_MAIN, st);
    if (cudaLaunchKernelEx(&cfg, main, bp) != cudaSuccess) return PQ_ERR_CUDA;
  }
  return PQ_OK;
}

// the descriptors are copied with every launch: small groups carry a small table
static int decode_launch(const DecodeItemArgs* items, int n, cudaStream_t st) {
  if (n <= 2) return decode_launch_as<2>(items, n, st);
  if (n <= 16) return decode_launch_as<16>(items, n, st);
  return decode_launch_as<kDecodeMaxBatch>(items, n, st);
}

int decode_stream_max_batch();   // pq_decode_stream.cu

// The run of items at the front that all carry the streaming kernel's weight layout: its length, at most `most`, and whether that kernel
// is the faster one for it.  It starts late (token work, then a barrier of the whole grid) and costs little per linear; what decides is
// the number of units of 16 features per SM, the number of tokens and whether there are experts.
struct StreamRun { int n; bool pays; };
static StreamRun stream_run(const DecodeItemArgs* items, int most) {
  StreamRun run{0, false};
  const int sms = sm_count();
  int max_m = 1;
  long long units = 0;
  bool experts = false, routed = false;
  while (run.n < most && items[run.n].bits_il) {
    const LayerArgs& a = items[run.n].a;
    max_m = std::max(max_m, a.T);
    units += a.N / kUnit;
    experts = experts || a.r > 0;
    routed = routed || (a.r > 0 && a.E > 1);
    ++run.n;
  }
  // us a call, small-group kernels / streaming kernel: eight experts of 160, one token, 8 linears of 2048 x 5632 31 / 30, 6 of 3200 x
  // 8640 33 / 31, 24 of 2048 x 2048 39 / 38; two tokens, 6 and 8 of 3200 x 8640 40 / 44, 50 / 47; three, 8 and 12 54 / 59, 75 / 70; four, 12 and
  // 24 77 / 80, 148 / 128; six, 24 of 2048 x 5632 123 / 127, of 3200 x 8640 179 / 172; eight, 78 619 / 635; sixteen 935 / 1215.  A dense
  // branch of 128, one token, 8 of 3200 x 8640 38 / 32; two, 12 53 / 50, 24 of 2048 x 5632 61 / 61; four, 78 of 3200 x 8640 283 / 317.  No
  // branch, one token, 8 and 12 24 / 27, 34 / 32; two, 12 and 24 35 / 39, 65 / 57; four, 48 of 2048 x 5632 84 / 81.  INT8 experts as bf16 ones.
  constexpr int kNever = 1 << 30;
  const int least = routed ? (max_m <= 1 ? 19 : max_m <= 2 ? 29 : max_m <= 3 ? 40 : max_m <= 4 ? 44 : max_m <= 6 ? 75 : kNever)
                    : experts ? (max_m <= 1 ? 19 : max_m <= 2 ? 50 : max_m <= 3 ? 150 : kNever)
                              : (max_m <= 1 ? 37 : max_m <= 2 ? 65 : max_m <= 4 ? 114 : kNever);
  run.pays = units >= (long long)least * sms;
  return run;
}

int decode_batch(const DecodeItemArgs* items, int n, cudaStream_t st) {
  const int mode = decode_stream_mode(), group = std::min(decode_stream_max_batch(), kDecodeMaxBatch);
  int i = 0;
  while (i < n) {
    const int most = std::min(n - i, group);
    const StreamRun run = stream_run(items + i, most);
    int rc = PQ_ERR_UNSUPPORTED, m = run.n;
    if (run.n > 0 && (mode > 1 || (mode == 1 && run.pays))) rc = decode_stream_launch(items + i, run.n, st);
    if (rc == PQ_ERR_UNSUPPORTED) {
      // The three kernels above take items with and without the layout together, up to the start of a run that the streaming kernel
      // takes.
      auto run_starts = [&](int k) {
        if (mode == 0 || !items[i + k].bits_il || items[i + k - 1].bits_il) return false;
        return mode > 1 || stream_run(items + i + k, std::min(n - i - k, group)).pays;
      };
      m = std::max(run.n, 1);
      while (m < most && !(mode > 1 && run.n > 0) && !run_starts(m)) ++m;
      rc = decode_launch(items + i, m, st);
      // shared memory is laid out for the largest of everything in a launch: what does not fit together may fit apart
      while (rc == PQ_ERR_UNSUPPORTED && m > 1) rc = decode_launch(items + i, m /= 2, st);
    }
    if (rc) return rc;
    i += m;
  }
  return PQ_OK;
}

int decode_forward(const LayerArgs& a, const uint16_t* X, const uint32_t* bits, uint16_t* Y, void* ws, bool dump, cudaStream_t st) {
  DecodeItemArgs it{a, X, bits, Y, ws, dump};
  return decode_launch(&it, 1, st);
}

}  // namespace pq
