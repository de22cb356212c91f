// Memory-bound kernels of the pQuant layer: weight scale reduction and
// binarize-and-pack (Eq. 3, 4, 6), router (Sec. 3.3), expert sort, activation
// quantisation (Eq. 7-9), and the small gather / scale / reduce helpers of the
// backward pass.
#include <mutex>

#include "pq_kernels.cuh"

namespace pq {

ProfileSlot g_profile[KID_COUNT] = {};
long long g_launches = 0;

// ---------------------------------------------------------------------------
// K2a: partial sums of W and |W| in fp64 (Eq. 6).  Fixed grid and a fixed
// reduction tree, so the result does not depend on scheduling.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_weight_partial_sums(const float4* __restrict__ W4, long long n4, double* __restrict__ partial) {
  pdl_launch_dependents();   // launched with programmatic stream serialisation: see launch_pdl
  pdl_wait();
  double s = 0.0, a = 0.0;
  const long long stride = gridDim.x * 256LL;
  long long i = blockIdx.x * 256LL + threadIdx.x;
  // One conversion to fp64 per element (the conversion is the slow instruction here); |x| is taken on the double,
  // which is the same number as the double of |x|.  The order of the additions is fixed by the launch shape alone.
  auto sums = [](const float4& v, double& ts, double& ta) {
    const double d0 = (double)v.x, d1 = (double)v.y, d2 = (double)v.z, d3 = (double)v.w;
    ts = d0 + d1 + d2 + d3;
    ta = fabs(d0) + fabs(d1) + fabs(d2) + fabs(d3);
  };
  // four loads in flight per thread
  for (; i + 3 * stride < n4; i += 4 * stride) {
    const float4 v0 = __ldg(W4 + i), v1 = __ldg(W4 + i + stride), v2 = __ldg(W4 + i + 2 * stride), v3 = __ldg(W4 + i + 3 * stride);
    double s0, a0, s1, a1, s2, a2, s3, a3;
    sums(v0, s0, a0); sums(v1, s1, a1); sums(v2, s2, a2); sums(v3, s3, a3);
    s += s0 + s1;
    s += s2 + s3;
    a += a0 + a1;
    a += a2 + a3;
  }
  for (; i < n4; i += stride) {
    double s0, a0;
    sums(__ldg(W4 + i), s0, a0);
    s += s0;
    a += a0;
  }
  for (int d = 16; d > 0; d >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, d);
    a += __shfl_xor_sync(0xffffffffu, a, d);
  }
  __shared__ double sh[2][8];
  if ((threadIdx.x & 31) == 0) { sh[0][threadIdx.x >> 5] = s; sh[1][threadIdx.x >> 5] = a; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double ts = 0.0, ta = 0.0;
    for (int w = 0; w < 8; ++w) { ts += sh[0][w]; ta += sh[1][w]; }
    partial[2 * blockIdx.x] = ts;
    partial[2 * blockIdx.x + 1] = ta;
  }
}

// Every block re-reduces the (few hundred) partials in the same order, so all blocks agree on mu without
// a grid-wide barrier: thread t sums partials t, t + 256, ... (ascending), then a fixed tree over the block.
// The partials were written by the kernel before this one and the buffer is reused from call to call, so they are
// read with L2 loads (ld.global.cg): a kernel launched with programmatic stream serialisation can be resident while
// an older kernel still reads the previous call's values on the same SM, and the read-only data path gives no
// guarantee against finding those in L1.
__device__ __forceinline__ void reduce_partials(const double* partial, int nparts, double inv_count, float* mu, float* lam) {
  __shared__ double sh[2][8];
  __shared__ double fin[2];
  double s = 0.0, a = 0.0;
  for (int i = threadIdx.x; i < nparts; i += 256) { s += __ldcg(partial + 2 * i); a += __ldcg(partial + 2 * i + 1); }
  for (int d = 16; d > 0; d >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, d);
    a += __shfl_xor_sync(0xffffffffu, a, d);
  }
  if ((threadIdx.x & 31) == 0) { sh[0][threadIdx.x >> 5] = s; sh[1][threadIdx.x >> 5] = a; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double ts = 0.0, ta = 0.0;
    for (int w = 0; w < 8; ++w) { ts += sh[0][w]; ta += sh[1][w]; }
    fin[0] = ts; fin[1] = ta;
  }
  __syncthreads();
  *mu = (float)(fin[0] * inv_count);
  *lam = (float)(fin[1] * inv_count);
}

// ---------------------------------------------------------------------------
// K2b: S = Sign(W - mu) as the comparison W >= mu (Eq. 3-4); emits the packed
// words (bit j of word i <-> k = 32 i + j, 1 <-> +1; App. A) and the +-1 int8
// tile the tensor cores read.  Each thread owns 4 consecutive k.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_binarize_pack(const float4* __restrict__ W4, long long n4, const double* partial,
                                                       int nparts, double inv_count, uint32_t* __restrict__ bits,
                                                       uint32_t* __restrict__ s8x4, float* __restrict__ scales) {
  pdl_launch_dependents();   // launched with programmatic stream serialisation: see launch_pdl
  pdl_wait();
  float mu, lam;
  reduce_partials(partial, nparts, inv_count, &mu, &lam);
  if (blockIdx.x == 0 && threadIdx.x == 0) { scales[0] = lam; scales[1] = mu; }
  // n4 is a multiple of 8 (K % 32 == 0), so whole groups of 8 lanes stay together
  const long long n4_pad = (n4 + 31) & ~31LL;
  const long long stride = gridDim.x * 256LL;
  for (long long i0 = blockIdx.x * 256LL + threadIdx.x; i0 < n4_pad; i0 += 2 * stride) {
    float4 v[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const long long i = i0 + u * stride;
      v[u] = i < n4 ? __ldg(W4 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const long long i = i0 + u * stride;
      if (i >= n4_pad) break;          // uniform over the warp: stride and n4_pad are multiples of 32
      uint32_t nib = 0;
      if (i < n4) {
        const uint32_t b0 = v[u].x >= mu, b1 = v[u].y >= mu, b2 = v[u].z >= mu, b3 = v[u].w >= mu;
        nib = b0 | (b1 << 1) | (b2 << 2) | (b3 << 3);
        // +1 -> 0x01, -1 -> 0xFF, little endian: byte j <-> k + j
        const uint32_t bytes = (b0 ? 0x01u : 0xFFu) | (b1 ? 0x0100u : 0xFF00u) | (b2 ? 0x010000u : 0xFF0000u) | (b3 ? 0x01000000u : 0xFF000000u);
        if (s8x4) s8x4[i] = bytes;
      }
      uint32_t word = nib << (4 * (threadIdx.x & 7));
      word |= __shfl_xor_sync(0xffffffffu, word, 1);
      word |= __shfl_xor_sync(0xffffffffu, word, 2);
      word |= __shfl_xor_sync(0xffffffffu, word, 4);
      if ((threadIdx.x & 7) == 0 && i < n4) bits[i >> 3] = word;
    }
  }
}

// RMSNorm fused in front of the quantiser (App. A): what every consumer of a token sees is
//   bf16( fl32( fl32(x * s_t) * g_k ) ),   s_t = fl32( 1 / sqrt(mean_k x^2 + eps) )  (mean and root in fp64, k_row_rms),
// the values a separate bf16 norm layer would have handed over.  One 16-byte piece (8 values) at a time.
__device__ __forceinline__ uint4 rms_apply(const uint4& v, float s, const uint4& g) {
  uint4 o;
  o.x = pack_bf16x2(__fmul_rn(__fmul_rn(bf16lo(v.x), s), bf16lo(g.x)), __fmul_rn(__fmul_rn(bf16hi(v.x), s), bf16hi(g.x)));
  o.y = pack_bf16x2(__fmul_rn(__fmul_rn(bf16lo(v.y), s), bf16lo(g.y)), __fmul_rn(__fmul_rn(bf16hi(v.y), s), bf16hi(g.y)));
  o.z = pack_bf16x2(__fmul_rn(__fmul_rn(bf16lo(v.z), s), bf16lo(g.z)), __fmul_rn(__fmul_rn(bf16hi(v.z), s), bf16hi(g.z)));
  o.w = pack_bf16x2(__fmul_rn(__fmul_rn(bf16lo(v.w), s), bf16lo(g.w)), __fmul_rn(__fmul_rn(bf16hi(v.w), s), bf16hi(g.w)));
  return o;
}

// s_t for every token: one warp per row, squares summed in fp64 (lane-strided pieces ascending, then the butterfly).
__global__ void __launch_bounds__(256) k_row_rms(const uint4* __restrict__ X, int T, int K, float eps, float* __restrict__ rms) {
  pdl_launch_dependents();
  pdl_wait();
  const int t = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (t >= T) return;
  const int chunks = K >> 3;
  const uint4* row = X + (long long)t * chunks;
  double ss = 0.0;
  for (int c = lane; c < chunks; c += 32) {
    const uint4 v = __ldg(row + c);
    const double d0 = bf16lo(v.x), d1 = bf16hi(v.x), d2 = bf16lo(v.y), d3 = bf16hi(v.y);
    const double d4 = bf16lo(v.z), d5 = bf16hi(v.z), d6 = bf16lo(v.w), d7 = bf16hi(v.w);
    ss += ((d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3)) + ((d4 * d4 + d5 * d5) + (d6 * d6 + d7 * d7));
  }
  for (int d = 16; d > 0; d >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, d);
  if (lane == 0) rms[t] = (float)(1.0 / sqrt(ss / (double)K + (double)eps));
}

// ---------------------------------------------------------------------------
// K4a: router (Sec. 3.3).  Logits in fp32 with a fixed summation order -- lane j owns the 8-element
// chunks c with c mod 32 == j, ascending k, fused multiply-add; lanes combined by the xor butterfly
// 16, 8, 4, 2, 1 -- so that the top-1 index is reproducible bit for bit.  Softmax in fp32; ties go to
// the lowest index.  Also counts tokens per expert for each block of kRouterTokensPerBlock tokens.
//
// Bound by the fused multiply-adds (T K E of them; with the unpacking about 350 issue slots of a scheduler per
// 16 tokens x 256 elements x 8 experts) and, about equally, by reading X.  The order above leaves one lane's
// chain per (token, expert) and no way to split K over threads, so what keeps the chip busy is many small CTAs, each
// with enough of X in flight: 16 tokens per CTA, four per warp, and a ring of kRouterStages steps of 256 elements
// filled by 16-byte asynchronous copies (X of the warp's tokens, and the CTA's Wr, unpacked once per four tokens).
// Two experts share one instruction (fma.rn.f32x2: two independent roundings, the same values).
// Measured with eight experts, before (32 tokens per CTA, one step prefetched in registers, scalar fma) and now: 8192 tokens
// x 2048 29 -> 13.8 us, x 5632 56 -> 31 us, 2048 tokens x 3200 41 -> 10.2 us.  Three stages and four CTAs per SM beat five
// and three (31 against 33 us); scalar fma 41; two tokens per warp 39.
// ---------------------------------------------------------------------------
constexpr int kRouterWarps = 4, kRouterTpw = kRouterTokensPerBlock / kRouterWarps, kRouterStages = 3;

template <int EMAX>
constexpr int router_smem() { return kRouterStages * (kRouterTokensPerBlock + EMAX) * 32 * (int)sizeof(uint4); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {   // invalid: zeros
  const int n = valid ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ uint64_t pack_f32x2(float lo, float hi) {
  uint64_t v;
  asm("mov.b64 %0, {%1, %2};" : "=l"(v) : "f"(lo), "f"(hi));
  return v;
}
__device__ __forceinline__ uint64_t fma_f32x2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// EMAX: compile-time bound on E, a power of two (experts past E have zero weights and are left out at the end)
template <int EMAX>
__global__ void __launch_bounds__(32 * kRouterWarps, EMAX <= 8 ? 4 : 2) k_router(const uint4* __restrict__ X, const uint4* __restrict__ Wr, int T, int K, int E,
                                                              int* __restrict__ expert, float* __restrict__ gate_tok, float* __restrict__ probs_tok,
                                                              int* __restrict__ block_counts, const uint4* __restrict__ norm_w,
                                                              const float* __restrict__ rms) {
  pdl_launch_dependents();   // launched with programmatic stream serialisation: see launch_pdl
  constexpr int TPW = kRouterTpw, S = kRouterStages, ROWS = kRouterTokensPerBlock + EMAX;
  extern __shared__ uint4 ring[];                       // [stage][token or expert][32 chunks]
  __shared__ __align__(16) float logit[kRouterTokensPerBlock * EMAX];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunks = K >> 3, steps = (chunks + 31) >> 5;
  const int t0 = blockIdx.x * kRouterTokensPerBlock + warp * TPW;   // this warp's first token
  pdl_wait();
  // a token past the end repeats the last one, unused
  auto fetch = [&](int step) {
    if (step < steps) {
      const int c = step * 32 + lane;
      const bool in = c < chunks;
      const uint32_t dst = smem_u32(ring + (step % S) * ROWS * 32 + lane);
#pragma unroll
      for (int u = 0; u < TPW; ++u)
        cp_async16(dst + (warp * TPW + u) * 512, X + (long long)min(t0 + u, T - 1) * chunks + (in ? c : 0), in);
#pragma unroll
      for (int i = 0; i < EMAX / kRouterWarps; ++i) {
        const int e = warp + i * kRouterWarps;
        cp_async16(dst + (kRouterTokensPerBlock + e) * 512, Wr + (long long)(e < E ? e : 0) * chunks + (in ? c : 0), in && e < E);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float srow[TPW];
#pragma unroll
  for (int u = 0; u < TPW; ++u) srow[u] = norm_w ? __ldcg(rms + min(t0 + u, T - 1)) : 1.0f;
  uint64_t acc[TPW][EMAX / 2];
#pragma unroll
  for (int u = 0; u < TPW; ++u)
#pragma unroll
    for (int e = 0; e < EMAX / 2; ++e) acc[u][e] = 0ull;
#pragma unroll
  for (int i = 0; i < S - 1; ++i) fetch(i);
  for (int step = 0; step < steps; ++step) {
    asm volatile("cp.async.wait_group %0;" ::"n"(S - 2) : "memory");
    __syncthreads();
    fetch(step + S - 1);                                // into the stage every warp has left
    const uint4* st = ring + (step % S) * ROWS * 32 + lane;
    uint4 g = make_uint4(0u, 0u, 0u, 0u);
    if (norm_w && step * 32 + lane < chunks) g = __ldg(norm_w + step * 32 + lane);
    uint64_t x[TPW][8];
#pragma unroll
    for (int u = 0; u < TPW; ++u) {
      uint4 v = st[(warp * TPW + u) * 32];
      if (norm_w) v = rms_apply(v, srow[u], g);         // the router sees the normalised token
      const float f[8] = {bf16lo(v.x), bf16hi(v.x), bf16lo(v.y), bf16hi(v.y), bf16lo(v.z), bf16hi(v.z), bf16lo(v.w), bf16hi(v.w)};
#pragma unroll
      for (int i = 0; i < 8; ++i) x[u][i] = pack_f32x2(f[i], f[i]);
    }
#pragma unroll
    for (int e = 0; e < EMAX / 2; ++e) {
      const uint4 a = st[(kRouterTokensPerBlock + 2 * e) * 32], b = st[(kRouterTokensPerBlock + 2 * e + 1) * 32];
      const uint64_t w[8] = {pack_f32x2(bf16lo(a.x), bf16lo(b.x)), pack_f32x2(bf16hi(a.x), bf16hi(b.x)), pack_f32x2(bf16lo(a.y), bf16lo(b.y)),
                             pack_f32x2(bf16hi(a.y), bf16hi(b.y)), pack_f32x2(bf16lo(a.z), bf16lo(b.z)), pack_f32x2(bf16hi(a.z), bf16hi(b.z)),
                             pack_f32x2(bf16lo(a.w), bf16lo(b.w)), pack_f32x2(bf16hi(a.w), bf16hi(b.w))};
#pragma unroll
      for (int u = 0; u < TPW; ++u)
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[u][e] = fma_f32x2(x[u][i], w[i], acc[u][e]);
    }
  }
  // butterfly 16, 8, 4, 2, 1 over the lanes; a lane keeps half of its sums at each level (the same additions)
  constexpr int NV = TPW * EMAX;
  float v[NV];
#pragma unroll
  for (int u = 0; u < TPW; ++u)
#pragma unroll
    for (int e = 0; e < EMAX / 2; ++e) {
      v[u * EMAX + 2 * e] = __uint_as_float((uint32_t)acc[u][e]);
      v[u * EMAX + 2 * e + 1] = __uint_as_float((uint32_t)(acc[u][e] >> 32));
    }
  int n = NV, idx = 0;
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) {
    if (n > 1) {
      n >>= 1;
      const bool up = lane & d;
      idx += up ? n : 0;
#pragma unroll
      for (int i = 0; i < NV / 2; ++i) {
        if (i < n) {
          const float keep = up ? v[i + n] : v[i], send = up ? v[i] : v[i + n];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, d);
        }
      }
    } else {
      v[0] = v[0] + __shfl_xor_sync(0xffffffffu, v[0], d);
    }
  }
#pragma unroll
  for (int i = 0; i < (NV > 32 ? NV / 32 : 1); ++i) logit[warp * NV + idx + i] = v[i];
  __syncthreads();
  // a lane of the first warp per token
  if (warp == 0) {
    const int t = blockIdx.x * kRouterTokensPerBlock + lane;
    const bool own = lane < kRouterTokensPerBlock && t < T;
    int best = -1;
    if (own) {
      float l[EMAX];
      const float4* row = reinterpret_cast<const float4*>(logit + lane * EMAX);
#pragma unroll
      for (int e = 0; e < EMAX; e += 4) { const float4 q = row[e >> 2]; l[e] = q.x; l[e + 1] = q.y; l[e + 2] = q.z; l[e + 3] = q.w; }
      best = 0;
      float lmax = l[0];
#pragma unroll
      for (int e = 1; e < EMAX; ++e)
        if (e < E && l[e] > lmax) { lmax = l[e]; best = e; }
      float den = 0.f;
#pragma unroll
      for (int e = 0; e < EMAX; ++e) {
        l[e] = e < E ? expf(l[e] - lmax) : 0.f;
        den += l[e];
      }
      const float inv = 1.0f / den;
      expert[t] = best;
#pragma unroll
      for (int e = 0; e < EMAX; ++e) {
        if (e < E) {
          const float pr = l[e] * inv;
          probs_tok[(long long)t * E + e] = pr;
          if (e == best) gate_tok[t] = pr;
        }
      }
    }
    for (int e = 0; e < E; ++e) {
      const int cnt = __popc(__ballot_sync(0xffffffffu, best == e));
      if (lane == 0) block_counts[e * gridDim.x + blockIdx.x] = cnt;
    }
  }
}

// ---------------------------------------------------------------------------
// K4b: expert offsets, per-block bases for the stable scatter, and the item
// table.  An item is the intersection of a 128-row tile of the sorted token
// order with one expert's range: {tile, expert, first row, end row} (rows
// relative to the tile).  Items are sorted by tile and therefore by expert.
// One block; the work is a few hundred integers.
// ---------------------------------------------------------------------------
// All of it is latency (a few thousand integers), so nothing is carried from step to step: a warp takes an expert,
// 512 blocks of tokens loaded and scanned together; and the number of items before a tile has a closed form,
// so every table entry is one thread's own sum over the experts.  Measured at 8192 tokens, eight experts: 5.6 us with the
// blocks 32 at a time and block-wide scans over the tiles, 4.4 us now.
// items in the tiles before `tile`, tiles of `rows` rows: a non-empty expert has one in every tile that it meets
__device__ __forceinline__ int items_before(const int* off, int Ee, int rows_log2, int tile) {
  int n = 0;
  for (int e = 0; e < Ee; ++e) {
    const int lo = off[e], hi = off[e + 1];
    if (hi > lo) n += max(0, min(tile - 1, (hi - 1) >> rows_log2) - (lo >> rows_log2) + 1);
  }
  return n;
}

__global__ void __launch_bounds__(512) k_route_scan(int T, int E, int nblocks, const int* __restrict__ block_counts,
                                                    int* __restrict__ block_base, int* __restrict__ offsets, RoutingTables rt) {
  pdl_launch_dependents();   // launched with programmatic stream serialisation: see launch_pdl
  pdl_wait();
  constexpr int kPer = 16, kTileLog2 = 7;
  static_assert(kTileRows == 1 << kTileLog2 && kMaxExperts <= 16, "a warp per expert");
  __shared__ int off[kMaxExperts + 1];
  __shared__ int total[kMaxExperts];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int Ee = E < 1 ? 1 : E;
  if (E > 1 && warp < E) {
    // exclusive scan of this expert's per-block counts
    int carry = 0;
    for (int b0 = 0; b0 < nblocks; b0 += 32 * kPer) {
      const int* src = block_counts + (long long)warp * nblocks + b0 + lane;
      int* dst = block_base + (long long)warp * nblocks + b0 + lane;
      int v[kPer], inc[kPer];
#pragma unroll
      for (int i = 0; i < kPer; ++i) v[i] = inc[i] = b0 + 32 * i + lane < nblocks ? __ldcg(src + 32 * i) : 0;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
          const int u = __shfl_up_sync(0xffffffffu, inc[i], d);
          if (lane >= d) inc[i] += u;
        }
      }
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        if (b0 + 32 * i + lane < nblocks) dst[32 * i] = carry + inc[i] - v[i];
        carry += __shfl_sync(0xffffffffu, inc[i], 31);
      }
    }
    if (lane == 0) total[warp] = carry;
  }
  __syncthreads();
  if (threadIdx.x <= Ee) {
    int run = threadIdx.x > 0 && E <= 1 ? T : 0;
    if (E > 1)
      for (int e = 0; e < threadIdx.x; ++e) run += total[e];
    off[threadIdx.x] = offsets[threadIdx.x] = run;
  }
  __syncthreads();

  const int mtiles = (T + kTileRows - 1) / kTileRows, mpairs = (mtiles + 1) / 2;
  for (int tile = threadIdx.x; tile <= mtiles; tile += blockDim.x) {
    int k = items_before(off, Ee, kTileLog2, tile);
    rt.tile_item_begin[tile] = k;
    if (tile == mtiles) { rt.n_items[0] = k; break; }
    const int r0 = tile * kTileRows, r1 = min(T, r0 + kTileRows);
    for (int e = 0; e < Ee; ++e) {
      const int lo = max(off[e], r0), hi = min(off[e + 1], r1);
      if (hi > lo) rt.items[k++] = make_int4(tile, e, lo - r0, hi - r0);
    }
  }
  // first item of each expert: the first item of the tile holding its first row, plus the items of the
  // non-empty experts below it in that tile; an empty expert points at its successor's first item
  if (threadIdx.x >= 480 && threadIdx.x - 480 <= Ee) {
    const int i = threadIdx.x - 480;
    int e = i;
    while (e < Ee && off[e + 1] == off[e]) ++e;
    const int tile = e < Ee ? off[e] >> kTileLog2 : mtiles;
    int idx = items_before(off, Ee, kTileLog2, tile);
    if (e < Ee)
      for (int f = 0; f < e; ++f) idx += off[f + 1] > off[f] && off[f + 1] > tile * kTileRows;
    rt.expert_item_begin[i] = idx;
  }
  // the same for pairs of tiles; the items of a tile are in expert order, so each expert of the pair takes the next one
  for (int pair = (int)blockDim.x - 1 - (int)threadIdx.x; pair <= mpairs; pair += blockDim.x) {
    int k = items_before(off, Ee, kTileLog2 + 1, pair);
    rt.pair_begin[pair] = k;
    if (pair == mpairs) break;
    const int r0 = pair * 2 * kTileRows, r1 = min(T, r0 + 2 * kTileRows), mid = r0 + kTileRows;
    int i0 = items_before(off, Ee, kTileLog2, 2 * pair), i1 = items_before(off, Ee, kTileLog2, 2 * pair + 1);
    for (int e = 0; e < Ee; ++e) {
      const int lo = max(off[e], r0), hi = min(off[e + 1], r1);
      if (hi > lo) rt.pair_items[k++] = make_int4(e, lo < mid ? i0++ : -1, hi > mid ? i1++ : -1, pair);
    }
  }
}

// ---------------------------------------------------------------------------
// K1: activation quantisation (Eq. 7-9), one to eight warps per token.  gamma_t = 128 /
// max(amax, 1e-5) (IEEE division), q = clamp(rint(x * gamma_t), -128, 127).
// Rows are written at their sorted position p (tokens ordered by expert,
// stable): q (int8), xt = q / gamma (bf16, the backward's operand) and, with
// routing, a bf16 copy of the row itself plus its gate and probabilities.
// ---------------------------------------------------------------------------
// Hidden activation of the 1-bit FFN (Eq. 11): bf16(silu(g) * u), element by element (fp32)
__device__ __forceinline__ uint4 swiglu8(const uint4& g, const uint4& u) {
  const uint32_t gw[4] = {g.x, g.y, g.z, g.w}, uw[4] = {u.x, u.y, u.z, u.w};
  uint32_t o[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float g0 = bf16lo(gw[j]), g1 = bf16hi(gw[j]);
    o[j] = pack_bf16x2(g0 / (1.0f + __expf(-g0)) * bf16lo(uw[j]), g1 / (1.0f + __expf(-g1)) * bf16hi(uw[j]));
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}

// SWIGLU: the row is made from gate and up (X = gate) on the way in and left in `mid`, instead of by a kernel that writes it for
// this one to read back: 2048 tokens x 5504 13.9 + 11.3 us as two launches, 22.5 us as one.
// WPR warps share one token row.  CH > 0: every lane keeps its CH 16-byte pieces of the row in registers
// between the absmax pass and the quantising pass (rows of up to 256 * CH * WPR elements), so X is read
// once; CH = 0 reads the row twice.
// Bound by memory (routed training layer: 7 bytes written and 2 read per value), and to reach it by the rows in flight: four
// pieces per lane and as many warps per row as that takes leave room for five blocks per SM; for rows of one warp, four: held to 48
// registers that form went to memory with 52 bytes a thread (8192 x 1024 with the forward tile 23.2 us, 21.3 so).  Eight pieces per lane (two blocks)
// and four, routed: 8192 x 2048 21.2 -> 17.3 us, 8192 x 5632 67 -> 58 us (5.6 TB/s); with the SwiGLU 38 -> 22.5 us.
template <int CH, int WPR, bool SWIGLU = false>
__global__ void __launch_bounds__(256, CH == 0 ? 2 : WPR == 1 ? 4 : 5) k_act_quant(const uint4* __restrict__ X, int T, int K, int E, const int* __restrict__ expert,
                                                   const int* __restrict__ block_base, const int* __restrict__ offsets,
                                                   const float* __restrict__ gate_tok, const float* __restrict__ probs_tok,
                                                   uint2* __restrict__ q, uint4* __restrict__ xt, uint4* __restrict__ xs,
                                                   float* __restrict__ gamma_s, float* __restrict__ gate_s, float* __restrict__ probs_s,
                                                   int* __restrict__ perm, int* __restrict__ pos, const uint4* __restrict__ norm_w,
                                                   const float* __restrict__ rms, const uint4* __restrict__ up, uint4* __restrict__ mid) {
  pdl_launch_dependents();   // launched with programmatic stream serialisation: see launch_pdl
  pdl_wait();
  __shared__ float amax_sh[8];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sub = warp % WPR, slot = sub * 32 + lane;   // this lane's first 16-byte piece of the row
  const int t_raw = blockIdx.x * (8 / WPR) + warp / WPR;
  const bool valid = t_raw < T;
  if (WPR == 1 && !valid) return;
  const int t = valid ? t_raw : T - 1;                  // idle warps of a shared row keep the barrier company
  const int chunks = K >> 3;
  const uint4* xrow = X + (long long)t * chunks;
  const float srow = norm_w ? rms[t] : 1.0f;
  auto fetch_x = [&](int c) {                      // with a fused RMSNorm every later step sees the normalised token
    const uint4 v = __ldg(xrow + c);
    if (SWIGLU) {
      const uint4 m = swiglu8(v, __ldg(up + (long long)t * chunks + c));
      if (valid) mid[(long long)t * chunks + c] = m;
      return m;
    }
    return norm_w ? rms_apply(v, srow, __ldg(norm_w + c)) : v;
  };
  uint4 held[CH > 0 ? CH : 1];
  float amax = 0.f;
  auto fold = [&](const uint4& v) {
    amax = fmaxf(amax, fmaxf(fmaxf(fabsf(bf16lo(v.x)), fabsf(bf16hi(v.x))), fmaxf(fabsf(bf16lo(v.y)), fabsf(bf16hi(v.y)))));
    amax = fmaxf(amax, fmaxf(fmaxf(fabsf(bf16lo(v.z)), fabsf(bf16hi(v.z))), fmaxf(fabsf(bf16lo(v.w)), fabsf(bf16hi(v.w)))));
  };
  if (CH > 0) {
#pragma unroll
    for (int i = 0; i < CH; ++i) {
      const int c = slot + 32 * WPR * i;
      held[i] = c < chunks ? fetch_x(c) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int i = 0; i < CH; ++i) fold(held[i]);
  } else {
    for (int c = slot; c < chunks; c += 32 * WPR) fold(fetch_x(c));
  }
  int p = t;
  if (E > 1) {
    const int e = expert[t];
    const int blk = t / kRouterTokensPerBlock, first = blk * kRouterTokensPerBlock;
    const int other = lane < kRouterTokensPerBlock && first + lane < T ? expert[first + lane] : -1;
    const unsigned same = __ballot_sync(0xffffffffu, other == e);
    const int rank = __popc(same & ((1u << (t - first)) - 1u));
    const int nblocks = (T + kRouterTokensPerBlock - 1) / kRouterTokensPerBlock;
    p = offsets[e] + block_base[(long long)e * nblocks + blk] + rank;
  }
  for (int d = 16; d > 0; d >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, d));
  if (WPR > 1) {
    if (lane == 0) amax_sh[warp] = amax;
    __syncthreads();
    const int w0 = warp - sub;
#pragma unroll
    for (int w = 0; w < WPR; ++w) amax = fmaxf(amax, amax_sh[w0 + w]);
    if (!valid) return;
  }
  const float gamma = __fdiv_rn(kActQmax, fmaxf(amax, kActAmaxFloor));
  const float inv_gamma = __fdiv_rn(1.0f, gamma);
  if (lane == 0 && sub == 0) {
    gamma_s[p] = gamma;
    perm[p] = t;
    pos[t] = p;
    gate_s[p] = (E > 1) ? gate_tok[t] : 1.0f;
  }
  if (E > 1 && sub == 0 && lane < E) probs_s[(long long)p * E + lane] = probs_tok[(long long)t * E + lane];
  uint2* qrow = q + (long long)p * chunks;
  uint4* xtrow = xt ? xt + (long long)p * chunks : nullptr;
  uint4* xsrow = xs ? xs + (long long)p * chunks : nullptr;
  auto emit = [&](int c, const uint4& v) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    int qi[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float lo = __fmul_rn(bf16lo(w[j]), gamma), hi = __fmul_rn(bf16hi(w[j]), gamma);
      qi[2 * j] = max(-128, min(127, __float2int_rn(lo)));
      qi[2 * j + 1] = max(-128, min(127, __float2int_rn(hi)));
    }
    uint2 qo;
    qo.x = (qi[0] & 0xFF) | ((qi[1] & 0xFF) << 8) | ((qi[2] & 0xFF) << 16) | ((qi[3] & 0xFF) << 24);
    qo.y = (qi[4] & 0xFF) | ((qi[5] & 0xFF) << 8) | ((qi[6] & 0xFF) << 16) | ((qi[7] & 0xFF) << 24);
    qrow[c] = qo;
    if (xtrow) {
      uint4 o;
      o.x = pack_bf16x2(qi[0] * inv_gamma, qi[1] * inv_gamma);
      o.y = pack_bf16x2(qi[2] * inv_gamma, qi[3] * inv_gamma);
      o.z = pack_bf16x2(qi[4] * inv_gamma, qi[5] * inv_gamma);
      o.w = pack_bf16x2(qi[6] * inv_gamma, qi[7] * inv_gamma);
      xtrow[c] = o;
    }
    if (xsrow) xsrow[c] = v;
  };
  if (CH > 0) {
#pragma unroll
    for (int i = 0; i < CH; ++i) {
      const int c = slot + 32 * WPR * i;
      if (c < chunks) emit(c, held[i]);
    }
  } else {
    for (int c = slot; c < chunks; c += 32 * WPR) emit(c, fetch_x(c));
  }
}

// What the products of the backward read, in one launch (blocks [0, rows) / [rows, signs) / [signs, end)):
//   dys[pos[t], :] = dY[t, :]             routed layers: the gradient rows in expert order, one warp per row
//   Sb[n,k] = bf16(scale_n) * S[n,k]      scale_n = beta_n (vector form) or 1
//   Ba[e,n,j] = bf16(alpha_n * B[e,n,j])  vector form only
// and the counters of the call's later kernels cleared (arrivals of k_finalize_scales; tickets and finished dH tiles of
// k_gemm_bwd).  Bound by memory; the three are independent and small enough that a launch of its own cost each of them
// as much as the work at a thousand tokens.
struct BwdPrepArgs {
  const uint4* dY; uint4* dys; const int* pos; int T, chunks;
  const uint4* s8; uint4* sb; const float* beta; int beta_stride, N, K;
  const uint4* B; uint4* ba; const float* alpha; int E, r;
  unsigned* counters;
  int rows, signs;
};
__global__ void __launch_bounds__(256) k_bwd_prep(BwdPrepArgs a) {
  pdl_launch_dependents();   // launched with programmatic stream serialisation: see launch_pdl
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x < 3) a.counters[threadIdx.x] = 0u;
  if ((int)blockIdx.x < a.rows) {
    const int t = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (t >= a.T) return;
    const uint4* s = a.dY + (long long)t * a.chunks;
    uint4* d = a.dys + (long long)a.pos[t] * a.chunks;
    int c = lane;
    for (; c + 96 < a.chunks; c += 128) {
      uint4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = __ldg(s + c + 32 * u);
#pragma unroll
      for (int u = 0; u < 4; ++u) d[c + 32 * u] = v[u];
    }
    for (; c < a.chunks; c += 32) d[c] = __ldg(s + c);
    return;
  }
  if ((int)blockIdx.x < a.signs) {
    const long long n16 = (long long)a.N * a.K / 16;
    const int per_row = a.K / 16;
    for (long long i = (blockIdx.x - a.rows) * 256LL + threadIdx.x; i < n16; i += (a.signs - a.rows) * 256LL) {
      const float sc = a.beta_stride ? a.beta[(int)(i / per_row)] : 1.0f;
      const uint4 v = __ldg(a.s8 + i);
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
      uint4 o[2];
      uint32_t* ow = reinterpret_cast<uint32_t*>(o);
      const uint32_t one = pack_bf16x2(sc, sc);            // +-1 bytes: bit 7 set <-> -1
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        ow[2 * j] = one ^ (((w[j] << 8) & 0x8000u) | ((w[j] << 16) & 0x80000000u));
        ow[2 * j + 1] = one ^ (((w[j] >> 8) & 0x8000u) | (w[j] & 0x80000000u));
      }
      a.sb[2 * i] = o[0];
      a.sb[2 * i + 1] = o[1];
    }
    return;
  }
  const long long n8 = (long long)a.E * a.N * a.r / 8;
  const int per_row = a.r / 8;
  for (long long i = (blockIdx.x - a.signs) * 256LL + threadIdx.x; i < n8; i += (gridDim.x - a.signs) * 256LL) {
    const float al = a.alpha[(int)((i / per_row) % a.N)];
    const uint4 v = __ldg(a.B + i);
    a.ba[i] = make_uint4(pack_bf16x2(bf16lo(v.x) * al, bf16hi(v.x) * al), pack_bf16x2(bf16lo(v.y) * al, bf16hi(v.y) * al),
                         pack_bf16x2(bf16lo(v.z) * al, bf16hi(v.z) * al), pack_bf16x2(bf16lo(v.w) * al, bf16hi(v.w) * al));
  }
}

// Feature-scale gradients from their per-tile partials:
//   dbeta_n = lam * sum_s dbeta_partial[s, n]      dalpha_n = sum_e dalpha_partial[e, n]
// A block takes 32 features; its eight warps take every eighth partial each (one trip to memory for up to 64 of them: a
// thread per feature that walked all 44 made six dependent trips), and the warps' sums are added in order.
// Vector scales: written per feature.  Scalar scales (blk_sums != null): every block adds its features in fp64 (fixed
// tree) into blk_sums[2 * block], the block that arrives last adds the blocks' sums in index order -- the result does
// not depend on which block that is -- and writes the two scalars; `arrivals` was cleared by an earlier kernel of the call.
__global__ void __launch_bounds__(256) k_finalize_scales(const float* __restrict__ dbeta_partial, int nslots,
                                                         const float* __restrict__ dalpha_partial, int E, int N,
                                                         const float* __restrict__ w_scales, float* __restrict__ dbeta,
                                                         float* __restrict__ dalpha, double* blk_sums, unsigned* arrivals) {
  pdl_launch_dependents();   // launched with programmatic stream serialisation: see launch_pdl
  pdl_wait();
  __shared__ float sh[2][8][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n = blockIdx.x * 32 + lane;
  float b = 0.f, a = 0.f;
  if (n < N) {
#pragma unroll 8
    for (int s = warp; s < nslots; s += 8) b += __ldcg(dbeta_partial + (long long)s * N + n);
    if (dalpha_partial) {
#pragma unroll 4
      for (int e = warp; e < E; e += 8) a += __ldcg(dalpha_partial + (long long)e * N + n);
    }
  }
  sh[0][warp][lane] = b;
  sh[1][warp][lane] = a;
  __syncthreads();
  if (warp > 0) return;
  b = a = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) { b += sh[0][w][lane]; a += sh[1][w][lane]; }
  b *= w_scales[0];
  if (!blk_sums) {
    if (n < N) {
      dbeta[n] = b;
      if (dalpha_partial) dalpha[n] = a;
    }
    return;
  }
  double sb = (double)b, sa = (double)a;
  for (int d = 16; d > 0; d >>= 1) {
    sb += __shfl_xor_sync(0xffffffffu, sb, d);
    sa += __shfl_xor_sync(0xffffffffu, sa, d);
  }
  unsigned last = 0u;
  if (lane == 0) {
    blk_sums[2 * blockIdx.x] = sb;
    blk_sums[2 * blockIdx.x + 1] = sa;
    __threadfence();
    last = atomicAdd(arrivals, 1u) == gridDim.x - 1;
  }
  if (!__shfl_sync(0xffffffffu, last, 0)) return;
  __threadfence();
  double tb = 0.0, ta = 0.0;
  for (int i = lane; i < (int)gridDim.x; i += 32) { tb += __ldcg(blk_sums + 2 * i); ta += __ldcg(blk_sums + 2 * i + 1); }
  for (int d = 16; d > 0; d >>= 1) {
    tb += __shfl_xor_sync(0xffffffffu, tb, d);
    ta += __shfl_xor_sync(0xffffffffu, ta, d);
  }
  if (lane == 0) {
    dbeta[0] = (float)tb;
    if (dalpha_partial) dalpha[0] = (float)ta;
  }
}

// ---------------------------------------------------------------------------
// INT8 high-precision branch (Sec. 3.2): the expert matrices quantised the way the 8-bit activations are
// (Eq. 7-9 with one scale per matrix): gamma = 128 / max(amax, 1e-5), code = clamp(rint(w * gamma), -128, 127).
// Matrix id = 2 e + (0: A_e [r,K], 1: B_e [N,r]); grid (blocks, 2 E).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_expert_amax(const uint4* __restrict__ A, const uint4* __restrict__ B, long long nA, long long nB,
                                                     uint32_t* amax_bits) {
  pdl_launch_dependents();
  pdl_wait();
  const int mat = blockIdx.y, e = mat >> 1;
  const long long n = (mat & 1) ? nB : nA;                      // 16-byte pieces (8 values) of one matrix
  const uint4* src = ((mat & 1) ? B : A) + (long long)e * n;
  float amax = 0.f;
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += gridDim.x * 256LL) {
    const uint4 v = __ldg(src + i);
    amax = fmaxf(amax, fmaxf(fmaxf(fabsf(bf16lo(v.x)), fabsf(bf16hi(v.x))), fmaxf(fabsf(bf16lo(v.y)), fabsf(bf16hi(v.y)))));
    amax = fmaxf(amax, fmaxf(fmaxf(fabsf(bf16lo(v.z)), fabsf(bf16hi(v.z))), fmaxf(fabsf(bf16lo(v.w)), fabsf(bf16hi(v.w)))));
  }
  for (int d = 16; d > 0; d >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, d));
  // non-negative floats order like their bit patterns; the maximum does not depend on the order of the updates
  if ((threadIdx.x & 31) == 0) atomicMax(amax_bits + mat, __float_as_uint(amax));
}

__global__ void __launch_bounds__(256) k_expert_quant(const uint4* __restrict__ A, const uint4* __restrict__ B, long long nA, long long nB,
                                                      const uint32_t* amax_bits, uint2* __restrict__ A8, uint2* __restrict__ B8,
                                                      float* __restrict__ hp_scales) {
  pdl_launch_dependents();
  pdl_wait();
  const int mat = blockIdx.y, e = mat >> 1;
  const long long n = (mat & 1) ? nB : nA;
  const uint4* src = ((mat & 1) ? B : A) + (long long)e * n;
  uint2* dst = ((mat & 1) ? B8 : A8) + (long long)e * n;
  const float gamma = __fdiv_rn(kActQmax, fmaxf(__uint_as_float(__ldcg(amax_bits + mat)), kActAmaxFloor));
  if (blockIdx.x == 0 && threadIdx.x == 0) hp_scales[mat] = gamma;
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < n; i += gridDim.x * 256LL) {
    const uint4 v = __ldg(src + i);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    int qi[8];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      qi[2 * j] = max(-128, min(127, __float2int_rn(__fmul_rn(bf16lo(w[j]), gamma))));
      qi[2 * j + 1] = max(-128, min(127, __float2int_rn(__fmul_rn(bf16hi(w[j]), gamma))));
    }
    uint2 o;
    o.x = (qi[0] & 0xFF) | ((qi[1] & 0xFF) << 8) | ((qi[2] & 0xFF) << 16) | ((qi[3] & 0xFF) << 24);
    o.y = (qi[4] & 0xFF) | ((qi[5] & 0xFF) << 8) | ((qi[6] & 0xFF) << 16) | ((qi[7] & 0xFF) << 24);
    dst[i] = o;
  }
}

cudaError_t launch_pack_experts(const uint16_t* A, const uint16_t* B, int E, int r, int K, int N, int8_t* A8, int8_t* B8, float* hp_scales,
                                uint32_t* amax_bits, cudaStream_t st) {
  const long long nA = (long long)r * K / 8, nB = (long long)N * r / 8;
  if (cudaMemsetAsync(amax_bits, 0, sizeof(uint32_t) * 2 * E, st) != cudaSuccess) return cudaGetLastError();
  long long g = ((nA > nB ? nA : nB) + 1023) / 1024;
  const int gx = (int)(g < 1 ? 1 : (g > 296 ? 296 : g));
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)gx, (unsigned)(2 * E), 1); cfg.blockDim = dim3(256, 1, 1); cfg.stream = st;
  cfg.attrs = attr; cfg.numAttrs = 0;     // the first kernel follows a memset: plain stream order
  { LaunchScope ls(KID_PACK_SUMS, st);
    cudaLaunchKernelEx(&cfg, k_expert_amax, reinterpret_cast<const uint4*>(A), reinterpret_cast<const uint4*>(B), nA, nB, amax_bits); }
  cfg.numAttrs = 1;
  { LaunchScope ls(KID_BINARIZE_PACK, st);
    cudaLaunchKernelEx(&cfg, k_expert_quant, reinterpret_cast<const uint4*>(A), reinterpret_cast<const uint4*>(B), nA, nB,
                       static_cast<const uint32_t*>(amax_bits), reinterpret_cast<uint2*>(A8), reinterpret_cast<uint2*>(B8), hp_scales); }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FFN-level decoupling (Eq. 11): the small kernel between the INT8 FFN's projections (the 1-bit FFN's is part of
// the quantiser).
// ---------------------------------------------------------------------------
// Hidden activation of the INT8 FFN, one warp per token: from the exact sums g_int = G8 q, u_int = U8 q
//   g = fl(fl(g_int) * fl(1 / fl(gamma_G gamma_t))), u likewise, m = fl(fl(g * s) * u) with the logistic factor s taken
//   in fp64 and rounded once to fp32 (an fp32 exponential would not be reproducible, and m feeds a quantiser),
// then Eq. 7-9 on the row of m: gamma_m = 128 / max(max|m|, 1e-5), codes clamp(rint(m gamma_m)).  r <= 128.
__global__ void __launch_bounds__(256) k_ffn8_act(const int* __restrict__ g_int, const int* __restrict__ u_int, const float* __restrict__ gamma,
                                                  const float* __restrict__ hp_scales, int T, int r, int8_t* __restrict__ qm,
                                                  float* __restrict__ gamma_m) {
  pdl_launch_dependents();
  pdl_wait();
  const int t = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (t >= T) return;
  const float gt = gamma[t];
  const float deq_g = __fdiv_rn(1.0f, __fmul_rn(hp_scales[0], gt)), deq_u = __fdiv_rn(1.0f, __fmul_rn(hp_scales[1], gt));
  float m[4];
  float amax = 0.f;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int j = lane + 32 * k;
    m[k] = 0.f;
    if (j < r) {
      const float g = __fmul_rn(__int2float_rn(g_int[(long long)t * r + j]), deq_g);
      const float u = __fmul_rn(__int2float_rn(u_int[(long long)t * r + j]), deq_u);
      const float s = (float)(1.0 / (1.0 + exp(-(double)g)));
      m[k] = __fmul_rn(__fmul_rn(g, s), u);
      amax = fmaxf(amax, fabsf(m[k]));
    }
  }
  for (int d = 16; d > 0; d >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, d));
  const float gm = __fdiv_rn(kActQmax, fmaxf(amax, kActAmaxFloor));
  if (lane == 0) gamma_m[t] = gm;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int j = lane + 32 * k;
    if (j < r) qm[(long long)t * r + j] = (int8_t)max(-128, min(127, __float2int_rn(__fmul_rn(m[k], gm))));
  }
}

cudaError_t launch_ffn8_act(const int* g_int, const int* u_int, const float* gamma, const float* hp_scales, int T, int r, int8_t* qm,
                            float* gamma_m, cudaStream_t st) {
  launch_pdl(k_ffn8_act, (T + 7) / 8, 256, 0, st, g_int, u_int, gamma, hp_scales, T, r, qm, gamma_m);
  ++g_launches;
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// host launchers
// ---------------------------------------------------------------------------
static inline int grid_for(long long work, int per_block, int cap) {
  long long g = (work + per_block - 1) / per_block;
  if (g < 1) g = 1;
  return (int)(g > cap ? cap : g);
}

cudaError_t launch_pack(const float* W, int N, int K, uint32_t* bits, int8_t* s8, float* scales, double* partial, cudaStream_t st) {
  const long long n4 = (long long)N * K / 4;
  const int nparts = grid_for(n4, 256 * 8, 6 * 148);   // six blocks per SM, each thread keeps four loads in flight (~14 MB in all)
  static_assert(6 * 148 <= kPackPartials, "partial sums of the weight reduction");
  { LaunchScope ls(KID_PACK_SUMS, st);
  launch_pdl(k_weight_partial_sums, nparts, 256, 0, st, reinterpret_cast<const float4*>(W), n4, partial); }
  const int grid = grid_for(n4, 256 * 4, 148 * 8);
  LaunchScope ls(KID_BINARIZE_PACK, st);
  launch_pdl(k_binarize_pack, grid, 256, 0, st, reinterpret_cast<const float4*>(W), n4, partial, nparts, 1.0 / ((double)N * K), bits,
                                        reinterpret_cast<uint32_t*>(s8), scales);
  return cudaGetLastError();
}

// The router's opt-in limit is set once per device, to the largest request: it belongs to the kernel, not to a launch, so that a
// call which set a smaller one would take it from under a call of another thread, or from under a launch recorded in a CUDA graph.
// The quantiser of long SwiGLU rows asks for shared memory that it does not use, under the same limit.
constexpr int kRouterSmemLimit = 116 * 1024;
static_assert(router_smem<kMaxExperts>() <= kRouterSmemLimit, "the bare ring fits too");
static cudaError_t smem_limits() {
  constexpr int kMaxDevices = 64;
  static std::once_flag done[kMaxDevices];
  static cudaError_t result[kMaxDevices] = {};
  int dev = 0;
  if (const cudaError_t e = cudaGetDevice(&dev)) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::call_once(done[dev], [&] {
    auto set = [](auto k) { return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kRouterSmemLimit); };
    result[dev] = set(k_router<4>);
    if (result[dev] == cudaSuccess) result[dev] = set(k_router<8>);
    if (result[dev] == cudaSuccess) result[dev] = set(k_router<kMaxExperts>);
    if (result[dev] == cudaSuccess) result[dev] = set(k_act_quant<0, 1, true>);
  });
  return result[dev];
}
// Shared memory to ask for so that an SM holds no more blocks of this grid than an even spread puts there (`most` at most, else what is
// needed): they become resident while the kernel before ends, and the SMs that end first would otherwise take all they can hold.
// One more block of each size, with the KB that every block takes beside it, is more than the 228 KB of an SM.
static int smem_for_spread(int grid, int most, int needed) {
  constexpr int kKB[] = {kRouterSmemLimit / 1024, 76, 57, 45, 38};
  const int per_sm = (grid + sm_count() - 1) / sm_count();
  return per_sm <= most ? kKB[per_sm - 1] * 1024 : needed;
}

cudaError_t launch_route_and_quant(const uint16_t* X, const uint16_t* Wr, int T, int K, int E, const SavedPtrs& sv, const FwdScratch& sc,
                                   cudaStream_t st, cudaStream_t st_quant, const uint16_t* norm_weight, float norm_eps, const uint16_t* up, uint16_t* mid, bool tables) {
  if (E > 1) st_quant = st;   // the sorted position of a token comes from the router and the scan
  const uint4* nw = reinterpret_cast<const uint4*>(norm_weight);
  if (nw) {
    st_quant = st;
    LaunchScope ls(KID_ROUTER, st);
    launch_pdl(k_row_rms, (T + 7) / 8, 256, 0, st, reinterpret_cast<const uint4*>(X), T, K, norm_eps, sc.rms);
  }
  const int nblocks = (T + kRouterTokensPerBlock - 1) / kRouterTokensPerBlock;
  if (E > 1) {
    LaunchScope ls(KID_ROUTER, st);
    auto kern = k_router<kMaxExperts>;
    int smem = router_smem<kMaxExperts>();
    if (E <= 4) { kern = k_router<4>; smem = router_smem<4>(); }
    else if (E <= 8) { kern = k_router<8>; smem = router_smem<8>(); }
    smem = smem_for_spread(nblocks, 2, smem);     // 2048 tokens x 3200: 17 us without this, 10 with it
    if (const cudaError_t e = smem_limits()) return e;
    const cudaError_t e = launch_pdl(kern, nblocks, 32 * kRouterWarps, smem, st, reinterpret_cast<const uint4*>(X), reinterpret_cast<const uint4*>(Wr), T, K,
                                     E, sv.expert, sc.gate_tok, sc.probs_tok, sc.block_counts, nw, sc.rms);
    if (e != cudaSuccess) return e;   // the kernels behind this one store where its counts say
  }
  if (tables) {
    LaunchScope ls(KID_ROUTE_SCAN, st);
    if (const cudaError_t e = launch_pdl(k_route_scan, 1, 512, 0, st, T, E, nblocks, sc.block_counts, sc.block_base, sv.offsets, sv.rt)) return e;
  }
  LaunchScope ls(KID_ACT_QUANT, st_quant);
  const int per_lane = (K / 8 + 31) / 32;   // 16-byte pieces of a row per lane if one warp took the whole row
  auto kern = up ? k_act_quant<0, 1, true> : k_act_quant<0, 1>;
  int wpr = 1;
  if (per_lane <= 4) kern = up ? k_act_quant<4, 1, true> : k_act_quant<4, 1>;
  else if (per_lane <= 8) { kern = up ? k_act_quant<4, 2, true> : k_act_quant<4, 2>; wpr = 2; }
  else if (per_lane <= 16) { kern = up ? k_act_quant<4, 4, true> : k_act_quant<4, 4>; wpr = 4; }
  else if (per_lane <= 32) { kern = up ? k_act_quant<4, 8, true> : k_act_quant<4, 8>; wpr = 8; }
  const int rows_per_block = 8 / wpr, grid = (T + rows_per_block - 1) / rows_per_block;
  // A warp with a SwiGLU row that no registers hold is bound by the instructions of two passes, and directly behind the gate / up tile the
  // blocks of a short batch would share the first few SMs that are free.  Whole FFN form, behind two other kernels / there / there
  // and spread, replayed from a graph: 1024 tokens of 512 and 8640 127 / 183 / 108 us, 512 of 3200 and 8640 169-198 / 173 / 117, 256 of 512 and
  // 8640 123 / 131 / 94, 2048 of 3200 and 8640 302 / 275 / 226.  Rows in registers are bound by memory and do not differ (1024 of 2048
  // and 5504 64.5 / 64.6).
  size_t smem = 0;
  if (up && per_lane > 32) {
    if (const cudaError_t e = smem_limits()) return e;
    smem = smem_for_spread(grid, 5, 0);
  }
  launch_pdl(kern, grid, 256, smem, st_quant, reinterpret_cast<const uint4*>(X), T, K, E, sv.expert, sc.block_base, sv.offsets, sc.gate_tok,
                                    sc.probs_tok, reinterpret_cast<uint2*>(sv.q), reinterpret_cast<uint4*>(sv.xt),
                                    reinterpret_cast<uint4*>(sv.xs), sv.gamma, sv.gate, sv.probs, sv.perm, sv.pos, nw, sc.rms,
                                    reinterpret_cast<const uint4*>(up), reinterpret_cast<uint4*>(mid));
  return cudaGetLastError();
}

cudaError_t launch_bwd_prep(const LayerArgs& a, const uint16_t* dY, uint16_t* dys, const int* pos, const int8_t* s8, uint16_t* sb,
                            uint16_t* ba, unsigned* counters, cudaStream_t st) {
  BwdPrepArgs p{};
  p.dY = reinterpret_cast<const uint4*>(dY); p.dys = reinterpret_cast<uint4*>(dys); p.pos = pos; p.T = a.T; p.chunks = a.N / 8;
  p.s8 = reinterpret_cast<const uint4*>(s8); p.sb = reinterpret_cast<uint4*>(sb); p.beta = a.beta; p.beta_stride = a.scale_stride;
  p.N = a.N; p.K = a.K;
  p.B = reinterpret_cast<const uint4*>(a.B); p.ba = reinterpret_cast<uint4*>(ba); p.alpha = a.alpha; p.E = a.E; p.r = a.r;
  p.counters = counters;
  p.rows = dys ? (a.T + 7) / 8 : 0;
  p.signs = p.rows + grid_for((long long)a.N * a.K / 16, 256 * 2, 148 * 8);
  const int end = p.signs + (ba ? grid_for((long long)a.E * a.N * a.r / 8, 256 * 2, 148 * 8) : 0);
  LaunchScope ls(KID_SCALED_SIGN, st);
  launch_pdl(k_bwd_prep, end, 256, 0, st, p);
  return cudaGetLastError();
}

cudaError_t launch_finalize_scales(const float* dbeta_partial, int nslots, const float* dalpha_partial, int E, int N, const float* w_scales,
                                   int vec, float* dbeta, float* dalpha, double* blk_sums, unsigned* arrivals, cudaStream_t st) {
  LaunchScope ls(vec ? KID_SUM_PARTIALS : KID_SUM_SCALAR, st);
  launch_pdl(k_finalize_scales, (N + 31) / 32, 256, 0, st, dbeta_partial, nslots, dalpha_partial, E, N, w_scales, dbeta, dalpha,
             vec ? nullptr : blk_sums, vec ? nullptr : arrivals);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// experts' down-projections side by side: out[n, e r + j] = B[e, n, j] (the all-experts test mode of the forward)
// ---------------------------------------------------------------------------
__global__ void k_concat_experts(const uint4* __restrict__ B, uint4* __restrict__ out, int E, int N, int r8) {
  const long long o = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= (long long)N * E * r8) return;
  const int jc = (int)(o % r8);
  const long long t = o / r8;
  const int e = (int)(t % E);
  const long long n = t / E;
  out[o] = B[((long long)e * N + n) * r8 + jc];
}
cudaError_t launch_concat_experts(const uint16_t* B, int E, int N, int r, uint16_t* out, cudaStream_t st) {
  const long long total = (long long)N * E * (r / 8);
  LaunchScope ls(KID_SCATTER_ROWS, st);
  k_concat_experts<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(reinterpret_cast<const uint4*>(B), reinterpret_cast<uint4*>(out), E, N, r / 8);
  return cudaGetLastError();
}

}  // namespace pq
