// Channel mask m_s by top-k (Sec. 4.1 second indicator, top-k form of the appendix) with a cluster of blocks per token.
//
// Exact k2-th score by three radix steps (11 + 10 + 10 bits) over per-block histograms that the blocks of the
// cluster read from each other's shared memory, then the ordered list of the kept channels (ties: lower channel first).
// One block per token did this in 13.9 us (eight tokens, 12288 channels, from the proxy sums) and 11.7 us (one token,
// from scores): the scores of a token fall into few bins, and the increments of a bin in one SM's shared memory go one by
// one.  With the channels spread over eight blocks: 11.8 and 10.4 us (cold, under the
// profiler; most of what is left are the five cluster barriers and the reads behind them).
#pragma once

#include <cooperative_groups.h>

#include "prox_kernels.cuh"

namespace prox {

constexpr int kTkThreads = 512;
constexpr int kTkBlocks = 8;             // blocks of a cluster (the portable size); each takes an eighth of the channels

// Bin of the k-th largest (k >= 1) over 512 * N bins; thread t holds the counts of bins top, top - 1, .. with
// top = 512 * N - 1 - N * t.  res[0] = bin, res[1] = elements above it.  All 512 threads call.
template <int N>
__device__ __forceinline__ void kth_of_counts(const unsigned (&c)[N], unsigned k, unsigned* wsum, unsigned* res) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned s = 0;
#pragma unroll
  for (int j = 0; j < N; ++j) s += c[j];
  unsigned inc = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  unsigned run = __reduce_add_sync(0xffffffffu, lane < warp ? wsum[lane] : 0u) + inc - s;
  if (run < k && k <= run + s) {
    const unsigned top = (unsigned)(kTkThreads * N - 1 - N * (int)threadIdx.x);
#pragma unroll
    for (int j = 0; j < N; ++j) {
      if (run < k && k <= run + c[j]) { res[0] = top - (unsigned)j; res[1] = run; }
      run += c[j];
    }
  }
  __syncthreads();
}

enum ScoreSource { kFromScores = 0, kFromSums, kSharedSums };

// Cluster b of the grid is token b.  SRC: where the scores come from
//   kFromScores    scores[b][F]
//   kFromSums      |up~ SiLU(gate~)| of the proxy sums pacc [token][gate | up][F], which are cleared for the next call
//   kSharedSums    one mask for the batch: these scores added token after token in fp32 (one cluster); the list goes to
//                  every token's row
// From the sums, the tokens' scores are also written to scores[b][F] if that is given.  (A kernel of its own that formed
// and wrote them, in front of this one: 44 us for Stage 1 of eight tokens with scores at 4096 x 12288 against 32.)
// cmask: a byte per channel with the tokens' bits (NULL: not wanted).  Dynamic shared memory: the block's scores.
template <int SRC>
__global__ void __cluster_dims__(kTkBlocks, 1, 1) __launch_bounds__(kTkThreads)
channel_topk_kernel(float* __restrict__ scores, float* __restrict__ pacc, int B, int F, int k2, int* __restrict__ sel_out,
                    int sel_stride, unsigned* __restrict__ cmask) {
  constexpr int NT = kTkThreads;
  constexpr bool SHARED = SRC == kSharedSums, SUMS = SRC != kFromScores;
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ __align__(16) uint8_t tk_smem[];
  uint4* skey = reinterpret_cast<uint4*>(tk_smem);               // score bits of the block's channels, four a piece
  __shared__ __align__(16) unsigned hist[4096];                  // 2048 | 1024 | 1024 bins of the three steps
  __shared__ unsigned wsum[32], res[2], total;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x / kTkBlocks, rank = blockIdx.x % kTkBlocks;
  const int nq = F / 4, q0 = (int)((long long)nq * rank / kTkBlocks), n = (int)((long long)nq * (rank + 1) / kTkBlocks) - q0;
  for (int i = tid; i < 1024; i += NT) reinterpret_cast<uint4*>(hist)[i] = make_uint4(0u, 0u, 0u, 0u);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __syncthreads();
  for (int i = tid; i < n; i += NT) {
    const int q = q0 + i;
    float s[4] = {0.f, 0.f, 0.f, 0.f};
    if (SUMS) {
      const int b0 = SHARED ? 0 : b, b1 = SHARED ? B : b + 1;
      float4 g[SHARED ? 8 : 1], u[SHARED ? 8 : 1];
#pragma unroll
      for (int t = 0; t < (SHARED ? 8 : 1); ++t) {               // all loads before the first store
        if (b0 + t < b1) {
          const float4* pg = reinterpret_cast<const float4*>(pacc + (size_t)(b0 + t) * 2 * F) + q;
          g[t] = __ldcg(pg); u[t] = __ldcg(pg + F / 4);
        }
      }
#pragma unroll
      for (int t = 0; t < (SHARED ? 8 : 1); ++t) {
        if (b0 + t < b1) {
          float4* pg = reinterpret_cast<float4*>(pacc + (size_t)(b0 + t) * 2 * F) + q;
          pg[0] = make_float4(0.f, 0.f, 0.f, 0.f); pg[F / 4] = make_float4(0.f, 0.f, 0.f, 0.f);
          const float4 v = make_float4(fabsf(u[t].x * silu_fast(g[t].x)), fabsf(u[t].y * silu_fast(g[t].y)),
                                       fabsf(u[t].z * silu_fast(g[t].z)), fabsf(u[t].w * silu_fast(g[t].w)));
          if (scores) reinterpret_cast<float4*>(scores + (size_t)(b0 + t) * F)[q] = v;
          s[0] += v.x; s[1] += v.y; s[2] += v.z; s[3] += v.w;
        }
      }
    } else {
      const float4 v = __ldcg(reinterpret_cast<const float4*>(scores + (size_t)b * F) + q);
      // (scores are magnitudes; whatever a Stage 1 that gave up has left in the buffer must order like one too, or more
      // or fewer than k2 channels would pass)
      s[0] = fabsf(v.x); s[1] = fabsf(v.y); s[2] = fabsf(v.z); s[3] = fabsf(v.w);
    }
    const uint4 k = make_uint4(__float_as_uint(s[0]), __float_as_uint(s[1]), __float_as_uint(s[2]), __float_as_uint(s[3]));
    skey[i] = k;
    atomicAdd(&hist[k.x >> 20], 1u); atomicAdd(&hist[k.y >> 20], 1u); atomicAdd(&hist[k.z >> 20], 1u); atomicAdd(&hist[k.w >> 20], 1u);
  }
  // Only now: blocks of the next kernel that start earlier take issue slots from the histograms (one mask for eight
  // tokens, two calls: 146.4 -> 145.1 us; stages one by one, two layers: 91.8 -> 90.8; the other batch cases equal).
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  cl.sync();
  unsigned prefix, kleft = (unsigned)k2;
  {
    unsigned c[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int r = 0; r < kTkBlocks; ++r) {
      const uint4 h = reinterpret_cast<const uint4*>(cl.map_shared_rank(hist, r))[511 - tid];
      c[0] += h.w; c[1] += h.z; c[2] += h.y; c[3] += h.x;
    }
    kth_of_counts<4>(c, kleft, wsum, res);
    prefix = res[0]; kleft -= res[1];
  }
#pragma unroll
  for (int step = 0; step < 2; ++step) {
    unsigned* h = hist + 2048 + 1024 * step;
    const int sh = 10 - 10 * step;
    for (int i = tid; i < n; i += NT) {
      const uint4 kv = skey[i];
      const unsigned k4[4] = {kv.x, kv.y, kv.z, kv.w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if ((k4[e] >> (sh + 10)) == prefix) atomicAdd(&h[(k4[e] >> sh) & 1023u], 1u);
    }
    cl.sync();
    unsigned c[2] = {0u, 0u};
#pragma unroll
    for (int r = 0; r < kTkBlocks; ++r) {
      const uint2 v = reinterpret_cast<const uint2*>(cl.map_shared_rank(h, r))[511 - tid];
      c[0] += v.y; c[1] += v.x;
    }
    kth_of_counts<2>(c, kleft, wsum, res);
    prefix = (prefix << 10) | res[0]; kleft -= res[1];
  }
  const unsigned T = prefix, quota = kleft;
  // ordered list: a thread owns a run of quads; the blocks in front add their totals (above T | ties << 16)
  const int qpt = (n + NT - 1) / NT, i0 = min(n, tid * qpt), i1 = min(n, i0 + qpt);
  unsigned cnt = 0;
  for (int i = i0; i < i1; ++i) {
    const uint4 kv = skey[i];
    cnt += ((kv.x > T) + (kv.y > T) + (kv.z > T) + (kv.w > T)) + (((kv.x == T) + (kv.y == T) + (kv.z == T) + (kv.w == T)) << 16);
  }
  unsigned inc = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  const unsigned wv = lane < NT / 32 ? wsum[lane] : 0u;          // (at most 8192 channels per block: 16 bits each)
  const unsigned ex = __reduce_add_sync(0xffffffffu, lane < warp ? wv : 0u) + inc - cnt;
  if (tid == NT - 1) total = ex + cnt;
  cl.sync();
  const unsigned tot = lane < rank ? *cl.map_shared_rank(&total, lane) : 0u;
  unsigned rg = __reduce_add_sync(0xffffffffu, tot & 0xffffu) + (ex & 0xffffu);
  unsigned re = __reduce_add_sync(0xffffffffu, tot >> 16) + (ex >> 16);
  cl.barrier_arrive();                                           // (no block reads another's shared memory after that)
  for (int i = i0; i < i1; ++i) {
    const uint4 kv = skey[i];
    const unsigned k4[4] = {kv.x, kv.y, kv.z, kv.w};
    unsigned bits = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const bool gt = k4[e] > T, eq = k4[e] == T;
      if (gt || (eq && re < quota)) {
        const int ch = (q0 + i) * 4 + e;
        const unsigned pos = rg + min(re, quota);
        if (SHARED) for (int t = 0; t < B; ++t) sel_out[(size_t)t * sel_stride + pos] = ch;
        else sel_out[(size_t)b * sel_stride + pos] = ch;
        bits |= (SHARED ? (1u << B) - 1u : 1u << b) << (8 * e);
      }
      rg += gt ? 1u : 0u; re += eq ? 1u : 0u;
    }
    if (cmask && bits) {
      if (SHARED) cmask[q0 + i] = bits; else atomicOr(cmask + q0 + i, bits);
    }
  }
  cl.barrier_wait();
}

}  // namespace prox
