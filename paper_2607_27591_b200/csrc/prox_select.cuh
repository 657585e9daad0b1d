// Channel mask m_s by top-k (Sec. 4.1 second indicator, top-k form of the appendix): one block or a cluster of blocks per token.
//
// Exact k2-th score by three radix steps (11 + 10 + 10 bits) over histograms in shared memory (of a cluster: per block, and the
// blocks read each other's), then the ordered list of the kept channels (ties: lower channel first).
// The scores of a token fall into few bins, and the increments of a bin in one SM's shared memory go one by one; with the
// channels spread over eight blocks that is an eighth, but the cluster's five barriers and the reads of other blocks'
// memory behind them cost 5 us whatever the size.  Stage 1 of a 256-wide layer, us per call in a graph, one block | cluster:
//   one token     64 channels 10.5 | 15.8, 4096: 12.3 | 17.0, 8192: 14.1 | 17.4, 12288: 15.6 | 17.9, 14336: 17.0 | 18.0
//   two tokens    64: 9.5 | 14.7, 4096: 11.4 | 15.5, 10240: 15.9 | 17.1, 12288: 17.0 | 17.3
//   eight tokens  64: 9.9 | 14.9, 4096: 12.0 | 15.8, 10240: 16.9 | 17.4, 12288: 17.9 | 17.5
// so one block takes up to 12288 channels for one token and 10240 for several.  It has 1024 threads: with 512, eight
// tokens: 2048 channels 10.6 us against 11.0, 8192: 15.9 against 14.6.
#pragma once

#include <cooperative_groups.h>

#include "prox_kernels.cuh"

namespace prox {

constexpr int kTkBlocks = 8;             // blocks of a cluster (the portable size); each takes an eighth of the channels
constexpr int kTkOneBlock = 12288, kTkOneBlockBatch = 10240;     // channels that one block takes (see above)

// Bin of the k-th largest (k >= 1) over NT * N bins; thread t holds the counts of bins top, top - 1, .. with
// top = NT * N - 1 - N * t.  res[0] = bin, res[1] = elements above it.  All NT threads call.
template <int NT, int N>
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
    const unsigned top = (unsigned)(NT * N - 1 - N * (int)threadIdx.x);
#pragma unroll
    for (int j = 0; j < N; ++j) {
      if (run < k && k <= run + c[j]) { res[0] = top - (unsigned)j; res[1] = run; }
      run += c[j];
    }
  }
  __syncthreads();
}

__device__ __forceinline__ float4 proxy_score4(const float4& g, const float4& u) {
  return make_float4(fabsf(u.x * silu_fast(g.x)), fabsf(u.y * silu_fast(g.y)), fabsf(u.z * silu_fast(g.z)), fabsf(u.w * silu_fast(g.w)));
}

// c += the counts of a thread's N bins, in descending order
template <int N>
__device__ __forceinline__ void add_counts(const unsigned* h, int from_top, unsigned (&c)[N]) {
  if constexpr (N == 4) {
    const uint4 v = reinterpret_cast<const uint4*>(h)[from_top];
    c[0] += v.w; c[1] += v.z; c[2] += v.y; c[3] += v.x;
  } else if constexpr (N == 2) {
    const uint2 v = reinterpret_cast<const uint2*>(h)[from_top];
    c[0] += v.y; c[1] += v.x;
  } else {
    c[0] += h[from_top];
  }
}

// One mask for the batch: the tokens' scores |up~ SiLU(gate~)| of the proxy sums pacc [token][gate | up][F], added token
// after token in fp32, to `out`; also to scores[b][F] if the caller wants them.  The sums are cleared for the next call.
// On all SMs: one cluster of the top-k kernel that read the sums of all tokens itself took 3 us longer than this and that
// kernel on the summed scores for eight tokens and 3072 channels (32.3 -> 29.0 us per call at 1024 x 3072).
__global__ void __launch_bounds__(128)
shared_score_kernel(float* __restrict__ pacc, int B, int F, float* __restrict__ scores, float* __restrict__ out) {
  pdl_enter();
  const int q = blockIdx.x * 128 + threadIdx.x;
  if (q >= F / 4) return;
  float4 g[8], u[8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {                                  // all loads before the first store
    if (t < B) {
      const float4* pg = reinterpret_cast<const float4*>(pacc + (size_t)t * 2 * F) + q;
      g[t] = __ldcg(pg); u[t] = __ldcg(pg + F / 4);
    }
  }
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    if (t < B) {
      float4* pg = reinterpret_cast<float4*>(pacc + (size_t)t * 2 * F) + q;
      pg[0] = make_float4(0.f, 0.f, 0.f, 0.f); pg[F / 4] = make_float4(0.f, 0.f, 0.f, 0.f);
      const float4 v = proxy_score4(g[t], u[t]);
      if (scores) reinterpret_cast<float4*>(scores + (size_t)t * F)[q] = v;
      s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
  }
  reinterpret_cast<float4*>(out)[q] = s;
}

enum TopkForm { kFromScores = 0, kFromSums, kFromSumsOut, kRepeated };

// Block or cluster b of the grid is token b.  FORM (instantiations of their own: what a call does not need costs it 0.4 us
// each, code that runs once is fetched cold):
//   kFromScores    by scores[b][F]
//   kFromSums      by the scores of the proxy sums pacc [token][gate | up][F], which are cleared for the next call
//   kFromSumsOut   the same, and the scores are written to scores[b][F].  (A kernel of its own that formed and wrote them,
//                  in front of this one: 44 us for Stage 1 of eight tokens with scores at 4096 x 12288 against 32.)
//   kRepeated      kFromScores with one list for `tokens` tokens, written to every token's row
// cmask: a byte per channel with the tokens' bits (NULL: not wanted); one list is for tokens b * tokens and the next ones.
// Dynamic shared memory: the block's scores.
template <int FORM, int NB, int NT>
__device__ __forceinline__ void channel_topk(float* __restrict__ scores, float* __restrict__ pacc, int F, int k2, int* __restrict__ sel_out,
                                             int sel_stride, int tokens, unsigned* __restrict__ cmask) {
  constexpr bool SUMS = FORM == kFromSums || FORM == kFromSumsOut;
  constexpr int N1 = 2048 / NT, N2 = 1024 / NT;                  // bins of a thread: first step, the others
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  auto sync = [&]() { if constexpr (NB > 1) cl.sync(); else __syncthreads(); };
  auto of_rank = [&](unsigned* p, int r) -> unsigned* { if constexpr (NB > 1) return cl.map_shared_rank(p, r); else return p; };
  extern __shared__ __align__(16) uint8_t tk_smem[];
  uint4* skey = reinterpret_cast<uint4*>(tk_smem);               // score bits of the block's channels, four a piece
  __shared__ __align__(16) unsigned hist[4096];                  // 2048 | 1024 | 1024 bins of the three steps
  __shared__ unsigned wsum[32], res[2], span[2], total;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x / NB, rank = blockIdx.x % NB;
  const int nq = F / 4, q0 = (int)((long long)nq * rank / NB), n = (int)((long long)nq * (rank + 1) / NB) - q0;
  for (int i = tid; i < 1024; i += NT) reinterpret_cast<uint4*>(hist)[i] = make_uint4(0u, 0u, 0u, 0u);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __syncthreads();
  for (int i = tid; i < n; i += NT) {
    const int q = q0 + i;
    float4 s;
    if (SUMS) {
      float4* pg = reinterpret_cast<float4*>(pacc + (size_t)b * 2 * F) + q;
      const float4 g = __ldcg(pg), u = __ldcg(pg + F / 4);
      pg[0] = make_float4(0.f, 0.f, 0.f, 0.f); pg[F / 4] = make_float4(0.f, 0.f, 0.f, 0.f);
      s = proxy_score4(g, u);
      if (FORM == kFromSumsOut) reinterpret_cast<float4*>(scores + (size_t)b * F)[q] = s;
    } else {
      // (scores are magnitudes; whatever a Stage 1 that gave up has left in the buffer must order like one too, or more
      // or fewer than k2 channels would pass)
      const float4 v = __ldcg(reinterpret_cast<const float4*>(scores + (size_t)b * F) + q);
      s = make_float4(fabsf(v.x), fabsf(v.y), fabsf(v.z), fabsf(v.w));
    }
    const uint4 k = make_uint4(__float_as_uint(s.x), __float_as_uint(s.y), __float_as_uint(s.z), __float_as_uint(s.w));
    skey[i] = k;
    atomicAdd(&hist[k.x >> 20], 1u); atomicAdd(&hist[k.y >> 20], 1u); atomicAdd(&hist[k.z >> 20], 1u); atomicAdd(&hist[k.w >> 20], 1u);
  }
  // Only now: blocks of the next kernel that start earlier take issue slots from the histograms (one mask for eight
  // tokens, two calls: 146.4 -> 145.1 us; stages one by one, two layers: 91.8 -> 90.8; the other batch cases equal).
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  sync();
  unsigned prefix, kleft = (unsigned)k2;
  {
    unsigned c[N1] = {};
#pragma unroll
    for (int r = 0; r < NB; ++r) add_counts<N1>(of_rank(hist, r), NT - 1 - tid, c);
    kth_of_counts<NT, N1>(c, kleft, wsum, res);
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
    sync();
    unsigned c[N2] = {};
#pragma unroll
    for (int r = 0; r < NB; ++r) add_counts<N2>(of_rank(h, r), NT - 1 - tid, c);
    kth_of_counts<NT, N2>(c, kleft, wsum, res);
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
  const unsigned wv = lane < NT / 32 ? wsum[lane] : 0u;          // (at most 12288 channels per block: 16 bits each)
  const unsigned ex = __reduce_add_sync(0xffffffffu, lane < warp ? wv : 0u) + inc - cnt;
  unsigned rg = ex & 0xffffu, re = ex >> 16;
  if constexpr (NB > 1) {
    if (tid == NT - 1) total = ex + cnt;
    cl.sync();
    const unsigned tot = lane < rank ? *cl.map_shared_rank(&total, lane) : 0u;
    rg += __reduce_add_sync(0xffffffffu, tot & 0xffffu);
    re += __reduce_add_sync(0xffffffffu, tot >> 16);
    cl.barrier_arrive();                                         // (no block reads another's shared memory after that)
  }
  int* const list = sel_out + (size_t)b * sel_stride;
  const unsigned token_bits = ((1u << tokens) - 1u) << (b * tokens);
  if (FORM == kRepeated && tid == 0) span[0] = rg + min(re, quota);
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
        list[pos] = ch;
        bits |= token_bits << (8 * e);
      }
      rg += gt ? 1u : 0u; re += eq ? 1u : 0u;
    }
    if (cmask && bits) atomicOr(cmask + q0 + i, bits);
  }
  if (FORM == kRepeated) {                                       // the block's part of the list, in whole lines
    if (tid == NT - 1) span[1] = rg + min(re, quota);
    __syncthreads();
    for (unsigned i = span[0] + tid; i < span[1]; i += NT) {
      const int ch = list[i];
      for (int t = 1; t < tokens; ++t) list[(size_t)t * sel_stride + i] = ch;
    }
  }
  if constexpr (NB > 1) cl.barrier_wait();
}

template <int FORM>
__global__ void __launch_bounds__(1024)
channel_topk_kernel(float* __restrict__ scores, float* __restrict__ pacc, int F, int k2, int* __restrict__ sel_out, int sel_stride,
                    int tokens, unsigned* __restrict__ cmask) {
  channel_topk<FORM, 1, 1024>(scores, pacc, F, k2, sel_out, sel_stride, tokens, cmask);
}
template <int FORM>
__global__ void __cluster_dims__(kTkBlocks, 1, 1) __launch_bounds__(512)
channel_topk_cluster_kernel(float* __restrict__ scores, float* __restrict__ pacc, int F, int k2, int* __restrict__ sel_out, int sel_stride,
                            int tokens, unsigned* __restrict__ cmask) {
  channel_topk<FORM, kTkBlocks, 512>(scores, pacc, F, k2, sel_out, sel_stride, tokens, cmask);
}

}  // namespace prox
