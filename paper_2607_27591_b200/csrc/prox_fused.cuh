// One persistent kernel for the whole batch-1 path (Sec. 4.1 Stage 1 + Stage 2):
//
//   A  every block: exact top-k1 of |x| (redundantly; x is a few KB)
//   B  proxy GEMV on the tensor cores (tcgen05, integer MMA, accumulators in
//      tensor memory): a block owns an equal share of the packed proxy's columns
//      over ALL kept rows, so its channels' sums need no exchange with other
//      blocks; the rows' bytes are the A operand as they lie in memory, x enters
//      as signed base-256 digits; the block writes the scores |u~ SiLU(g~)| of
//      its channels and adds them to a global 2048-bin histogram
//   -- every block needs all scores: a bounded wait for a count of finished shares, after which the scores are read and
//      say themselves whether they are there --
//   C  every block (consumer warps only; the producer warps wait for them):
//      the histogram gives the threshold bin b1; channels in bins above b1 are
//      kept whatever the exact threshold is.  The kept list is laid out as
//      [those channels][kept members of b1] and block c owns the c-th share of
//      both parts.  One pass over the upper halves of the scores finds its
//      share of the first part, a warp lists it and the ring starts; half of the consumer warps
//      then settle the exact threshold inside b1 (four more bits from the half scores, whole scores for the members that
//      agree in them too) and append the block's share of the second part, while the other half already consumes rows
//   D  gate/up rows of its channels stream through a shared-memory ring filled
//      by bulk async copies (cp.async.bulk + mbarrier, four issuing warps); a
//      consumer warp takes the next channel nobody has taken:
//      h_j = SiLU(x.g_j) (x.u_j)
//   E  the matching rows of channel-major W_down follow in the same ring; warp
//      groups own whole rows; partial y vectors meet in shared memory and are
//      added to an fp32 accumulator with vector atomics
//   F  the last block to finish (ticket) rounds y once and clears the scratch.
//
// Launch: an ordinary one, one block per SM, with programmatic stream serialization.  No block waits for a block that
// may not be running: the shares of Stage 1 (columns) and of Stage 2 (kept channels) are claimed by tickets, a
// running block claims again until there are none left, and the wait is for finished shares, not blocks.  Where all
// blocks run, as always on a GPU of its own, every block has one share of each.  (With the cooperative attribute
// instead, launches of a stream did not overlap and started in steps of 2.05 us:
// 512 x 1536 20.5 -> 19.6 us per call, 1024 x 3072 layer form 22.4 -> 20.5, 4096 x 12288 38.9 -> 37.7.)
#pragma once

#include "prox_kernels.cuh"
#include "prox_umma.cuh"

namespace prox {

constexpr int kFusedConsumerWarps = 16;
constexpr int kFusedConsumers = kFusedConsumerWarps * 32;       // 512
constexpr int kSettlerWarps = 8;                                 // consumer warps that finish the channel mask
constexpr int kSettlers = kSettlerWarps * 32;
constexpr int kFusedProducers = 4;                               // warps whose lane 0 issues bulk copies
constexpr int kFusedThreads = kFusedConsumers + 32 * kFusedProducers;   // 640
constexpr int kFusedWarps = kFusedThreads / 32;                 // 20
constexpr int kMaxSlots = 32;
constexpr int kEmptyCount = 16;      // arrivals that free a ring slot
constexpr int kChanBatch = 256;      // channels whose h values are held at once
constexpr int kMySelCap = 512;       // channels one block may own
constexpr int kCand2Cap = 256;       // members of the threshold bin that agree with the threshold in their half scores and are ranked (one per settler)
// Proxy ring: a loader warp owns two stages of 32 rows x 128 bytes (4 KB each), for 4-bit codes a buffer of low
// nibbles (4 KB), and two stages of digits of x (512 bytes each).
__host__ __device__ constexpr int proxy_warp_bytes(int bits) { return bits == 4 ? 13312 : 9216; }
constexpr int kMinLoaders = 8;           // loader warps that must fit (at most all 16 consumer warps)
constexpr int kMaxSuper = 16;            // supergroups (4 scale groups) whose accumulators fit the tensor memory
constexpr unsigned kSpinLimit = 1u << 21;

enum FusedMode { kWhole = 0, kScoresOnly, kGivenList };   // whole path; A and B; D to F for the caller's channels

struct FusedParams {
  const int* sel_in; const int* sel_cnt;   // kGivenList: the channels, and how many (NULL: k2)
  const uint8_t* P; const __half* S;
  const uint16_t* wg; const uint16_t* wu; const uint16_t* wdt;
  const uint16_t* x; void* y;
  int D, F, k1, k2, gshift, out_fp32;
  int loaders;        // loader warps of the proxy GEMV whose stages fit
  // a share of Stage 1: plines whole 128-byte lines of the proxy rows, and of the chunks from pleft0 on an equal part:
  // ppart, in the first pmore shares cgran more
  int plines, pleft0, ppart, pmore, cgran;
  float* scores; unsigned* ghist; int* sel_out;
  // What the blocks hand to each other, in two sets that calls take in turn (all ones = not there yet): the upper halves of
  // the scores' bits (THRESH: per chunk of the proxy rows a word of marks, one bit per channel), and all bits.
  uint16_t* xhalf; unsigned* xkeys;   // [2][F] each
  int* idx_out;       // the kept input list as this kernel built it (block 0 writes it; for checking)
  unsigned spin_limit;        // polls after which a device-side wait gives up
  unsigned bar_bias;          // test knob (0 in normal use): the wait for the scores does not end; bits 30 and 31: see prox_debug_set_wait
  int* host_flag;             // mapped host word set to 1 when a wait expires (NULL = none)
  float* yacc; int* status;
  unsigned long long* exits;  // grows by 256 per call, complete when all its blocks have left: the call number
  unsigned* ctr;              // [2][8] counters of a call (calls alternate): see FusedCtr
  int nshare1, nshare;        // shares of Stage 1 and of Stage 2
  int big_bytes;      // bytes of the large shared buffer
  int nslots;         // ring slots of D*2 bytes inside it
  unsigned nslots_rcp;   // floor(2^32 / nslots) + 1: __umulhi(q, it) = q / nslots for q < 2^27 (nslots <= 32)
  unsigned long long* trace;   // optional [grid][32] phase time stamps (ns), NULL = off
  // Layer sub-block form (all NULL / 0 otherwise): the input is bf16(RMSNorm(xres) * norm_w) and the
  // result is xres + y, written as fp32 to xres_out (which may be xres itself).
  const float* xres; const uint16_t* norm_w; float* xres_out; RmsConst rc;
  // Threshold form (THRESH): keep |x_i| >= tau_x and score_j >= tau_s instead of the k1 / k2 largest.
  // tkey_x = smallest 15-bit bf16 magnitude that is >= tau_x, tkey_s = bits of tau_s (scores are >= 0, so
  // their bit patterns order like their values).  Counts go to cnt_x_out / count_out and into counters.
  unsigned tkey_x, tkey_s;
  int* cnt_x_out; int* count_out; unsigned long long* counters;
};

constexpr unsigned kNoKey = 0xffffffffu;      // no score: those have the sign bit clear
constexpr unsigned kBiasKeys = 1u << 30;      // bar_bias: no score is there as a whole
// shares claimed / finished, Stage 1 and Stage 2; kOut1: Stage-1 shares whose scores are on their way
enum FusedCtr { kClaim1 = 0, kDone1, kClaim2, kDone2, kOut1 };

// ---- PTX wrappers -----------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive_n(uint32_t bar, uint32_t n) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(n) : "memory");
}
__device__ __forceinline__ uint32_t mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok;
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ float4 lds128f(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ uint4 ld_relaxed4(const unsigned* p) {
  uint4 v;
  asm volatile("ld.relaxed.gpu.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(unsigned* p, unsigned v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void st_relaxed2(unsigned* p, unsigned a, unsigned b) {
  asm volatile("st.relaxed.gpu.global.v2.u32 [%0], {%1,%2};" ::"l"(p), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ unsigned every_other_bit(unsigned v) {          // bits 0..7 to bits 0, 2, .., 14
  v = (v | (v << 4)) & 0x0f0fu;
  v = (v | (v << 2)) & 0x3333u;
  return (v | (v << 1)) & 0x5555u;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
#define PROX_TRACE_AT(k, who) do { if (TRACE && tid == (who)) p.trace[(size_t)cta * 32 + (k)] = global_ns(); } while (0)
#define PROX_TRACE(k) do { if (TRACE && tid == 0) p.trace[(size_t)cta * 32 + (k)] = global_ns(); } while (0)
__device__ __forceinline__ bool elect_one() {          // the same lane every time for a full warp
  uint32_t pred;
  asm volatile("{\n\t.reg .pred P1;\n\telect.sync _|P1, 0xffffffff;\n\tselp.u32 %0, 1, 0, P1;\n\t}" : "=r"(pred));
  return pred != 0;
}
__device__ __forceinline__ void settler_sync() {      // the lower half of the consumer warps
  asm volatile("bar.sync 3, %0;" ::"n"(kSettlers) : "memory");
}
__device__ __forceinline__ void consumer_sync() {     // the 512 consumer threads only
  asm volatile("bar.sync 1, %0;" ::"n"(kFusedConsumers) : "memory");
}

// Bounded wait on an mbarrier phase.  Gives up (and raises the block's abort
// flag) after kSpinLimit polls; once the flag is up every wait returns at once.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, unsigned limit = kSpinLimit) {
  if (mbar_try_wait(bar, parity)) return true;
  if (*abort_flag) return false;
#pragma unroll 1
  for (unsigned it = 0; it < limit; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if (it > 256) __nanosleep(64);
    if ((it & 255u) == 255u && *abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}

// Wait for use number `use` of a ring slot.  Different warps consume different
// uses of one slot, and a parity wait cannot tell phase u from phase u-2, so a
// warp first waits (bounded) until the consumer of the previous use has seen
// its data complete; from then on the barrier can only be in phase `use`.
__device__ __forceinline__ bool slot_wait(uint32_t bar, volatile unsigned* seen, unsigned use,
                                          volatile int* abort_flag, unsigned limit) {
  if (use > 0 && *seen < use) {
    bool ok = false;
#pragma unroll 1
    for (unsigned it = 0; it < limit; ++it) {
      if (*seen >= use) { ok = true; break; }
      if (it > 256) __nanosleep(32);
      if ((it & 255u) == 255u && *abort_flag) return false;
    }
    if (!ok) { *abort_flag = 1; return false; }
  }
  if (!mbar_wait(bar, use & 1u, abort_flag, limit)) return false;
  *seen = use + 1u;
  return true;
}

// The selection phases run once per call on every block, over code that is cold
// in the instruction caches: their time is set by the number of instructions
// fetched, not executed.  They are therefore written as small loops (one key per
// lane and trip) and the helpers below are shared between the phases.

__device__ __forceinline__ unsigned warp_scan_incl(unsigned v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// k-th largest (k >= 1, counted from the top) among the 32 * BPL bins that end
// below index `top`.  One warp; every lane returns the same bin and the count
// above it.  Lane l owns the l-th slice of BPL bins from the top.
template <int BPL>
__device__ __forceinline__ unsigned kth_in_segment(const unsigned* hist, int top, unsigned k, int lane, unsigned* above) {
  const int base = top - (lane + 1) * BPL;
  unsigned s = 0;
#pragma unroll 1
  for (int j = 0; j < BPL; ++j) s += hist[base + j];
  const unsigned inc = warp_scan_incl(s, lane);
  const unsigned ex = inc - s;
  const unsigned m = __ballot_sync(0xffffffffu, ex < k && k <= inc);
  const int src = m ? (__ffs(m) - 1) : 31;
  unsigned run = __shfl_sync(0xffffffffu, ex, src);
  const int b0 = top - (src + 1) * BPL;                 // all lanes walk the same slice (broadcast reads)
  unsigned bin = (unsigned)b0, ab = run;
#pragma unroll 1
  for (int j = BPL - 1; j >= 0; --j) {
    const unsigned c = hist[b0 + j];
    if (run < k && k <= run + c) { bin = (unsigned)(b0 + j); ab = run; }
    run += c;
  }
  *above = ab;
  return bin;
}

// Same over 512 * BPL bins with the 16 consumer warps (one barrier of theirs inside):
// warps 0..15 total their segment, then every warp locates the segment and
// finishes on its own, so the result is in the registers of every thread.
template <int BPL>
__device__ __forceinline__ unsigned kth_in_block(const unsigned* hist, unsigned k, unsigned* wsum, int lane, int warp,
                                                 unsigned* above) {
  constexpr int NB = 512 * BPL, SEG = 32 * BPL;
  {
    const int base = NB - warp * SEG - (lane + 1) * BPL;
    unsigned s = 0;
#pragma unroll 1
    for (int j = 0; j < BPL; ++j) s += hist[base + j];
    s = __reduce_add_sync(0xffffffffu, s);
    if (lane == 0) wsum[warp] = s;
  }
  consumer_sync();
  const unsigned v = (lane < 16) ? wsum[lane] : 0u;
  const unsigned inc = warp_scan_incl(v, lane);
  const unsigned ex = inc - v;
  const unsigned m = __ballot_sync(0xffffffffu, ex < k && k <= inc);
  const int seg = m ? (__ffs(m) - 1) : 15;
  const unsigned aseg = __shfl_sync(0xffffffffu, ex, seg);
  unsigned ab;
  const unsigned bin = kth_in_segment<BPL>(hist, NB - seg * SEG, k - aseg, lane, &ab);
  *above = aseg + ab;
  return bin;
}

// ---- shared memory map --------------------------------------------------------
struct FusedSmem {
  unsigned hist[2048];
  unsigned hist2[256];
  unsigned wsum[32];
  unsigned res[8];
  unsigned long long mbar_full[kMaxSlots];
  unsigned long long mbar_empty[kMaxSlots];
  int mysel[kMySelCap];
  float hval[kChanBatch];
  unsigned warp_cnt[kFusedWarps][2];
  unsigned cand2_key[kCand2Cap];
  int cand2_idx[kCand2Cap];
  int abort_flag;
  int s_last;
  unsigned call_par;          // parity of the handle's call number: which set of global histogram and counters is this call's
  unsigned vid;               // Stage 1: share of this block (none: >= number of shares)
  int late;                   // the block started after Stage 1 was complete: it has no part in the call
  int again;                  // another Stage-1 share was claimed
  unsigned shr, shr_next;     // Stage 2: share of this block, and the next one
  // warps that have finished their share of soff (here, because the fields behind it have their offsets by it: four bytes
  // further up, 28 layers of 1024 x 3072 took 0.7 % longer)
  unsigned soff_cnt;
  unsigned ncand2;
  unsigned prod_seq;       // rows the producers have armed so far (for the give-up path)
  unsigned next_c;         // next channel of the batch to take in the gate/up phase
  int n_mine;              // channels of this block (for the producer warps)
  int nready;              // entries of mysel that are final (the definite share first, all of them later)
  int keys_done;           // the consumer warps no longer read the half scores near the end of the big buffer
  int c_done;              // ... nor the list of the threshold bin's members
  int keys_s0, keys_s1;    // ring slots [s0, s1) that overlap them
  int list_s0, list_s1;    // ... and the list
  unsigned slot_use[kMaxSlots];   // uses of each ring slot whose data has been seen complete
  unsigned long long pempty[kFusedConsumerWarps];   // proxy ring: the MMAs of a warp's block are complete
  unsigned long long acc_bar;            // all MMAs of a tile are complete (one arrival per loader warp)
  uint32_t tmem_base;
  float soff[4 * kMaxSuper];             // per scale group: code offset (8 or 128) * sum of the kept x, as integers
  int gstart[4 * kMaxSuper + 2];         // first kept row of every scale group (and k1)
  unsigned wmax[32];
  float nsum[kFusedWarps][2];     // RMSNorm: the warps' sums of squares (hi, lo)
  float ninv[2];                  // ... and 1 / sqrt(mean + eps) (hi, lo)
  unsigned poll[2][kFusedConsumerWarps];   // the warps' counts of scores in the histogram; and whether scores are missing
};

// k-th largest (k >= 1) over a histogram held in registers: thread t < 512 has the counts of N bins in descending order,
// the first of them bin `top`; the threads' runs follow each other downwards (threads from 512 on: zeros).  One scan and two
// barriers where reading the bins segment by segment took three passes over shared memory (0.8 -> 0.4 us for 1024 bins).
// res[0], res[1] = bin, elements above it.
template <int N>
__device__ __forceinline__ void find_kth(FusedSmem& sm, const unsigned (&c)[N], int top, unsigned k, int lane, int warp) {
  unsigned s = 0;
#pragma unroll
  for (int j = 0; j < N; ++j) s += c[j];
  const unsigned inc = warp_scan_incl(s, lane);
  if (lane == 31) sm.wsum[warp] = inc;
  __syncthreads();
  unsigned run = __reduce_add_sync(0xffffffffu, (lane < warp) ? sm.wsum[lane] : 0u) + inc - s;
  if (run < k && k <= run + s) {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      if (run < k && k <= run + c[j]) { sm.res[0] = (unsigned)(top - j); sm.res[1] = run; }
      run += c[j];
    }
  }
  __syncthreads();
}

// All bits of the scores of eight channels: a bounded wait, which ends once the abort flag is up.
__device__ __forceinline__ void full_keys(const unsigned* xkeys, const int (&i)[8], unsigned (&k)[8], unsigned spin, unsigned bias, volatile int* abortp) {
#pragma unroll 1
  for (unsigned it = 0;; ++it) {
    unsigned any = 0;
#pragma unroll
    for (int u = 0; u < 8; ++u) asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(k[u]) : "l"(xkeys + i[u]) : "memory");
#pragma unroll
    for (int u = 0; u < 8; ++u) any |= k[u];
    if (!(any >> 31) && !(bias & kBiasKeys)) break;
    if (it >= spin || *abortp) { *abortp = 1; break; }
  }
}
__device__ __forceinline__ unsigned lds32(uint32_t a) {
  unsigned v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}

// Channel mask where shared memory has no room for the half scores and the list of the threshold bin b1's members (a very large
// d_model and d_ff, or a huge bin such as an all-zero input gives): the consumer warps settle the threshold by two radix steps of
// 10 bits over all scores, and the block gets its share of the plain ascending list of k2 channels.  Returns the share's length.
// (A function of its own, as the next one: inside the kernel, the two cost calls that never get here 1 % of 8192 x 28672.)
__device__ __noinline__ int settle_over_all_channels(const unsigned* xkeys, int F, unsigned k2, unsigned shr, unsigned nsh, unsigned b1, unsigned kk,
                                                     int* sel_out, unsigned spin, unsigned bias) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  FusedSmem& sm = *reinterpret_cast<FusedSmem*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int R0 = (int)((k2 * shr) / nsh), R1 = (int)((k2 * (shr + 1u)) / nsh);
  const int per = ((F + 32 * kFusedConsumerWarps - 1) / (32 * kFusedConsumerWarps)) * 32;        // channels per warp run
  const int i0 = min(F, warp * per), i1 = min(F, i0 + per);
  const int n_mine = min(R1 - R0, kMySelCap);
  int ch[8];
  unsigned key[8];
  unsigned prefix = b1, kleft = kk;
#pragma unroll 1
  for (int sh = 10; sh >= 0; sh -= 10) {
    consumer_sync();
#pragma unroll 1
    for (int i = tid; i < 1024; i += kFusedConsumers) sm.hist[i] = 0;
    consumer_sync();
#pragma unroll 1
    for (int ib = tid; ib < F; ib += 8 * kFusedConsumers) {
#pragma unroll
      for (int u = 0; u < 8; ++u) ch[u] = min(ib + u * kFusedConsumers, F - 1);
      full_keys(xkeys, ch, key, spin, bias, &sm.abort_flag);
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (ib + u * kFusedConsumers < F && (key[u] >> (sh + 10)) == prefix) atomicAdd(&sm.hist[(key[u] >> sh) & 1023u], 1u);
    }
    consumer_sync();
    unsigned ab;
    const unsigned bb = kth_in_block<2>(sm.hist, kleft, sm.wsum, lane, warp, &ab);
    prefix = (prefix << 10) | bb;
    kleft -= ab;
  }
  const unsigned T = prefix, quota = kleft;
  consumer_sync();
  {
    unsigned cg = 0, ce = 0;                 // separate words: the ties alone may be 65536
#pragma unroll 1
    for (int ib = i0 + lane; ib < i1; ib += 8 * 32) {
#pragma unroll
      for (int u = 0; u < 8; ++u) ch[u] = min(ib + u * 32, F - 1);
      full_keys(xkeys, ch, key, spin, bias, &sm.abort_flag);
#pragma unroll
      for (int u = 0; u < 8; ++u) { cg += (ib + u * 32 < i1 && key[u] > T) ? 1u : 0u; ce += (ib + u * 32 < i1 && key[u] == T) ? 1u : 0u; }
    }
    cg = __reduce_add_sync(0xffffffffu, cg);
    ce = __reduce_add_sync(0xffffffffu, ce);
    if (lane == 0) { sm.wsum[warp] = cg; sm.warp_cnt[warp][1] = ce; }
  }
  consumer_sync();
  unsigned bg = __reduce_add_sync(0xffffffffu, (lane < warp) ? sm.wsum[lane] : 0u);
  unsigned be = __reduce_add_sync(0xffffffffu, (lane < warp) ? sm.warp_cnt[lane][1] : 0u);
  const int first_pos = (int)(bg + min(be, quota));
  const int end = (int)(bg + sm.wsum[warp] + min(be + sm.warp_cnt[warp][1], quota));
  if (first_pos < R1 && end > R0) {
#pragma unroll 1
    for (int ib = i0; ib < i1; ib += 8 * 32) {
#pragma unroll
      for (int u = 0; u < 8; ++u) ch[u] = min(ib + u * 32 + lane, F - 1);
      full_keys(xkeys, ch, key, spin, bias, &sm.abort_flag);
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int i = ib + u * 32 + lane;
        const bool gt = i < i1 && key[u] > T, eq = i < i1 && key[u] == T;
        const unsigned mg = __ballot_sync(0xffffffffu, gt), me = __ballot_sync(0xffffffffu, eq);
        const unsigned myre = be + (unsigned)__popc(me & lt_mask);
        const int pos = (int)(bg + (unsigned)__popc(mg & lt_mask) + min(myre, quota));
        if ((gt || (eq && myre < quota)) && pos >= R0 && pos < R0 + n_mine) {
          sm.mysel[pos - R0] = i;
          if (sel_out) sel_out[pos] = i;
        }
        bg += (unsigned)__popc(mg); be += (unsigned)__popc(me);
      }
    }
  }
  return n_mine;
}

// Members of the threshold bin (list entries: four bits of the half score above the channel) of which more than kCand2Cap agree with the
// threshold in their half scores, i.e. have `sub` there: the kk2 of them that come first by (score descending, channel
// ascending) follow at place `above` of the members that are kept, of which the block has Rc0 .. Rc1 - 1.  Radix steps of 8 bits
// over the lower halves and the inverted channels, which a thread puts in the place of its entries first.  By the settler warps.
// An input of zeros at 4096 x 12288: 52 us per call; 152 with the lower halves fetched one at a time in every step, 65 when
// all scores were whole ones in shared memory.
__device__ __noinline__ void settle_equal_halves(uint32_t list_u32, unsigned nb1, unsigned sub, unsigned kk2, const unsigned* xkeys, int above, int Rc0,
                                                 int Rc1, int ndm, int* sel_out, unsigned spin, unsigned bias) {
  extern __shared__ __align__(128) uint8_t smem_raw[];
  FusedSmem& sm = *reinterpret_cast<FusedSmem*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  unsigned mine = tid, low = ~0u, high = 0;       // end of the thread's values; lowest and highest lower half
  settler_sync();                                 // the list is read by other threads than write it here
#pragma unroll 1
  for (unsigned c = tid; c < nb1; c += 8 * kSettlers) {
    unsigned e[8], key[8];
    int ch[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      e[u] = c + u * kSettlers < nb1 ? lds32(list_u32 + (c + u * kSettlers) * 4u) : ~0u;
      ch[u] = (e[u] >> 16) == sub ? (int)(e[u] & 0xffffu) : 0;
    }
    full_keys(xkeys, ch, key, spin, bias, &sm.abort_flag);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      if ((e[u] >> 16) == sub) {
        asm volatile("st.shared.u32 [%0], %1;" ::"r"(list_u32 + mine * 4u), "r"((key[u] << 16) | (0xffffu ^ (unsigned)ch[u])) : "memory");
        mine += kSettlers;
        low = min(low, key[u] & 0xffffu); high = max(high, key[u] & 0xffffu);
      }
    }
  }
  // (all the same score, as where there are many: two steps less)
  low = __reduce_min_sync(0xffffffffu, low); high = __reduce_max_sync(0xffffffffu, high);
  if (lane == 0) { sm.cand2_key[warp] = low; sm.cand2_key[kSettlerWarps + warp] = high; }
  settler_sync();
  low = __reduce_min_sync(0xffffffffu, lane < kSettlerWarps ? sm.cand2_key[lane] : ~0u);
  high = __reduce_max_sync(0xffffffffu, lane < kSettlerWarps ? sm.cand2_key[kSettlerWarps + lane] : 0u);
  // (four entries at a time: one would wait for its load and its bin before the next)
  unsigned prefix = low == high ? low : 0u, kleft = kk2;
#pragma unroll 1
  for (int sh = low == high ? 8 : 24; sh >= 0; sh -= 8) {
    settler_sync();                               // everyone is done with the previous histogram
    sm.hist2[tid] = 0;
    settler_sync();
#pragma unroll 1
    for (unsigned c = tid; c < mine; c += 4 * kSettlers) {
      unsigned v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = c + u * kSettlers < mine ? lds32(list_u32 + (c + u * kSettlers) * 4u) : 0u;
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (c + u * kSettlers < mine && (unsigned)((unsigned long long)v[u] >> (sh + 8)) == prefix) atomicAdd(&sm.hist2[(v[u] >> sh) & 255u], 1u);
    }
    settler_sync();
    unsigned ab;
    const unsigned bb = kth_in_segment<8>(sm.hist2, 256, kleft, lane, &ab);
    prefix = (prefix << 8) | bb;
    kleft -= ab;
  }
  unsigned wk = 0;
#pragma unroll 4
  for (unsigned c = tid; c < mine; c += kSettlers) wk += lds32(list_u32 + c * 4u) >= prefix ? 1u : 0u;
  const unsigned inck = warp_scan_incl(wk, lane);
  if (lane == 31) sm.warp_cnt[warp][1] = inck;
  settler_sync();
  int at = above + (int)(__reduce_add_sync(0xffffffffu, lane < warp ? sm.warp_cnt[lane][1] : 0u) + inck - wk);
  if (at < Rc1 && at + (int)wk > Rc0) {
#pragma unroll 1
    for (unsigned c = tid; c < mine; c += kSettlers) {
      const unsigned v = lds32(list_u32 + c * 4u);
      if (v < prefix) continue;
      if (at >= Rc0 && at < Rc1) {
        sm.mysel[ndm + at - Rc0] = (int)(0xffffu ^ (v & 0xffffu));
        if (sel_out) sel_out[at] = (int)(0xffffu ^ (v & 0xffffu));
      }
      ++at;
    }
  }
}

// NG = warp groups of the down projection (4: d_model <= 4096, 2: <= 8192, 1: <= 16384)
// NORM = layer sub-block form (RMSNorm in the prologue, residual add at the end); THRESH = threshold
// form of the two masks (Sec. 4.1 indicators with calibrated thresholds; no k-th element search at all).
// Instantiations of their own, so that the plain call carries none of their code or registers.
// TRACE: with time stamps (the tests for them cost the plain kernel up to 4 %: code that runs once is fetched cold).
// MODE: instantiations of their own for the two stages called alone (as a run-time switch it cost the whole path 1 %).
template <int BITS, int NG, bool NORM = false, bool THRESH = false, int MODE = kWhole, bool TRACE = false>
__global__ void __launch_bounds__(kFusedThreads, 1) prox_fused_kernel(const FusedParams p) {
  constexpr int CH = ProxyFmt<BITS>::CH;
  constexpr int NT = kFusedThreads;
  // Only the top-k form of the whole path starts its channel mask from the score histogram; filled in the threshold form as
  // well, it cost that 0.4 us in front of the exchange (4096 x 12288 layer form: 34.5 -> 33.9 us per call).
  constexpr bool HIST = MODE == kWhole && !THRESH;
  extern __shared__ __align__(128) uint8_t smem_raw[];
  FusedSmem& sm = *reinterpret_cast<FusedSmem*>(smem_raw);
  const int D = p.D, F = p.F, k2 = p.k2;
  int k1 = p.k1;                         // THRESH: becomes the number of kept inputs after phase A
  uint16_t* xs = reinterpret_cast<uint16_t*>(smem_raw + ((sizeof(FusedSmem) + 127) & ~size_t(127)));
  uint16_t* idx16 = xs + D;
  // x as fp32, written after phase B: until then its place belongs to the proxy ring, as the big buffer behind it does
  float* xf = reinterpret_cast<float*>(idx16 + D);
  uint8_t* big = reinterpret_cast<uint8_t*>(xf + D);           // 128-byte aligned: D % 128 == 0
  const uint32_t big_u32 = smem_u32(big);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x, cta = blockIdx.x;
  volatile int* abortp = &sm.abort_flag;
  const unsigned lt_mask = (1u << lane) - 1u;
  const unsigned spin = p.spin_limit;

  auto prefetch_row = [&](int i) {              // row i of the packed proxy to L2, by a warp
    const int prow = F / CH * 16;
    const uint8_t* src = p.P + (size_t)i * (size_t)prow;
#pragma unroll 1
    for (int o = lane * 32; o < prow; o += 1024) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + o) : "memory");
  };
  // ------------------------------------------------------------------ set-up
  PROX_TRACE(0);
  if (tid < kMaxSlots) {
    mbar_init(smem_u32(&sm.mbar_full[tid]), 1);
    mbar_init(smem_u32(&sm.mbar_empty[tid]), kEmptyCount);
    fence_mbar_init();
  }
  if (warp == 0) tmem_alloc_all(smem_u32(&sm.tmem_base));      // all 512 columns: one block per SM
  if (tid < kFusedConsumerWarps) {
    mbar_init(smem_u32(&sm.pempty[tid]), 1);
    if (tid == 0) mbar_init(smem_u32(&sm.acc_bar), (uint32_t)p.loaders);
    fence_mbar_init();
  }
  if (tid == 0) sm.soff_cnt = 0;
  if (tid == 0) { sm.abort_flag = 0; sm.ncand2 = 0; sm.prod_seq = 0; sm.next_c = 0; sm.again = 0; }
  if (tid < kMaxSlots) sm.slot_use[tid] = 0;
  // the launch may have been set up while the previous kernel of the stream was still draining: nothing of
  // global memory is touched before that kernel has completed
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // Two global score histograms take turns: this call adds to one and clears the other for the next call (it was
  // last used by the previous call, which has completed), so nothing is left to clean up when the call ends.
  // The call number is exits / 256: blocks of this call that have left add less than 256 until the last one does.
  if (tid == NT - 1) {                          // a thread with no share of the input load below
    unsigned long long ex;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(ex) : "l"(p.exits) : "memory");
    sm.call_par = (unsigned)(ex >> 8) & 1u;
  }
  if (NORM) {
    // FFN input = bf16(RMSNorm(residual stream) * norm weight), the correctly rounded value (the masks
    // depend on it).  Every block does all of it; x and w pass through shared memory once.
    float hi = 0.f, lo = 0.f;
    {
      // both loads of a round are issued before the first use (a load per dependent iteration would put
      // the latency of global memory on every one of them)
      const float4* x4 = reinterpret_cast<const float4*>(p.xres);
      const uint2* w2 = reinterpret_cast<const uint2*>(p.norm_w);
      const int n4 = D / 4;
#pragma unroll 1
      for (int i0 = tid; i0 < n4; i0 += 2 * NT) {
        const int i1 = i0 + NT;
        const bool two = i1 < n4;
        const float4 a = __ldcg(x4 + i0);
        const uint2 wa = __ldg(w2 + i0);
        const float4 b = two ? __ldcg(x4 + i1) : make_float4(0.f, 0.f, 0.f, 0.f);
        const uint2 wb = two ? __ldg(w2 + i1) : make_uint2(0u, 0u);
        reinterpret_cast<float4*>(xf)[i0] = a;
        reinterpret_cast<uint2*>(idx16)[i0] = wa;
        f2_add_square(hi, lo, a.x); f2_add_square(hi, lo, a.y); f2_add_square(hi, lo, a.z); f2_add_square(hi, lo, a.w);
        if (two) {
          reinterpret_cast<float4*>(xf)[i1] = b;
          reinterpret_cast<uint2*>(idx16)[i1] = wb;
          f2_add_square(hi, lo, b.x); f2_add_square(hi, lo, b.y); f2_add_square(hi, lo, b.z); f2_add_square(hi, lo, b.w);
        }
      }
    }
#pragma unroll 1
    for (int i = tid; i < 1024 + 32; i += NT) { if (i < 1024) sm.hist[i] = 0; else sm.hist2[i - 1024] = 0; }
    f2_warp_sum(hi, lo);
    if (lane == 0) { sm.nsum[warp][0] = hi; sm.nsum[warp][1] = lo; }
    __syncthreads();
    if (warp == 0) {
      hi = lane < kFusedWarps ? sm.nsum[lane][0] : 0.f;
      lo = lane < kFusedWarps ? sm.nsum[lane][1] : 0.f;
      f2_warp_sum(hi, lo);
      if (lane == 0) rms_inverse(hi, lo, p.rc, sm.ninv[0], sm.ninv[1]);
    }
    __syncthreads();
    const float ih = sm.ninv[0], il = sm.ninv[1];
#pragma unroll 1
    for (int i = tid; i < D; i += NT) {
      const uint16_t b = rms_scale_to_bf16(xf[i], __uint_as_float((uint32_t)idx16[i] << 16), ih, il);
      xs[i] = b;
    }
  } else {
    const uint4* xg = reinterpret_cast<const uint4*>(p.x);
#pragma unroll 1
    for (int i = tid; i < D / 8; i += NT) reinterpret_cast<uint4*>(xs)[i] = __ldg(xg + i);
#pragma unroll 1
    for (int i = tid; i < 1024 + 32; i += NT) { if (i < 1024) sm.hist[i] = 0; else sm.hist2[i - 1024] = 0; }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  unsigned* const ghist = p.ghist + 2048u * sm.call_par;
  unsigned* const ctr = p.ctr + 8u * sm.call_par;
  unsigned* const xkeys = p.xkeys + (size_t)F * sm.call_par;
  uint16_t* const xhalf = p.xhalf + (size_t)F * sm.call_par;
  // Stage-1 share of this block; the answers are first looked at after phase A.  A block that gets none and finds
  // Stage 1 complete has started late: it leaves (what it read may be a residual stream that is being added to).
  unsigned claim1 = 0, done1 = 0;
  if (tid == NT - 1 && MODE != kGivenList) {
    asm volatile("atom.relaxed.gpu.global.add.u32 %0, [%1], 1;" : "=r"(claim1) : "l"(ctr + kClaim1) : "memory");
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(done1) : "l"(ctr + kDone1) : "memory");
  }
  {
    unsigned* const other = p.ghist + 2048u * (sm.call_par ^ 1u);
    const int per = (2048 + G - 1) / G;
#pragma unroll 1
    for (int i = cta * per + tid; i < min(2048, (cta + 1) * per); i += NT) other[i] = 0u;
    if (cta == 0 && tid < 8) p.ctr[8u * (sm.call_par ^ 1u) + tid] = 0u;
    unsigned* const okeys = p.xkeys + (size_t)F * (sm.call_par ^ 1u);
    uint16_t* const ohalf = p.xhalf + (size_t)F * (sm.call_par ^ 1u);
    const int perk = (F + G - 1) / G;
#pragma unroll 1
    for (int i = cta * perk + tid; i < min(F, (cta + 1) * perk); i += NT) { okeys[i] = kNoKey; ohalf[i] = 0xffffu; }
  }
  if (warp < 4 && MODE != kGivenList) {
    // the accumulators of the proxy GEMV start at zero: 16 columns per supergroup, two sets 256 columns apart
    const int ngz = (p.gshift >= 31) ? 1 : (D >> p.gshift);
    const uint32_t tz = sm.tmem_base + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
    for (int c = 0; c < 16 * ((ngz + 3) >> 2); c += 16) { tmem_st16_zero(tz + (uint32_t)c); tmem_st16_zero(tz + 256u + (uint32_t)c); }
    tmem_st_wait();
    tc_fence_before();
  }
  PROX_TRACE(1);

  // every block counts its leaving
  auto leave = [&]() {
    if (tid == 0) atomicAdd(p.exits, cta == 0 ? 257ull - (unsigned long long)G : 1ull);
  };
  auto widen_x = [&](int t0) {                  // x as fp32 for phase D, by the threads from t0 on
#pragma unroll 1
    for (int i = tid - t0; i < D / 8; i += NT - t0) {
      const uint4 v = reinterpret_cast<const uint4*>(xs)[i];
      reinterpret_cast<float4*>(xf)[2 * i] = make_float4(bf16_lo(v.x), bf16_hi(v.x), bf16_lo(v.y), bf16_hi(v.y));
      reinterpret_cast<float4*>(xf)[2 * i + 1] = make_float4(bf16_lo(v.z), bf16_hi(v.z), bf16_lo(v.w), bf16_hi(v.w));
    }
  };
  int ebase = 1;
  if (MODE == kGivenList) {
    unsigned share2 = 0;
    if (tid == 0) asm volatile("atom.relaxed.gpu.global.add.u32 %0, [%1], 1;" : "=r"(share2) : "l"(ctr + kClaim2) : "memory");
    widen_x(0);
    if (tid == 0) sm.shr = share2;
    __syncthreads();
  } else {
  // ------------------------------------------------- A: input mask (top-k1 of |x|)
  const bool per_row_a = p.gshift >= 31;
  {
    const uint32_t* xs32 = reinterpret_cast<const uint32_t*>(xs);
    const bool all = THRESH ? (p.tkey_x == 0u) : (k1 >= D);
    unsigned T = 0, quota = 0;
    if (THRESH) {
      T = p.tkey_x - 1u;                 // kept: key > T, i.e. |x| >= tau_x; no ties to ration
    } else if (!all) {
      // level 1: the top 10 of the 15 key bits; level 2: the other 5
#pragma unroll 1
      for (int i = tid; i < D / 2; i += NT) {
        const uint32_t w = xs32[i];
        atomicAdd(&sm.hist[(w >> 5) & 0x3ffu], 1u);
        atomicAdd(&sm.hist[(w >> 21) & 0x3ffu], 1u);
      }
      __syncthreads();
      PROX_TRACE(10);
      unsigned hb[2] = {0u, 0u};
      if (tid < 512) { const uint2 v = reinterpret_cast<const uint2*>(sm.hist)[511 - tid]; hb[0] = v.y; hb[1] = v.x; }
      find_kth<2>(sm, hb, 1023 - 2 * tid, (unsigned)k1, lane, warp);
      const unsigned bin1 = sm.res[0], above1 = sm.res[1];
      PROX_TRACE(11);
      if (warp < kFusedConsumerWarps) {
#pragma unroll 1
        for (int i = tid; i < D / 2; i += kFusedConsumers) {
          const uint32_t w = xs32[i];
          const unsigned ka = w & 0x7fffu, kb = (w >> 16) & 0x7fffu;
          if ((ka >> 5) == bin1) atomicAdd(&sm.hist2[ka & 31u], 1u);
          if ((kb >> 5) == bin1) atomicAdd(&sm.hist2[kb & 31u], 1u);
        }
        consumer_sync();
        PROX_TRACE(12);
        // the exact threshold among the bin's 32 values (every warp on its own)
        const unsigned c = sm.hist2[31 - lane], inc = warp_scan_incl(c, lane), need = (unsigned)k1 - above1;
        const int src = __ffs((int)__ballot_sync(0xffffffffu, inc >= need)) - 1;
        T = (bin1 << 5) | (unsigned)(31 - src);
        quota = need - __shfl_sync(0xffffffffu, inc - c, src);      // ties at T to accept, lowest index first
        PROX_TRACE(13);
      }
    }
    // Ordered compaction: a consumer thread owns a run of 8-input groups, counts its kept
    // inputs and its ties (packed in one word), and places them behind those of the threads
    // in front (one warp scan plus the totals of the warps in front).
    if (warp < kFusedConsumerWarps) {
      const int ngrp = D / 8, gpt = (ngrp + kFusedConsumers - 1) / kFusedConsumers;
      const int g0 = min(ngrp, tid * gpt), g1 = min(ngrp, g0 + gpt);
      unsigned cnt = 0, mk = 0;
#pragma unroll 1
      for (int g = g0; g < g1; ++g) {
        const uint4 kv = *reinterpret_cast<const uint4*>(xs + g * 8);
        const uint32_t w4[4] = {kv.x, kv.y, kv.z, kv.w};
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const unsigned key = (w4[e >> 1] >> ((e & 1) * 16)) & 0x7fffu;
          cnt += (all || key > T) ? 1u : 0u;
          if (!THRESH) cnt += (!all && key == T) ? 0x10000u : 0u;
          mk = max(mk, key);
        }
      }
      const unsigned inc = warp_scan_incl(cnt, lane);
      mk = __reduce_max_sync(0xffffffffu, mk);
      if (lane == 31) { sm.wsum[warp] = inc; sm.wmax[warp] = mk; }
      consumer_sync();
      PROX_TRACE(14);
      const unsigned before = __reduce_add_sync(0xffffffffu, (lane < warp) ? sm.wsum[lane] : 0u) + inc - cnt;
      unsigned re = before >> 16, at = (before & 0xffffu) + min(re, quota);
      // (also, for the proxy GEMV: where every scale group starts in the list)
      const int gmask = per_row_a ? 0x7fffffff : ((1 << p.gshift) - 1);
#pragma unroll 1
      for (int g = g0; g < g1; ++g) {
        const uint4 kv = *reinterpret_cast<const uint4*>(xs + g * 8);
        const uint32_t w4[4] = {kv.x, kv.y, kv.z, kv.w};
        if (((g * 8) & gmask) == 0) sm.gstart[per_row_a ? 0 : ((g * 8) >> p.gshift)] = (int)at;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const unsigned key = (w4[e >> 1] >> ((e & 1) * 16)) & 0x7fffu;
          bool keep = all || key > T;
          if (!THRESH && !all && key == T) { keep = re < quota; ++re; }
          if (keep) idx16[at] = (uint16_t)(g * 8 + e);
          at += keep ? 1u : 0u;
        }
      }
      if (THRESH) k1 = (int)__reduce_add_sync(0xffffffffu, (lane < kFusedConsumerWarps) ? (sm.wsum[lane] & 0xffffu) : 0u);
      if (tid == 0) sm.gstart[per_row_a ? 1 : (D >> p.gshift)] = k1;
    }
    if (tid == NT - 1) { sm.vid = claim1; sm.late = done1 >= (unsigned)p.nshare1 && claim1 >= (unsigned)p.nshare1; }
    __syncthreads();
    if (THRESH && warp >= kFusedConsumerWarps) k1 = (int)__reduce_add_sync(0xffffffffu, (lane < kFusedConsumerWarps) ? (sm.wsum[lane] & 0xffffu) : 0u);
    ebase = max(max((int)(__reduce_max_sync(0xffffffffu, (lane < kFusedConsumerWarps) ? sm.wmax[lane] : 0u) >> 7), 1) - 22, 1);
  }
  if (sm.late) {
    if (warp == 0) tmem_free_all(sm.tmem_base);
    leave();
    return;
  }
  if (sm.vid == 0) {
    if (p.idx_out) {
#pragma unroll 1
      for (int i = tid; i < k1; i += NT) p.idx_out[i] = (int)idx16[i];
    }
    if (THRESH && tid == 0) {
      if (p.cnt_x_out) p.cnt_x_out[0] = k1;
      if (p.counters) { atomicAdd(p.counters, 1ull); atomicAdd(p.counters + 1, (unsigned long long)k1); }
    }
  }
  }
  PROX_TRACE(2);
  unsigned uses = 0, acc_n = 0;                 // blocks of rows this warp has handed to the tensor core; tiles read back
  unsigned base_seq = 0;                        // ring rows consumed so far
  unsigned pseq = 0, puse = 0;                  // producers: rows armed or passed over, uses of the ring, ...
  int pslot = 0;                                // ... next slot
  // One trip per share: of Stage 1 (B) and then of Stage 2 (C to F).  Where all blocks run there is one trip; further
  // Stage-1 shares, of blocks that are not running, come before the channel mask, further Stage-2 shares at the end.
  bool with_b = MODE != kGivenList;
  unsigned vid = (unsigned)p.nshare1;           // share of Stage 1 (none: the number of shares)
#pragma unroll 1
  for (bool first = true;; first = false) {
  if (with_b) {
  // --------------------------------------- B: proxy GEMV (tensor cores), scores, score histogram
  // Per scale group g:  sum_k x_k q_kj = 2^(ebase-134) * sum_k X_k (byte_kj - offset), X_k the integer
  // form of x_k (x_digits).  A block owns a share of the packed rows' 16-byte column chunks over all kept rows: whole
  // 128-byte lines, and half a line or a line of what is left over; a tile is a line or half of one.  The kept
  // rows are cut into blocks of at most 32 rows that stay inside one supergroup (4 scale groups); block b
  // accumulates into 16 tensor-memory columns of its supergroup: column 4 * (g % 4) + d holds digit d of
  // group g.  The loader warps bring the rows in with 16-byte asynchronous copies, a block ahead (what bounds this is
  // the bytes in flight: 64 KB per SM give 3.5 TB/s, 128 KB 5.2), add
  // the bytes with the high nibble masked off and the digits of x, and
  // issue the block's MMAs; after the last one the 16 warps read the accumulators, apply the
  // groups' scales and form the scores.
  // Measured (this phase, one call): 4096 x 14336 8-bit, all rows: 30 us, the lines of the first pass at 6.7 TB/s, the half
  // lines of the second at 3.5 (42.9 at first; 38 with shares of six 32-byte sectors, cut without regard to the lines: a
  // segment over two lines costs two requests, and 155 MB of whole lines took less time than 116 MB of those shares);
  // 8192 x 28672 4-bit, 2458 rows: 24 us; 4096 x 12288 4-bit, 1229 rows: 8 us (the first rows arrive 3 us after phase A,
  // the last 2.5 us later).
    constexpr bool LO = (BITS == 4);
    const int nchunks = F / CH;
    const int row_bytes = nchunks * 16;
    const unsigned n1 = (unsigned)p.nshare1;
    vid = sm.vid;
    const int lk0 = p.pleft0 + (int)vid * p.ppart + min((int)vid, p.pmore) * p.cgran;       // this block's part of the rest
    const int lk1 = min(nchunks, lk0 + p.ppart + ((int)vid < p.pmore ? p.cgran : 0));
    const int ntl = vid >= n1 ? 0 : p.plines + (lk1 > lk0 ? ((lk1 + 7) >> 3) - (lk0 >> 3) : 0);
    const bool per_row = p.gshift >= 31;
    const int ng = per_row ? 1 : (D >> p.gshift);
    const int nsuper = (ng + 3) >> 2;
    const uint32_t tbase = sm.tmem_base;
    if (!first) {                              // one more share: the accumulators go back to zero
      tc_fence_after();
      if (warp < 4) {
        const uint32_t tz = tbase + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
        for (int c = 0; c < 16 * nsuper; c += 16) { tmem_st16_zero(tz + (uint32_t)c); tmem_st16_zero(tz + 256u + (uint32_t)c); }
        tmem_st_wait();
        tc_fence_before();
      }
      __syncthreads();
      tc_fence_after();
    }
    const uint32_t ring = (smem_u32(xf) + 1023u) & ~1023u;
    const int NL = p.loaders;
    // partial sums of warps 4..15, [3][128][2], for tiles in turn: behind the ring, and over mysel and hval (not used yet)
    float* const red0 = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(xf) + (ring - smem_u32(xf)) + (uint32_t)(NL * proxy_warp_bytes(BITS)));
    float* const red1 = reinterpret_cast<float*>(sm.mysel);
    static_assert(offsetof(FusedSmem, hval) == offsetof(FusedSmem, mysel) + sizeof(int) * kMySelCap && kMySelCap * 4 + kChanBatch * 4 >= 3072, "");
    PROX_TRACE(29);
    if (warp < kFusedConsumerWarps) {
      // a warp owns its stages of the ring: it fills them and issues their MMAs itself (the tensor core
      // takes accumulating MMAs from several threads into the same columns; integer sums do not depend on the order)
      const uint32_t stg = ring + (uint32_t)warp * (uint32_t)proxy_warp_bytes(BITS);
      const uint32_t dig = stg + (LO ? 12288u : 8192u);
      const uint64_t adesc = umma_smem_desc(stg, 4096u, 1024u, 2u);                  // second stage: 4096 bytes on
      const uint64_t ldesc = umma_smem_desc(stg + 8192u, 4096u, 1024u, 2u);
      const uint64_t bdesc = umma_smem_desc(dig, 128u, 512u, 0u);                    // second stage: 512 bytes on
      constexpr uint32_t idesc = umma_idesc_u8s8(128, 16);
      const uint32_t my_empty = smem_u32(&sm.pempty[warp]);
      const int q4 = warp & 3, part = warp >> 2;
      const int col = q4 * 32 + lane;                          // byte column of the tile = data path lane
      // blocks of 32 rows: lane l knows supergroup l's first row, its end and the number of the first block behind it
      const int sg_r0 = sm.gstart[min(4 * lane, ng)], sg_r1 = sm.gstart[min(4 * lane + 4, ng)];
      const unsigned sg_nb = lane < nsuper ? (unsigned)((sg_r1 - sg_r0 + 31) >> 5) : 0u;
      const int sg_end = nsuper > 1 ? (int)warp_scan_incl(sg_nb, lane) : __shfl_sync(0xffffffffu, (int)sg_nb, 0);
      const int nblk = __shfl_sync(0xffffffffu, sg_end, 31);
#pragma unroll 1
      for (int tl = 0; tl < ntl; ++tl) {
        const int ln = (tl < p.plines ? (int)vid * p.plines : (lk0 >> 3) - p.plines) + tl;    // the tile's line
        const int tc0 = tl < p.plines ? ln * 8 : max(lk0, ln * 8);                            // and its chunks
        const int w = (tl < p.plines ? ln * 8 + 8 : min(lk1, ln * 8 + 8)) - tc0;
        // (8 or 4 of them)  a copy instruction covers 32 >> sc rows of 1 << sc chunks
        const int sc = w > 4 ? 3 : 2, rpi = 32 >> sc;
        const int kq = lane >> sc, c = lane & ((1 << sc) - 1);
        const uint8_t* tp = p.P + (size_t)tc0 * 16 + (size_t)c * 16;
        // copy instruction j takes the rows j * rpi + kq: where they go in a stage, for even and odd j (the chunk's place is xor-ed
        // with the row), a step of j by two further on
        const uint32_t sa0 = stg + (uint32_t)(kq * 128 + ((c ^ kq) << 4)), sstep = sc == 3 ? 1024u : 2048u;
        const uint32_t sa1 = sc == 3 ? stg + (uint32_t)((kq + 4) * 128 + ((c ^ (kq + 4)) << 4)) : sa0 + 1024u;
        const int chunk = tc0 + (col >> 4);                    // chunk of this thread's byte column
        const bool col_ok = (col >> 4) < w;
        bool alive_b = true;
        // The copies of a warp's block k are on their way while its block k - 1 goes to the tensor core.
        // (One copy of the code for all blocks: everything here is fetched cold on every call.)
        int r0 = 0, nrows = 0, sg = 0;
#pragma unroll 1
        for (int nxt = warp, k = 0; warp < NL; nxt += NL, ++k) {
          const int p_r0 = r0, p_nrows = nrows, p_sg = sg;
          // the stage to fill was last read by the MMAs of block k - 2 (the low-nibble buffer likewise)
          const bool free_ok = uses == 0 || mbar_wait(my_empty, (uses - 1u) & 1u, abortp, spin);
          if (!__all_sync(0xffffffffu, free_ok)) { alive_b = false; break; }
          if (nxt < nblk) {
            if (nsuper > 1) {
              sg = __popc(__ballot_sync(0xffffffffu, sg_end <= nxt));
              const int first = __shfl_sync(0xffffffffu, sg_end - (int)sg_nb, sg);
              r0 = __shfl_sync(0xffffffffu, sg_r0, sg) + ((nxt - first) << 5);
              nrows = min(32, __shfl_sync(0xffffffffu, sg_r1, sg) - r0);
            } else {
              r0 = nxt << 5;
              nrows = min(32, k1 - r0);
            }
            // rows beyond nrows and columns beyond the tile keep whatever is there: their digits are zero, their sums unused
            const uint16_t* const ip = idx16 + r0 + kq;
            const uint32_t so = (uint32_t)((k & 1) * 4096);
            const int left = nrows - kq;
#pragma unroll
            for (int j = 0; j < 8; ++j)
              if (j * rpi < left) cp_async16(((j & 1) ? sa1 : sa0) + so + (uint32_t)(j >> 1) * sstep, tp + (unsigned)ip[j * rpi] * (unsigned long long)(unsigned)row_bytes);
          }
          cp_async_commit();
          if (tl == 0 && k == 0) PROX_TRACE(22);
          if (k > 0) {
            const uint32_t st1 = (uint32_t)((k - 1) & 1);
            uint4 brow = make_uint4(0u, 0u, 0u, 0u);
            if (lane < p_nrows) {
              const int i = idx16[p_r0 + lane];
              const uint32_t dg = x_digits(xs[i], ebase);
              const int slot = per_row ? 0 : ((i >> p.gshift) & 3);
              brow.x = slot == 0 ? dg : 0u; brow.y = slot == 1 ? dg : 0u; brow.z = slot == 2 ? dg : 0u; brow.w = slot == 3 ? dg : 0u;
            }
            asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(dig + st1 * 512u + (uint32_t)lane * 16u), "r"(brow.x), "r"(brow.y), "r"(brow.z), "r"(brow.w) : "memory");
            cp_async_wait<1>();
            __syncwarp();
            if (LO) {
              uint4 v[8];
#pragma unroll
              for (int j = 0; j < 8; ++j) v[j] = lds128(stg + st1 * 4096u + (uint32_t)(j * 512 + lane * 16));
#pragma unroll
              for (int j = 0; j < 8; ++j)
                asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(stg + 8192u + (uint32_t)(j * 512 + lane * 16)), "r"(v[j].x & 0x0f0f0f0fu),
                             "r"(v[j].y & 0x0f0f0f0fu), "r"(v[j].z & 0x0f0f0f0fu), "r"(v[j].w & 0x0f0f0f0fu) : "memory");
            }
            fence_proxy_async();                 // the tensor core reads the stage through the async proxy
            __syncwarp();
            if (elect_one()) {
              umma_i8(tbase + (uint32_t)(16 * p_sg), adesc + (uint64_t)(st1 * 256u), bdesc + (uint64_t)(st1 * 32u), idesc, 1u);
              if (LO) umma_i8(tbase + 256u + (uint32_t)(16 * p_sg), ldesc, bdesc + (uint64_t)(st1 * 32u), idesc, 1u);
              umma_commit(my_empty);
            }
            __syncwarp();
            if (uses == 0 && tl == 0) PROX_TRACE(23);
            ++uses;
          }
          if (nxt >= nblk) break;
        }
        cp_async_wait<0>();
        if (warp < NL && elect_one()) umma_commit(smem_u32(&sm.acc_bar));   // one arrival per loader warp once its MMAs are complete
        __syncwarp();
        PROX_TRACE(24);
        // ---- read the accumulators back: thread = byte column, warp part p takes supergroups p, p + 4, ...
        // (the four groups' scales of this byte column: gate / up scales sit in the order of the bytes)
        auto load_scales = [&](int sgq, uint32_t* dst) {
#pragma unroll
          for (int gq = 0; gq < 4; ++gq) {
            const int g = 4 * sgq + gq;
            dst[gq] = 0u;
            if (col_ok && g < ng) {
              if (LO) dst[gq] = __ldg(reinterpret_cast<const uint32_t*>(p.S + ((size_t)g * nchunks + chunk) * 32) + (col & 15));
              else dst[gq] = (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(p.S + ((size_t)g * nchunks + chunk) * 16) + (col & 15));
            }
          }
        };
        uint32_t scn[4];
        load_scales(part, scn);
        bool acc_ok = __all_sync(0xffffffffu, alive_b && mbar_wait(smem_u32(&sm.acc_bar), acc_n & 1u, abortp, spin));
        ++acc_n;
        tc_fence_after();
        if (tl == 0) {                         // the groups' offsets come from the four warps that do not load
          const unsigned want = (unsigned)kFusedProducers + (vid == 0 ? p.bar_bias >> 31 : 0u);       // (test knob)
          volatile unsigned* const cnt = &sm.soff_cnt;
#pragma unroll 1
          for (unsigned it = 0; *cnt < want && it < spin; ++it) __nanosleep(32);
          if (!__all_sync(0xffffffffu, *cnt >= want)) { acc_ok = false; *abortp = 1; }
          __threadfence_block();
        }
        PROX_TRACE(25);
        float t0 = 0.f, t1 = 0.f;              // 4-bit: sums of the low / high nibble's channel; 8-bit: t0 only
        const bool more = tl + 1 < ntl;
#pragma unroll 1
        for (int sgd = part; sgd < nsuper; sgd += 4) {
          if (!acc_ok) break;
          uint32_t a[16], l[16];
          const uint32_t ta = tbase + ((uint32_t)(q4 * 32) << 16) + (uint32_t)(16 * sgd);
          tmem_ld16(ta, a);
          if (LO) tmem_ld16(ta + 256u, l);
          uint32_t sc4[4];
#pragma unroll
          for (int gq = 0; gq < 4; ++gq) sc4[gq] = scn[gq];
          load_scales(sgd + 4, scn);           // the next round's scales are on their way during this one
          tmem_ld_wait();
          if (more) { tmem_st16_zero(ta); if (LO) tmem_st16_zero(ta + 256u); }
#pragma unroll
          for (int gq = 0; gq < 4; ++gq) {
            const int g = 4 * sgd + gq;
            const float off = sm.soff[min(g, ng - 1)];
            const float fa = digits_to_float(a[4 * gq], a[4 * gq + 1], a[4 * gq + 2], a[4 * gq + 3]);
            if (LO) {
              const float fl = digits_to_float(l[4 * gq], l[4 * gq + 1], l[4 * gq + 2], l[4 * gq + 3]);
              const float2 sc = __half22float2(*reinterpret_cast<const __half2*>(&sc4[gq]));
              t0 = fmaf(sc.x, fl - off, t0);
              t1 = fmaf(sc.y, fmaf(fa - fl, 0.0625f, -off), t1);
            } else {
              const float sc = __half2float(__ushort_as_half((unsigned short)sc4[gq]));
              t0 = fmaf(sc, fa - off, t0);
            }
          }
        }
        PROX_TRACE(26);
        if (more) { tmem_st_wait(); tc_fence_before(); }
        float* const red = (tl & 1) ? red1 : red0;
        if (part > 0) { red[((part - 1) * 128 + col) * 2] = t0; red[((part - 1) * 128 + col) * 2 + 1] = t1; }
        consumer_sync();
        if (more) tc_fence_after();            // every warp's columns are back at zero before the next tile's MMAs
        if (part == 0) {
#pragma unroll
          for (int pp = 0; pp < 3; ++pp) { t0 += red[(pp * 128 + col) * 2]; t1 += red[(pp * 128 + col) * 2 + 1]; }
          t0 = scalbnf(t0, ebase - 134); t1 = scalbnf(t1, ebase - 134);
          // bytes 0..7 of a chunk hold gate codes, bytes 8..15 the up codes of the same channels
          const float u0 = __shfl_xor_sync(0xffffffffu, t0, 8), u1 = __shfl_xor_sync(0xffffffffu, t1, 8);
          unsigned n0 = 1u, n1 = 1u, b0 = 0u, b1 = 0u;          // (scores in front of this thread's in their bins)
          const bool give = MODE == kScoresOnly || *abortp == 0;          // a block that has given up hands nothing on
          // (the sign is cleared as a bit: it says "not there yet" to the other blocks, and bins go by the bits behind it; fabsf
          // need not clear it for what is not a number, as weights and inputs that are not finite make it)
          const unsigned k0 = __float_as_uint(u0 * silu_fast(t0)) & 0x7fffffffu, k1b = LO ? __float_as_uint(u1 * silu_fast(t1)) & 0x7fffffffu : 0u;
          const float s0 = __uint_as_float(k0), s1 = __uint_as_float(k1b);
          if (MODE == kWhole && THRESH) {
            // marks of a chunk: bit i = its channel i (4-bit codes: a lane has channels 2 i and 2 i + 1)
            const unsigned m0 = __ballot_sync(0xffffffffu, k0 >= p.tkey_s) >> (lane & 16), m1 = LO ? __ballot_sync(0xffffffffu, k1b >= p.tkey_s) >> (lane & 16) : 0u;
            if ((lane & 15) == 0 && col_ok && give) st_relaxed(reinterpret_cast<unsigned*>(xhalf) + chunk, LO ? every_other_bit(m0 & 0xffu) | (every_other_bit(m1 & 0xffu) << 1) : m0 & 0xffu);
          }
          const unsigned knext = LO ? k1b : (MODE == kWhole && !THRESH) ? __shfl_down_sync(0xffffffffu, k0, 1) : 0u;
          if ((col & 8) == 0 && col_ok && give) {
            const int ch = chunk * CH + (LO ? 2 : 1) * (col & 7);
            if (MODE == kWhole && !THRESH) {
              // (halves in whole words, as they are read: 8-bit codes have the odd channel's in the next lane)
              if (LO || (lane & 1) == 0) st_relaxed(reinterpret_cast<unsigned*>(xhalf + ch), __byte_perm(k0, knext, 0x7632));
              if (LO) st_relaxed2(xkeys + ch, k0, k1b);
              else st_relaxed(xkeys + ch, k0);
            }
            if (LO) __stcg(reinterpret_cast<float2*>(p.scores + ch), make_float2(s0, s1));
            else __stcg(p.scores + ch, s0);
            if (HIST) {
              b0 = k0 >> 20; n0 = atomicAdd(&sm.hist[b0], 1u);
              if (LO) { b1 = k1b >> 20; n1 = atomicAdd(&sm.hist[b1], 1u); }
            }
          }
          if (HIST && ntl == 1) {
            // one global atomic per occupied bin (thousands of single increments on a few hot bins serialise in L2), by the
            // thread that came first to the bin; with several tiles at the end of the share (done per tile, the pause between
            // tiles cost 1.2 % of 4096 x 14336 8-bit and of 8192 x 28672)
            __syncwarp();
            asm volatile("bar.sync 4, 128;" ::: "memory");
            if (n0 == 0u) { atomicAdd(ghist + b0, sm.hist[b0]); sm.hist[b0] = 0u; }
            if (n1 == 0u) { atomicAdd(ghist + b1, sm.hist[b1]); sm.hist[b1] = 0u; }
          }
        }
      }
      // nothing may be in flight when the block frees the tensor memory (only a block whose wait expired gets here early)
      if (sm.abort_flag && lane == 0) {
#pragma unroll 1
        for (unsigned it = 0; it < 65536u && uses > 0; ++it) {
          if (mbar_try_wait(my_empty, (uses - 1u) & 1u)) break;
          __nanosleep(64);
        }
      }
    }
    else {
      // Blocks without a column pull the kept rows into L2 (a warp a row at a time): the loader
      // warps of the other blocks then find them there instead of waiting for HBM one by one.
      if (vid >= n1 && first) {
        const int nidle = max(G - (int)n1, 1);
#pragma unroll 1
        for (int r = (int)(vid - n1) * kFusedProducers + warp - kFusedConsumerWarps; r < k1; r += nidle * kFusedProducers) prefetch_row(idx16[r]);
      }
      if (HIST && first) {                     // the block's own score histogram (used behind the wait for soff_cnt)
#pragma unroll 1
        for (int i = tid - kFusedConsumers; i < 512; i += 32 * kFusedProducers) reinterpret_cast<uint4*>(sm.hist)[i] = make_uint4(0u, 0u, 0u, 0u);
      }
      // the other four warps: per scale group, offset * sum of the kept x as integers (for the codes' offset binary)
#pragma unroll 1
      for (int g = warp - kFusedConsumerWarps; first && g < ng; g += kFusedProducers) {
        int d0 = 0, d1 = 0, d2 = 0, d3 = 0;
#pragma unroll 1
        for (int r = sm.gstart[g] + lane; r < sm.gstart[g + 1]; r += 32) {
          const uint32_t dg = x_digits(xs[idx16[r]], ebase);
          d0 += (int)(int8_t)(dg & 0xffu); d1 += (int)(int8_t)((dg >> 8) & 0xffu);
          d2 += (int)(int8_t)((dg >> 16) & 0xffu); d3 += (int)(int8_t)(dg >> 24);
        }
        d0 = __reduce_add_sync(0xffffffffu, d0); d1 = __reduce_add_sync(0xffffffffu, d1);
        d2 = __reduce_add_sync(0xffffffffu, d2); d3 = __reduce_add_sync(0xffffffffu, d3);
        if (lane == 0) sm.soff[g] = (LO ? 8.f : 128.f) * digits_to_float((uint32_t)d0, (uint32_t)d1, (uint32_t)d2, (uint32_t)d3);
      }
      __syncwarp();
      if (first && lane == 0) { __threadfence_block(); atomicAdd(&sm.soff_cnt, 1u); }
    }
    tc_fence_before();
    fence_proxy_async();                        // phase B's plain accesses to the big buffer come before the ring's bulk copies
    __syncthreads();
    if (HIST && ntl > 1 && warp < kFusedConsumerWarps) {      // (only by them: phase C counts in sm.hist behind their barrier, not the block's)
#pragma unroll 1
      for (int i = tid; i < 2048; i += kFusedConsumers) { const unsigned v = sm.hist[i]; if (v) { atomicAdd(ghist + i, v); sm.hist[i] = 0u; } }
    }
    PROX_TRACE(3);
    if (MODE == kWhole && tid == 0 && vid < n1 && sm.abort_flag == 0)
      asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(ctr + kOut1) : "memory");
    if (MODE == kScoresOnly) {
      if (tid == 0) {
        // a block that has given up does not finish its share
        unsigned more1 = (unsigned)p.nshare1;
        if (vid < more1 && sm.abort_flag == 0) {
          asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ctr + kDone1) : "memory");
          asm volatile("atom.relaxed.gpu.global.add.u32 %0, [%1], 1;" : "=r"(more1) : "l"(ctr + kClaim1) : "memory");
        }
        sm.again = more1 < (unsigned)p.nshare1; sm.vid = more1;
      }
      __syncthreads();
    }
  }
  if (MODE == kScoresOnly) {
    if (!sm.again) break;
  } else {
  // ---------------------------------------- C: channel mask (top-k2 of the scores)
  // The blocks wait for a count of finished shares that is not ordered behind the scores; the scores themselves say that
  // they are there (all ones = not yet), and the histogram that it is complete (it counts all channels): what is missing is read
  // again.  That needs every aligned 32-bit word to be written and read as one, and a later read to see what has been written by
  // then: relaxed stores and loads at gpu scope promise both.  The copies of the first round promise neither by the letter
  // (they are weak); they go to L2, where the words are whole, and a word that they miss is one more round, of relaxed loads.  (With a barrier, i.e. a count released behind the acknowledgement of all the block's writes and acquired, and with whole
  // scores, counted by every thread in a run of its own, the first copy of phase D came 6.2 us after the last block's scores at
  // 4096 x 12288 where it comes after 4.8, and 3.6 instead of 2.9 at 512 x 1536.  What goes to every block is 2 bytes per channel;
  // the threshold form hands on one bit, which the block that has the score decides.  Reading histogram and scores in a loop
  // without waiting for the count, 148 blocks on the same lines, kept the last scores from getting there: 15 % slower.)
  // The first histogram level tells which channels are kept whatever the exact
  // threshold turns out to be (their bin lies above the threshold bin b1:
  // "definite", nd of them) and which are still open (the nb1 members of b1).
  // The kept list is laid out as [definite][kept members of b1], either part in the order of the threads that hold the
  // scores; block c owns the c-th share of either part.  Its definite share is known after one pass over the half scores,
  // so its weight rows start to stream while the consumer warps still settle the threshold inside b1.
  int n_mine = 0;
  unsigned nd = 0, b1 = 0, kk = 0, nb1 = 0;     // (THRESH: nd = the kept channels)
  unsigned cnt = 0, ex = 0;                     // packed: definite channels (low half) and members of b1 of this thread / in front of it
  const int ngrp = THRESH ? F / CH / 4 : F / 8;  // 16-byte groups of half scores (THRESH: of mark words)
  const unsigned NSH = (unsigned)p.nshare;
  int ndm = 0, ncm = 0, Rc0 = 0, Rc1 = 0;
  // Shared-memory plan: the half scores (THRESH: marks) sit at the END of the big buffer (the ring fills from slot 0 and
  // reaches those slots last); the list of b1's members goes where the input index list was (free since phase B), or in
  // front of the half scores if it is long.  Consumer thread t owns the groups t, t + 512, ... (THRESH: a run of them, so
  // that the list is ascending)
  const int q0 = THRESH ? tid * ((ngrp + kFusedConsumers - 1) / kFusedConsumers) : tid, qstep = THRESH ? 1 : kFusedConsumers;
  const int qend = THRESH ? min(ngrp, q0 + (ngrp + kFusedConsumers - 1) / kFusedConsumers) : ngrp;
  const bool in_smem = (size_t)F * 2 + 256 <= (size_t)p.big_bytes;
  const uint32_t key_off = in_smem ? (((uint32_t)p.big_bytes - (uint32_t)ngrp * 16u) & ~127u) : 0u;
  const uint32_t skey_u32 = big_u32 + key_off;
  uint32_t list_u32 = smem_u32(idx16);          // 2 * D bytes: room for D / 2 members
  unsigned klo = 0, khi = 0;                    // half scores from khi on are definite, from klo on members of b1
  auto full_key = [&](int i) {                  // all bits of a score (a bounded wait, which ends once the abort flag is up)
    unsigned v;
#pragma unroll 1
    for (unsigned it = 0;; ++it) {
      asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(xkeys + i) : "memory");
      if (v != kNoKey && !(p.bar_bias & kBiasKeys)) break;
      if (it >= spin || *abortp) { *abortp = 1; break; }
    }
    return v;
  };
  if (warp >= kFusedConsumerWarps) {
    if (MODE == kWhole && with_b) {
      // (in the layer form in place, the blocks wait for this count before they add to the residual stream that others read)
      if (tid == kFusedConsumers && vid < (unsigned)p.nshare1 && sm.abort_flag == 0)
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(ctr + kDone1) : "memory");
      widen_x(kFusedConsumers);
    }
  } else if (MODE == kGivenList) {
    const unsigned shr = sm.shr;
    const unsigned n = (unsigned)(p.sel_cnt ? min(max(__ldcg(p.sel_cnt), 0), F) : k2);
    const int R0 = (int)((n * shr) / NSH);
    n_mine = shr < NSH ? min((int)((n * (shr + 1u)) / NSH) - R0, kMySelCap) : 0;
#pragma unroll 1
    for (int i = tid; i < n_mine; i += kFusedConsumers) {
      const int j = p.sel_in[R0 + i];
      if (j < 0 || j >= F) atomicOr(p.status, kBadChannel);
      sm.mysel[i] = (j < 0 || j >= F) ? -1 : j;
    }
    if (tid == 0) { sm.keys_s0 = sm.keys_s1 = sm.list_s0 = sm.list_s1 = 0; sm.n_mine = n_mine; sm.nready = n_mine; sm.keys_done = 1; sm.c_done = 1; }
  } else if (sm.abort_flag == 0) {
    uint4 hv = make_uint4(0u, 0u, 0u, 0u);
    unsigned hsum = 0, hbase = 0;
    if (tid == 0) {
      unsigned more1 = (unsigned)p.nshare1, share2 = 0, out = 0;
      // another share of Stage 1 (there is none unless a block of the grid is not running), and one of Stage 2
      if (with_b && vid < more1) asm volatile("atom.relaxed.gpu.global.add.u32 %0, [%1], 1;" : "=r"(more1) : "l"(ctr + kClaim1) : "memory");
      if (with_b && first) asm volatile("atom.relaxed.gpu.global.add.u32 %0, [%1], 1;" : "=r"(share2) : "l"(ctr + kClaim2) : "memory");
#pragma unroll 1
      for (unsigned it = 0; it < spin; ++it) {
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(out) : "l"(ctr + kOut1) : "memory");
        if (out >= (unsigned)p.nshare1 || more1 < (unsigned)p.nshare1) break;
      }
      sm.again = more1 < (unsigned)p.nshare1;
      if (with_b) { sm.vid = more1; if (first) sm.shr = share2; }
      sm.res[7] = out >= (unsigned)p.nshare1;
    }
    consumer_sync();
    PROX_TRACE(17);
    bool ok = false;
    const bool again = sm.again != 0;
    // (a block that has given up hands nothing on, so that the scores are never complete and the call ends before
    // anything is written to y or to the residual stream; neither are they with the test knob)
    const unsigned target = (p.bar_bias & (kBiasKeys - 1u)) ? ~0u : (THRESH ? 0u : (unsigned)F);
    const unsigned tries = !again && sm.res[7] ? spin : 0u;
#pragma unroll 1
    for (unsigned it = 0; it < tries; ++it) {
      if (!THRESH) hv = ld_relaxed4(ghist + 4 * (511 - tid));
      if (in_smem) {
#pragma unroll 1
        for (int q = q0; q < qend; q += qstep) {
          if (it == 0) {
            cp_async16(skey_u32 + (uint32_t)q * 16u, xhalf + 8 * q);
          } else {
            const uint4 v = ld_relaxed4(reinterpret_cast<const unsigned*>(xhalf) + 4 * q);
            asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(skey_u32 + (uint32_t)q * 16u), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
          }
        }
      }
      cp_async_commit();
      if (tid < 256) sm.hist2[tid] = 0;
      hsum = hv.x + hv.y + hv.z + hv.w;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) { const unsigned t = __shfl_up_sync(0xffffffffu, hsum, o); if (lane >= o) hsum += t; }
      if (lane == 31) sm.poll[0][warp] = hsum;
      consumer_sync();
      const unsigned pv = lane < kFusedConsumerWarps ? sm.poll[0][lane] : 0u;
      const unsigned tot = __reduce_add_sync(0xffffffffu, pv);
      hbase = __reduce_add_sync(0xffffffffu, lane < warp ? pv : 0u);
      if (tot != target) { cp_async_wait<0>(); consumer_sync(); continue; }
      if (!THRESH) {
        // the bin of the k2-th score: thread t has the counts of four bins in descending order, the threads' runs follow
        // each other downwards
        unsigned run = hbase + hsum - (hv.x + hv.y + hv.z + hv.w);
        if (run < (unsigned)k2 && (unsigned)k2 <= hbase + hsum) {
          unsigned c = hv.w, bin = 2047u - 4u * (unsigned)tid;
          if (run + c < (unsigned)k2) { run += c; c = hv.z; --bin; }
          if (run + c < (unsigned)k2) { run += c; c = hv.y; --bin; }
          if (run + c < (unsigned)k2) { run += c; c = hv.x; --bin; }
          sm.res[0] = bin; sm.res[1] = run; sm.res[2] = c;
        }
        consumer_sync();
        b1 = sm.res[0]; nd = sm.res[1]; nb1 = sm.res[2];
        kk = (unsigned)k2 - nd;                              // members of b1 to keep (>= 1)
      }
      PROX_TRACE(16);
      // a consumer thread counts its definite channels and its members of b1
      klo = b1 << 4; khi = (b1 + 1u) << 4;
      unsigned from_lo = 0, from_hi = 0, any = 0;
      cp_async_wait<0>();
#pragma unroll 1
      for (int q = q0; q < qend; q += qstep) {
        const uint4 v = in_smem ? lds128(skey_u32 + (uint32_t)q * 16u) : ld_relaxed4(reinterpret_cast<const unsigned*>(xhalf) + 4 * q);
        any |= v.x | v.y | v.z | v.w;
        const unsigned w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (THRESH) {
            from_hi += (unsigned)__popc(w4[e] & 0xffffu);
          } else {
            from_hi += (w4[e] >= khi << 16 ? 1u : 0u) + (w4[e] << 16 >= khi << 16 ? 1u : 0u);
            from_lo += (w4[e] >= klo << 16 ? 1u : 0u) + (w4[e] << 16 >= klo << 16 ? 1u : 0u);
          }
        }
      }
      if (THRESH) from_lo = from_hi;
      cnt = from_hi | ((from_lo - from_hi) << 16);
      ex = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) { const unsigned t = __shfl_up_sync(0xffffffffu, ex, o); if (lane >= o) ex += t; }
      const bool bad = __any_sync(0xffffffffu, any & (THRESH ? 0x80000000u : 0x80008000u));     // the sign of what is not there
      if (lane == 31) { sm.wsum[warp] = ex; sm.poll[1][warp] = bad ? 1u : 0u; }
      consumer_sync();
      if (!__any_sync(0xffffffffu, lane < kFusedConsumerWarps && sm.poll[1][lane] != 0u)) { ok = true; break; }
      consumer_sync();
    }
    PROX_TRACE(4);
    if (!ok) {
      if (!again && tid == 0) { sm.abort_flag = 1; atomicOr(p.status, kWaitExpired); if (p.host_flag) *reinterpret_cast<volatile int*>(p.host_flag) = 1; }
    } else {
      const unsigned shr = sm.shr;
      ex = __reduce_add_sync(0xffffffffu, (lane < warp) ? sm.wsum[lane] : 0u) + ex - cnt;
      uint32_t list_off = 0;                                 // offset in the big buffer when the list has to go there
      bool list_in_big = false;
      bool staged = in_smem;                                 // the same in every block
      if (in_smem && (size_t)nb1 * 4 > (size_t)D * 2) {
        if ((size_t)nb1 * 4 + 128 <= (size_t)key_off) {
          list_off = (key_off - nb1 * 4u) & ~127u; list_u32 = big_u32 + list_off; list_in_big = true;
        } else {
          staged = false;
        }
      }
      if (THRESH) {
        nd = __reduce_add_sync(0xffffffffu, (lane < kFusedConsumerWarps) ? (sm.wsum[lane] & 0xffffu) : 0u);
        if (shr == 0 && tid == 0) {
          if (p.count_out) p.count_out[0] = (int)nd;
          if (p.counters) atomicAdd(p.counters + 2, (unsigned long long)nd);
        }
      }
      if (staged && shr < NSH) {
        // k2 * G < 2^31 is checked on the host, so the share bounds fit 32 bits
        const int Rd0 = (int)((nd * shr) / NSH);
        ndm = min((int)((nd * (shr + 1u)) / NSH) - Rd0, kMySelCap);
        Rc0 = (int)((kk * shr) / NSH);
        ncm = THRESH ? 0 : min((int)((kk * (shr + 1u)) / NSH) - Rc0, kMySelCap - ndm);
        Rc1 = Rc0 + ncm;
        const int Rd1 = Rd0 + ndm;
        n_mine = ndm + ncm;
        if (tid == 0) {
          const uint32_t rb = (uint32_t)D * 2u;
          sm.keys_s0 = (int)(key_off / rb); sm.keys_s1 = (int)((key_off + (uint32_t)ngrp * 16u + rb - 1u) / rb);
          sm.list_s0 = list_in_big ? (int)(list_off / rb) : 0;
          sm.list_s1 = list_in_big ? (int)((list_off + nb1 * 4u + rb - 1u) / rb) : 0;
          sm.n_mine = n_mine; sm.nready = ndm; sm.keys_done = sm.c_done = (ncm == 0) ? 1 : 0;
        }
        // the threads whose definite channels meet the block's share (a few neighbours): their warp lists them, one
        // thread's channels after the other
        const int dpos = (int)(ex & 0xffffu), cdef = (int)(cnt & 0xffffu);
        constexpr int GC = THRESH ? 4 * CH : 8;              // channels of a group
        const int nel = (THRESH ? (ngrp + kFusedConsumers - 1) / kFusedConsumers : (ngrp - warp * 32 + kFusedConsumers - 1) / kFusedConsumers) * GC;
#pragma unroll 1
        for (unsigned lanes = __ballot_sync(0xffffffffu, cdef > 0 && dpos < Rd1 && dpos + cdef > Rd0); lanes; lanes &= lanes - 1) {
          const int l = __ffs((int)lanes) - 1;
          int at = __shfl_sync(0xffffffffu, dpos, l) - Rd0;
          const int ql = __shfl_sync(0xffffffffu, q0, l);
#pragma unroll 1
          for (int i = lane; i < ((nel + 31) & ~31); i += 32) {
            const int q = ql + (i / GC) * qstep, c = i % GC;
            bool def = i < nel && q < ngrp;
            if (def) {
              unsigned v;
              if (THRESH) {
                asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(skey_u32 + (uint32_t)(q * 16 + (c / CH) * 4)));
                def = (v >> (c % CH)) & 1u;
              } else {
                asm volatile("{\n\t.reg .u16 h;\n\tld.shared.u16 h, [%1];\n\tcvt.u32.u16 %0, h;\n\t}" : "=r"(v) : "r"(skey_u32 + (uint32_t)(q * 16 + c * 2)));
                def = v >= khi;
              }
            }
            const unsigned b = __ballot_sync(0xffffffffu, def);
            const int pos = at + __popc(b & lt_mask);
            if (def && pos >= 0 && pos < ndm) sm.mysel[pos] = q * GC + c;
            at += __popc(b);
          }
        }
      } else if (!THRESH && shr < NSH) {
        // no room for the list: the block's share of the plain ascending mask, before the ring starts (the threshold form has no list
        // and is not launched where its marks do not fit; with the call in it, 3072 x 8896 8-bit took 59.5 us for two layers instead of 58.4)
        n_mine = settle_over_all_channels(xkeys, F, (unsigned)k2, shr, NSH, b1, kk, p.sel_out, spin, p.bar_bias);
        if (tid == 0) { sm.keys_s0 = sm.keys_s1 = sm.list_s0 = sm.list_s1 = 0; sm.n_mine = n_mine; sm.nready = n_mine; sm.keys_done = 1; sm.c_done = 1; }
      }
    }
  }
  __syncthreads();                              // the block's definite share is listed: the producer warps may start
  PROX_TRACE(21);
  const bool alive = sm.abort_flag == 0;        // block-uniform; a dead block skips to the end
  if (MODE == kWhole && alive && with_b && sm.again) continue;      // one more share of Stage 1
  with_b = false;
  if (alive && sm.shr >= NSH) break;
  if (MODE == kWhole && alive && p.sel_out && warp == kFusedConsumerWarps - 1 && ndm > 0) {       // the mask, for prox_ffn_last_mask
    const int Rd0 = (int)((nd * sm.shr) / NSH);
#pragma unroll 1
    for (int i = lane; i < ndm; i += 32) p.sel_out[Rd0 + i] = sm.mysel[i];
  }
  if (MODE == kWhole && !THRESH && warp < kFusedConsumerWarps && ncm > 0) {
        // ---- consumer warps only: the list of b1's members (channel, and the four bits that its half score has below the
        // bin's, with their histogram) ...
        if (cnt >> 16) {
          unsigned cpos = ex >> 16;
#pragma unroll 1
          for (int q = q0; q < qend; q += qstep) {
            const uint4 v = lds128(skey_u32 + (uint32_t)q * 16u);
            const unsigned w4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const unsigned h = e & 1 ? w4[e >> 1] >> 16 : w4[e >> 1] & 0xffffu;
              if (h >= klo && h < khi) {
                if (cpos < nb1) asm volatile("st.shared.u32 [%0], %1;" ::"r"(list_u32 + cpos * 4u), "r"((h & 15u) << 16 | (unsigned)(8 * q + e)) : "memory");
                atomicAdd(&sm.hist2[h & 15u], 1u);
                ++cpos;
              }
            }
          }
        }
        // The upper half of the consumer warps goes on to the gate/up rows that are streaming in
        // already; the lower half ("settlers") finishes the mask and joins them later.
        if (warp >= kSettlerWarps) {
          asm volatile("bar.arrive 2, %0;" ::"n"(kFusedConsumers) : "memory");
        } else {
        asm volatile("bar.sync 2, %0;" ::"n"(kFusedConsumers) : "memory");      // the list is complete, the half scores are free
        if (tid == 0) *reinterpret_cast<volatile int*>(&sm.keys_done) = 1;
        PROX_TRACE(15);
        // ... the value of those bits at which the kk-th of them lies (every warp on its own): members above it are kept ...
        const unsigned hc = lane < 16 ? sm.hist2[15 - lane] : 0u, hi = warp_scan_incl(hc, lane);
        const int src = __ffs((int)__ballot_sync(0xffffffffu, hi >= kk)) - 1;
        const unsigned sub = 15u - (unsigned)src, above = __shfl_sync(0xffffffffu, hi - hc, src), kk2 = kk - above;
        const unsigned n2 = __shfl_sync(0xffffffffu, hc, src);
        // ... in list order (a thread owns a run of the list), and of the n2 with that value those that rank among the first
        // kk2 by (score descending, channel ascending), in that order
        const int ept = ((int)nb1 + kSettlers - 1) / kSettlers;
        const int c0 = min((int)nb1, tid * ept), c1 = min((int)nb1, c0 + ept);
        unsigned wt = 0;
#pragma unroll 1
        for (int c = c0; c < c1; ++c) {
          const unsigned e = lds32(list_u32 + (uint32_t)c * 4u);
          wt += (e >> 16) > sub ? 1u : 0u;
          if ((e >> 16) == sub && n2 <= (unsigned)kCand2Cap) {
            const unsigned slot = atomicAdd(&sm.ncand2, 1u);
            sm.cand2_key[slot] = full_key((int)(e & 0xffffu)); sm.cand2_idx[slot] = (int)(e & 0xffffu);
          }
        }
        const unsigned inc3 = warp_scan_incl(wt, lane);
        if (lane == 31) sm.warp_cnt[warp][0] = inc3;
        settler_sync();
        PROX_TRACE(19);
        auto keep = [&](int pos, unsigned ch) {
          if (pos >= Rc0 && pos < Rc1) {
            sm.mysel[ndm + pos - Rc0] = (int)ch;
            if (p.sel_out) p.sel_out[(int)nd + pos] = (int)ch;
          }
        };
        int pos = (int)(__reduce_add_sync(0xffffffffu, lane < warp ? sm.warp_cnt[lane][0] : 0u) + inc3 - wt);
        if (wt > 0 && pos < Rc1 && pos + (int)wt > Rc0) {
#pragma unroll 1
          for (int c = c0; c < c1; ++c) {
            const unsigned e = lds32(list_u32 + (uint32_t)c * 4u);
            if ((e >> 16) > sub) keep(pos++, e & 0xffffu);
          }
        }
        if (n2 <= (unsigned)kCand2Cap) {
          if (tid < (int)n2) {
            const unsigned key = sm.cand2_key[tid];
            const int id = sm.cand2_idx[tid];
            unsigned rank = 0;
#pragma unroll 4
            for (unsigned c = 0; c < n2; ++c) {
              const unsigned ok = sm.cand2_key[c];
              const int oi = sm.cand2_idx[c];
              rank += (ok > key || (ok == key && oi < id)) ? 1u : 0u;
            }
            if (rank < kk2) keep((int)(above + rank), (unsigned)id);
          }
        } else {
          settle_equal_halves(list_u32, nb1, sub, kk2, xkeys, (int)above, Rc0, Rc1, ndm, p.sel_out ? p.sel_out + (int)nd : nullptr, spin, p.bar_bias);
        }
        PROX_TRACE(20);
        __threadfence_block();
        settler_sync();                          // the list is free from here on
        if (tid == 0 && !*abortp) {              // (without all scores the list may have gaps: no rows are asked for by it)
          *reinterpret_cast<volatile int*>(&sm.nready) = n_mine;
          __threadfence_block();
          *reinterpret_cast<volatile int*>(&sm.c_done) = 1;
        }
        PROX_TRACE(6);
        }
  }

  PROX_TRACE(5);
  // -------------------------------- D + E: exact gate/up, SwiGLU, masked down
  const int nv = D / 8;                       // 16-byte vectors per row
  const uint32_t row_bytes2 = (uint32_t)D * 2u;
  const int NS = p.nslots;
  constexpr int TG = kFusedConsumers / NG;    // threads of one down-projection group
  constexpr int EV = 4;                       // 16-byte vectors a thread owns in the down projection
  float yr[EV][8];
#pragma unroll
  for (int m = 0; m < EV; ++m)
#pragma unroll
    for (int j = 0; j < 8; ++j) yr[m][j] = 0.f;

  if (warp >= kFusedConsumerWarps) {
    // ---- producer warps: lane 0 of each feeds every kFusedProducers-th slot of
    // the ring (one thread can only start a few million bulk copies a second)
    if (lane == 0 && alive) {
      fence_proxy_async();                      // the big buffer becomes a bulk-copy target now
      n_mine = sm.n_mine;
      const unsigned pq = (unsigned)(warp - kFusedConsumerWarps);
      unsigned seq = pseq, use = puse;
      int slot = pslot;
      bool dead = false;
      int ready = *reinterpret_cast<volatile int*>(&sm.nready);
      bool kdone = *reinterpret_cast<volatile int*>(&sm.keys_done) != 0;
      bool cdone = *reinterpret_cast<volatile int*>(&sm.c_done) != 0;
      const int ks0 = sm.keys_s0, ks1 = sm.keys_s1, ls0 = sm.list_s0, ls1 = sm.list_s1;
#pragma unroll 1
      for (int b0 = 0; b0 < n_mine && !dead; b0 += kChanBatch) {
        const int nb = min(kChanBatch, n_mine - b0);
#pragma unroll 1
        for (int q = 0; q < 3 * nb; ++q, ++seq) {
          // A slot always belongs to the same producer: its uses are then armed
          // in program order, so the parity wait below is never two phases behind.
          if (((unsigned)slot & (unsigned)(kFusedProducers - 1)) == pq) {
            const int mi = b0 + ((q < 2 * nb) ? (q >> 1) : (q - 2 * nb));
            // The tail of the list (the share of the threshold bin) is written late, and the ring
            // may not touch the slots under the half scores and the list before the consumer warps are done with them.
            auto blocked = [&]() {
              return mi >= ready || (!kdone && slot >= ks0 && slot < ks1) || (!cdone && slot >= ls0 && slot < ls1);
            };
            if (blocked()) {
#pragma unroll 1
              for (unsigned it = 0; it < spin; ++it) {
                ready = *reinterpret_cast<volatile int*>(&sm.nready);
                kdone = *reinterpret_cast<volatile int*>(&sm.keys_done) != 0;
                cdone = *reinterpret_cast<volatile int*>(&sm.c_done) != 0;
                if (!blocked() || *abortp) break;
                __nanosleep(64);
              }
              if (blocked()) { sm.abort_flag = 1; dead = true; break; }
              __threadfence_block();
              fence_proxy_async();
            }
            if (use > 0 && !mbar_wait(smem_u32(&sm.mbar_empty[slot]), (use - 1u) & 1u, abortp, spin)) { dead = true; break; }
            const uint16_t* src;
            if (q < 2 * nb) {
              src = ((q & 1) ? p.wu : p.wg) + (size_t)max(sm.mysel[mi], 0) * D;
            } else {
              src = p.wdt + (size_t)max(sm.mysel[mi], 0) * D;
            }
            const uint32_t bar = smem_u32(&sm.mbar_full[slot]);
            if (seq == 0) PROX_TRACE_AT(28, tid);
            if (seq == 2u * (unsigned)min(n_mine, kChanBatch)) PROX_TRACE_AT(30, tid);
            mbar_expect_tx(bar, row_bytes2);
            bulk_g2s(big_u32 + (uint32_t)slot * row_bytes2, src, row_bytes2, bar);
            atomicMax(&sm.prod_seq, seq + 1u);
          }
          if (++slot == NS) { slot = 0; ++use; }
        }
      }
      pseq = seq; puse = use; pslot = slot;
      if (pq == 0) {
        // all rows of the share are on their way: the next share, if there is one
        unsigned nx;
        asm volatile("atom.relaxed.gpu.global.add.u32 %0, [%1], 1;" : "=r"(nx) : "l"(ctr + kClaim2) : "memory");
        sm.shr_next = nx;
      }
    }
  } else {
    // ---- consumer warps
    const uint32_t xf_u32 = smem_u32(xf);
    if (NORM && alive && p.xres_out == p.xres && warp == kFusedConsumerWarps - 1) {
      // y goes straight into the residual stream below: not before all blocks with a share of Stage 1 have said that
      // they have read it (they said so when their scores were out, which are all here: no wait in practice)
      if (lane == 0) {
        bool seen = false;
#pragma unroll 1
        for (unsigned it = 0; !seen && it < spin; ++it) seen = ld_acquire(ctr + kDone1) >= (unsigned)p.nshare1;
        if (!seen) sm.abort_flag = 1;
      }
      __syncwarp();
    }
#pragma unroll 1
    for (int b0 = 0; b0 < n_mine; b0 += kChanBatch) {
      const int nb = min(kChanBatch, n_mine - b0);
      // D: a warp takes the next channel of the batch that nobody has taken yet (the warps
      // that finish the channel mask join late; rows are consumed in the order they arrive)
      for (;;) {
        int c = 0;
        if (lane == 0) c = (int)atomicAdd(&sm.next_c, 1u);
        c = __shfl_sync(0xffffffffu, c, 0);
        if (c >= nb) break;
        const unsigned sq = base_seq + 2u * (unsigned)c;
        const unsigned ug = __umulhi(sq, p.nslots_rcp);
        const int sg = (int)(sq - ug * (unsigned)NS), su = sg + 1 == NS ? 0 : sg + 1;
        const unsigned uu = ug + (su == 0 ? 1u : 0u);
        const bool ok1 = slot_wait(smem_u32(&sm.mbar_full[sg]), &sm.slot_use[sg], ug, abortp, spin);
        const bool ok2 = slot_wait(smem_u32(&sm.mbar_full[su]), &sm.slot_use[su], uu, abortp, spin);
        float ag = 0.f, au = 0.f, ag2 = 0.f, au2 = 0.f;
        if (ok1 && ok2) {
          const uint32_t pg = big_u32 + (uint32_t)sg * row_bytes2, pu = big_u32 + (uint32_t)su * row_bytes2;
#pragma unroll 2
          for (int v = lane; v < nv; v += 32) {
            const uint4 a = lds128(pg + (uint32_t)v * 16u);
            const uint4 b = lds128(pu + (uint32_t)v * 16u);
            const float4 x0 = lds128f(xf_u32 + (uint32_t)v * 32u);
            const float4 x1 = lds128f(xf_u32 + (uint32_t)v * 32u + 16u);
            ag = fmaf(bf16_lo(a.x), x0.x, ag); ag2 = fmaf(bf16_hi(a.x), x0.y, ag2);
            ag = fmaf(bf16_lo(a.y), x0.z, ag); ag2 = fmaf(bf16_hi(a.y), x0.w, ag2);
            ag = fmaf(bf16_lo(a.z), x1.x, ag); ag2 = fmaf(bf16_hi(a.z), x1.y, ag2);
            ag = fmaf(bf16_lo(a.w), x1.z, ag); ag2 = fmaf(bf16_hi(a.w), x1.w, ag2);
            au = fmaf(bf16_lo(b.x), x0.x, au); au2 = fmaf(bf16_hi(b.x), x0.y, au2);
            au = fmaf(bf16_lo(b.y), x0.z, au); au2 = fmaf(bf16_hi(b.y), x0.w, au2);
            au = fmaf(bf16_lo(b.z), x1.x, au); au2 = fmaf(bf16_hi(b.z), x1.y, au2);
            au = fmaf(bf16_lo(b.w), x1.z, au); au2 = fmaf(bf16_hi(b.w), x1.w, au2);
          }
        }
        ag = warp_sum(ag + ag2); au = warp_sum(au + au2);
        if (lane == 0) {
          const int j = sm.mysel[b0 + c];
          sm.hval[c] = (j >= 0 && j < F) ? au * silu_exact(ag) : 0.f;
          if (ok1 && ok2) {                       // never release a slot whose phase was not seen
            mbar_arrive_n(smem_u32(&sm.mbar_empty[sg]), kEmptyCount);
            mbar_arrive_n(smem_u32(&sm.mbar_empty[su]), kEmptyCount);
          }
        }
      }
      consumer_sync();
      if (tid == 0) sm.next_c = 0;               // for the next batch (nobody takes channels during E)
      // E: group gq (TG threads) owns rows gq, gq+NG, ... ; a thread owns EV vectors of y
      {
        const int gq = tid / TG, tg = tid % TG;
#pragma unroll 1
        for (int c = gq; c < nb; c += NG) {
          const unsigned sq = base_seq + 2u * (unsigned)nb + (unsigned)c;
          const unsigned ud = __umulhi(sq, p.nslots_rcp);
          const int sd = (int)(sq - ud * (unsigned)NS);
          const bool ok = slot_wait(smem_u32(&sm.mbar_full[sd]), &sm.slot_use[sd], ud, abortp, spin);
          if (ok) {
            const float hv = sm.hval[c];
            const uint32_t pd = big_u32 + (uint32_t)sd * row_bytes2;
#pragma unroll
            for (int m = 0; m < EV; ++m) {
              const int v = tg + m * TG;
              if (v < nv) {
                const uint4 wv = lds128(pd + (uint32_t)v * 16u);
                yr[m][0] = fmaf(hv, bf16_lo(wv.x), yr[m][0]); yr[m][1] = fmaf(hv, bf16_hi(wv.x), yr[m][1]);
                yr[m][2] = fmaf(hv, bf16_lo(wv.y), yr[m][2]); yr[m][3] = fmaf(hv, bf16_hi(wv.y), yr[m][3]);
                yr[m][4] = fmaf(hv, bf16_lo(wv.z), yr[m][4]); yr[m][5] = fmaf(hv, bf16_hi(wv.z), yr[m][5]);
                yr[m][6] = fmaf(hv, bf16_lo(wv.w), yr[m][6]); yr[m][7] = fmaf(hv, bf16_hi(wv.w), yr[m][7]);
              }
            }
          }
          __syncwarp();
          if (lane == 0 && ok) mbar_arrive_n(smem_u32(&sm.mbar_empty[sd]), (uint32_t)NG);   // TG/32 warps * NG = 16
        }
      }
      consumer_sync();                           // hval is reused by the next batch; all ring reads are done
      base_seq += 3u * (unsigned)nb;
    }
    PROX_TRACE(7);
    // the NG partial vectors of the block meet in shared memory (the ring is idle now)
    if (n_mine > 0) {
      float* ysum = reinterpret_cast<float*>(big);
      const int gq = tid / TG, tg = tid % TG;
#pragma unroll
      for (int m = 0; m < EV; ++m) {
        const int v = tg + m * TG;
        if (v < nv) {
          float4* dst = reinterpret_cast<float4*>(ysum + (size_t)gq * D + (size_t)v * 8);
          dst[0] = make_float4(yr[m][0], yr[m][1], yr[m][2], yr[m][3]);
          dst[1] = make_float4(yr[m][4], yr[m][5], yr[m][6], yr[m][7]);
        }
      }
      consumer_sync();
#pragma unroll 1
      for (int v4 = tid; v4 < D / 4 && !*abortp; v4 += kFusedConsumers) {       // (a block that has given up adds nothing)
        float4 s = reinterpret_cast<const float4*>(ysum)[v4];
#pragma unroll
        for (int g2 = 1; g2 < NG; ++g2) {
          const float4 t = reinterpret_cast<const float4*>(ysum + (size_t)g2 * D)[v4];
          s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
        }
        // layer form run in place on the residual stream: the block's share of y goes straight into it, and there is
        // nothing left to round at the end
        atomicAdd(reinterpret_cast<float4*>((NORM && p.xres_out == p.xres) ? p.xres_out : p.yacc) + v4, s);
      }
    }
  }

  // -------------------------------------- F: last block rounds y and cleans up
  __syncthreads();
  PROX_TRACE(8);
  if (sm.abort_flag) {
    // A wait expired: every copy this block armed was either consumed or is
    // waited for here (bounded) so that none lands after the block has left.
    if (tid == 0) {
      atomicOr(p.status, kWaitExpired);
      if (p.host_flag) *reinterpret_cast<volatile int*>(p.host_flag) = 1;
      const unsigned issued = sm.prod_seq;
      const unsigned first = issued > (unsigned)NS ? issued - (unsigned)NS : 0u;
#pragma unroll 1
      for (unsigned q = first; q < issued; ++q) {        // the latest use of every slot
        const uint32_t bar = smem_u32(&sm.mbar_full[q % (unsigned)NS]);
#pragma unroll 1
        for (unsigned it = 0; it < 8192u; ++it) {
          if (mbar_try_wait(bar, (q / (unsigned)NS) & 1u)) break;
          __nanosleep(256);
        }
      }
    }
    __syncthreads();
    if (warp == 0) tmem_free_all(sm.tmem_base);
    leave();
    return;
  }
  const unsigned next_shr = sm.shr_next;
  if (!(NORM && p.xres_out == p.xres)) {        // (in place y went straight into the residual stream: nothing to round)
  if (tid == 0) {
    // release: the block's atomics (ordered before this thread by the barrier above) are out before the ticket is
    // taken; acquire: the block that draws the last ticket sees every other block's
    unsigned t;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(t) : "l"(ctr + kDone2) : "memory");
    sm.s_last = (t == NSH - 1u);
  }
  __syncthreads();
  if (sm.s_last) {
#pragma unroll 1
    for (int i0 = tid * 4; i0 < D; i0 += NT * 4 * 4) {        // loads first: they must not queue behind the stores
      float4 v[4], r[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * NT * 4;
        v[u] = (i < D) ? __ldcg(reinterpret_cast<const float4*>(p.yacc + i)) : make_float4(0.f, 0.f, 0.f, 0.f);
        r[u] = (NORM && i < D) ? __ldcg(reinterpret_cast<const float4*>(p.xres + i)) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int i = i0 + u * NT * 4;
        if (i < D) {
          *reinterpret_cast<float4*>(p.yacc + i) = make_float4(0.f, 0.f, 0.f, 0.f);
          if (NORM) {
            *reinterpret_cast<float4*>(p.xres_out + i) =
                make_float4(r[u].x + v[u].x, r[u].y + v[u].y, r[u].z + v[u].z, r[u].w + v[u].w);
          } else if (p.out_fp32) {
            *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.y) + i) = v[u];
          } else {
            __nv_bfloat162 lo = __floats2bfloat162_rn(v[u].x, v[u].y), hi = __floats2bfloat162_rn(v[u].z, v[u].w);
            uint2 pk;
            pk.x = *reinterpret_cast<unsigned*>(&lo); pk.y = *reinterpret_cast<unsigned*>(&hi);
            *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.y) + i) = pk;
          }
        }
      }
    }
    __syncthreads();
    PROX_TRACE(9);
  }
  }
  if (next_shr >= NSH) break;
  __syncthreads();                              // everyone has read what is reset here
  if (tid == 0) { sm.shr = next_shr; sm.ncand2 = 0; sm.next_c = 0; sm.nready = 0; sm.n_mine = 0; sm.keys_done = 0; sm.c_done = 0; }
  __syncthreads();
  }
  }
  if (warp == 0) tmem_free_all(sm.tmem_base);
  if (MODE == kScoresOnly && tid == 0 && sm.abort_flag) { atomicOr(p.status, kWaitExpired); if (p.host_flag) *reinterpret_cast<volatile int*>(p.host_flag) = 1; }
  leave();
}

// The persistent kernel lists the kept channels as [definite][share of the
// threshold bin]; callers of the mask get it in ascending order.  One block:
// mark the members in a flag array, then an ordered compaction.  Off the hot path.
__global__ void __launch_bounds__(1024) mask_ascending_kernel(const int* __restrict__ sel, int k2, int F,
                                                              int* __restrict__ flags, int* __restrict__ out) {
  __shared__ unsigned long long ws[33];
  const int tid = threadIdx.x;
  for (int i = tid; i < F; i += 1024) flags[i] = 0;
  __syncthreads();
  for (int i = tid; i < k2; i += 1024) { const int j = sel[i]; if (j >= 0 && j < F) flags[j] = 1; }
  __syncthreads();
  unsigned long long run = 0;
  for (int base = 0; base < F; base += 1024) {
    const int j = base + tid;
    const unsigned long long f = (j < F && flags[j]) ? 1ull : 0ull;
    unsigned long long tot;
    const unsigned long long ex = block_scan_excl<1024>(f, ws, &tot);
    if (f && run + ex < (unsigned long long)k2) out[run + ex] = j;
    run += tot;
  }
}

}  // namespace prox
