// Offline packer (Sec. 4.3): scales, integer codes in input-major order, channel-major copy of W_down.
//
// Packed proxy layout ("input-major"): row i (one input coordinate) holds all
// channels; it is cut into 16-byte chunks, chunk c covering CH consecutive
// channels (CH = 16 for 4-bit, 8 for 8-bit):
//   words 0,1 : gate codes of channels c*CH .. c*CH+CH-1  (lowest bits first)
//   words 2,3 : up   codes of the same channels
// Codes are offset binary: q + 8 (4-bit) or q + 128 (8-bit).
// Scale layout: [group][chunk][2][CH] fp16 (gate scales then up scales).
#pragma once

#include "prox_kernels.cuh"

namespace prox {

// scale = fp16(absmax / qmax) from the magnitude bits of a bf16
template <int BITS>
__device__ __forceinline__ __half proxy_scale(unsigned absmax_bits) {
  constexpr float qmax = (float)((1 << (BITS - 1)) - 1);
  return __float2half_rn(__fdiv_rn(__uint_as_float(absmax_bits << 16), qmax));
}

__device__ __forceinline__ unsigned absmax4(const uint2& v) {   // largest of four bf16 magnitudes, as bits
  const unsigned m = __vmaxu2(v.x & 0x7fff7fffu, v.y & 0x7fff7fffu);
  return max(m & 0xffffu, m >> 16);
}

// Bits of 1.5 * 2^23 + offset + rint(v / s) for four weights of one channel, from inv = 1 / s (s a normal fp16 number, or 0 and so v).
// v has 8 significant bits and s = m 2^b has m < 2^11, so a quotient that is not a half integer itself is at least
// 1 / (2 m) > 2^-12 away from the next one (v - (k + 1/2) s is a multiple of 2^(b-1), unless v's last bit lies below 2^(b-1): then
// |v| < 2^(b+6) and the quotient is below 1/16, nowhere near a half), and v * inv within 1e-5 of it
// (|quotient| < 128.1): rounded to a multiple of 2^-12 first (the first addition: 3072 + quotient), what is a half
// integer becomes exactly one and nothing else does, and the second addition rounds to the nearest integer, halves to even,
// as the IEEE quotient would be.  No clamp: the scale is absmax / qmax to 2^-11.  With the start of the codes at bit 0 of the
// sum's mantissa a weight takes four instructions (unpack, multiply-add, add, shift-add into the word); with the quotient's
// distance from a half taken and divisions where it was close, clamps and masks it took eleven.
template <int BITS>
__device__ __forceinline__ void proxy_sums(const uint2& v, float inv, uint32_t (&t)[4]) {
  constexpr float magic = 12582912.f + (BITS == 4 ? 8.f : 128.f), grid = 3072.f;
  const float f[4] = {bf16_lo(v.x), bf16_hi(v.x), bf16_lo(v.y), bf16_hi(v.y)};
#pragma unroll
  for (int e = 0; e < 4; e += 2)             // two at a time: one issue slot for two multiply-adds
    asm("{\n\t.reg .b64 a, b, c, d;\n\t"
        "mov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %4};\n\tmov.b64 c, {%5, %5};\n\tmov.b64 d, {%6, %6};\n\t"
        "fma.rn.f32x2 a, a, b, c;\n\tadd.rn.f32x2 a, a, d;\n\tmov.b64 {%0, %1}, a;\n\t}"
        : "=r"(t[e]), "=r"(t[e + 1]) : "f"(f[e]), "f"(f[e + 1]), "f"(inv), "f"(grid), "f"(magic - grid));
}
// The same with the quotients themselves and clamped, for scales that are not normal fp16 numbers (nothing but a code may
// get into the words, whatever the weights are).
template <int BITS>
__device__ __noinline__ uint4 proxy_sums_small(uint2 v, float s) {
  constexpr float qmax = (float)((1 << (BITS - 1)) - 1), magic = 12582912.f + (BITS == 4 ? 8.f : 128.f);
  const float f[4] = {bf16_lo(v.x), bf16_hi(v.x), bf16_lo(v.y), bf16_hi(v.y)};
  uint32_t t[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float q = s != 0.f ? __fdiv_rn(f[e], s) : 0.f;
    t[e] = __float_as_uint(fminf(fmaxf(__fadd_rn(q, magic), magic - qmax), magic + qmax));
  }
  return make_uint4(t[0], t[1], t[2], t[3]);
}

// One scale per channel row: one warp per (matrix, channel), 16-byte loads, four in flight per lane.
template <int BITS>
__global__ void __launch_bounds__(256)
proxy_row_scale_kernel(const uint16_t* __restrict__ wg, const uint16_t* __restrict__ wu, int D, int F,
                       __half* __restrict__ S, float* __restrict__ s_plain) {
  constexpr int CH = ProxyFmt<BITS>::CH;
  const int lane = threadIdx.x & 31, j = blockIdx.x * 8 + (threadIdx.x >> 5), which = blockIdx.y;
  if (j >= F) return;
  const uint4* w = reinterpret_cast<const uint4*>((which ? wu : wg) + (size_t)j * D);
  unsigned a = 0;
  const int nv = D / 8;
  for (int i0 = lane; i0 < nv; i0 += 128) {
    uint4 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) v[u] = (i0 + 32 * u < nv) ? __ldg(w + i0 + 32 * u) : make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int u = 0; u < 4; ++u)
      a = max(a, max(absmax4(make_uint2(v[u].x, v[u].y)), absmax4(make_uint2(v[u].z, v[u].w))));
  }
  a = __reduce_max_sync(0xffffffffu, a);
  if (lane == 0) {
    const __half s = proxy_scale<BITS>(a);
    S[((size_t)(j / CH) * 2 + which) * CH + j % CH] = s;
    s_plain[(size_t)which * F + j] = __half2float(s);
  }
}

// Codes (and, GROUPED, the scales of 128-input groups) of a tile of 128 inputs x 128 (4-bit) or 64 (8-bit)
// channels, both matrices.  Each weight is read once, each packed byte written once.  A warp
// takes 8 channels x 128 inputs of one matrix (eight 256-byte row pieces, 8 bytes per lane each), which give a
// lane one word (4-bit) or two (8-bit) per input row of the packed layout; they meet in shared memory
// (word column xor lane: no bank conflicts either way) and leave as whole 128-byte pieces of the packed rows.
// Bound by instruction issue (2.7 instructions per clock and SM) and the loads in flight: 4096 x 12288, 4-bit, groups: 50 us
// (200 MB of weights and 50 MB of codes are 39 us of HBM); 82 with eleven instructions per weight (see proxy_sums), 55 with
// single multiply-adds and a branch per channel, 52 with four blocks per SM instead of five; with the next task's rows
// requested before one is worked on (80 registers) 54.  One scale per row: the scales are 34 us in front.  (The W_down copy is 31
// us; running its blocks between the packing ones in one launch was slower, its small blocks want more of them per SM.)
template <int BITS, bool GROUPED>
__global__ void __launch_bounds__(256, 5)
proxy_pack_kernel(const uint16_t* __restrict__ wg, const uint16_t* __restrict__ wu, int D, int F,
                  __half* __restrict__ S, float* __restrict__ s_plain, uint32_t* __restrict__ P) {
  constexpr int CH = ProxyFmt<BITS>::CH;
  constexpr int TILE = BITS == 4 ? 128 : 64;          // channels of a tile: 128 bytes of a packed row
  constexpr int NTASK = TILE / 8 * 2;
  __shared__ uint32_t out[128 * 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c0 = blockIdx.x * TILE, g = blockIdx.y, nchunks = F / CH, ngroups = GROUPED ? D / 128 : 1;
  for (int task = warp; task < NTASK; task += 8) {
    const int which = task & 1, grp = task >> 1, j0 = c0 + grp * 8;
    if (j0 >= F) continue;
    const uint16_t* w = (which ? wu : wg) + (size_t)j0 * D + (size_t)g * 128 + lane * 4;
    uint2 v[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) v[m] = __ldg(reinterpret_cast<const uint2*>(w + (size_t)m * D));
    uint32_t lo[4] = {0u, 0u, 0u, 0u}, hi[4] = {0u, 0u, 0u, 0u};
    // lane m (of every eight) makes the scale of channel m and its reciprocal for all
    float s_mine, inv_mine;
    if (GROUPED) {
      unsigned a_mine = 0;
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const unsigned a = __reduce_max_sync(0xffffffffu, absmax4(v[m]));
        if ((lane & 7) == m) a_mine = a;
      }
      const __half h = proxy_scale<BITS>(a_mine);
      s_mine = __half2float(h);
      if (lane < 8) {
        S[(((size_t)g * nchunks + j0 / CH) * 2 + which) * CH + j0 % CH + lane] = h;
        s_plain[((size_t)which * F + j0 + lane) * ngroups + g] = s_mine;
      }
    } else {
      s_mine = s_plain[(size_t)which * F + j0 + (lane & 7)];
    }
    inv_mine = s_mine != 0.f ? __fdiv_rn(1.0f, s_mine) : 0.f;     // scale 0: every code is 0
    // the codes' words as sums of what stands in the low bits of the sums above, whose upper bits add up to a constant
    auto add = [&](int m, const uint32_t (&t)[4]) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (BITS == 4) lo[e] += t[e] << (4 * m);
        else if (m < 4) lo[e] += t[e] << (8 * m);
        else hi[e] += t[e] << (8 * (m - 4));
      }
    };
    if (!__any_sync(0xffffffffu, (s_mine > 0.f && s_mine < 6.103515625e-5f) || !(s_mine <= 65504.f))) {
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        uint32_t t[4];
        proxy_sums<BITS>(v[m], __shfl_sync(0xffffffffu, inv_mine, m), t);
        add(m, t);
      }
    } else {
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const uint4 u = proxy_sums_small<BITS>(v[m], __shfl_sync(0xffffffffu, s_mine, m));
        const uint32_t t[4] = {u.x, u.y, u.z, u.w};
        add(m, t);
      }
    }
    constexpr uint32_t kUpper = BITS == 4 ? 0x4b400000u + 0xb4000000u + 0x40000000u : 0x4b400000u + 0x40000000u;
#pragma unroll
    for (int e = 0; e < 4; ++e) { lo[e] -= kUpper; hi[e] -= kUpper; }
    // word of the row: chunk * 4 + which * 2 + (half of the chunk's channels)
    const int col = BITS == 4 ? (grp >> 1) * 4 + which * 2 + (grp & 1) : grp * 4 + which * 2;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      out[(lane * 4 + e) * 32 + (col ^ lane)] = lo[e];
      if (BITS == 8) out[(lane * 4 + e) * 32 + ((col + 1) ^ lane)] = hi[e];
    }
  }
  __syncthreads();
  const int words_per_row = nchunks * 4, w0 = blockIdx.x * 32;
  if (w0 + lane < words_per_row) {
#pragma unroll 4
    for (int i = warp; i < 128; i += 8)
      P[(size_t)(g * 128 + i) * words_per_row + w0 + lane] = out[i * 32 + (lane ^ (i >> 2))];
  }
}

// 16-bit "proxies" (ablation A1 of Sec. "Ablation Studies"; also the 16-bit input-sparse GEMV that
// the cost ratio alpha of Sec. 4.2 is measured against): the original bf16 weights in the proxies'
// input-major order.  A 16-byte chunk of row i holds 4 channels: words 0,1 gate, words 2,3 up.
// One thread per 32-bit word (two channels of one matrix).
__global__ void proxy_pack16_kernel(const uint16_t* __restrict__ wg, const uint16_t* __restrict__ wu,
                                    int D, int F, uint32_t* __restrict__ P) {
  const long long words_per_row = (long long)(F / 4) * 4;
  const long long tid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tid >= words_per_row * D) return;
  const int i = (int)(tid % D);                    // consecutive threads: consecutive inputs (coalesced reads)
  const long long wword = tid / D;
  const int chunk = (int)(wword >> 2), word = (int)(wword & 3);
  const uint16_t* w = (word >> 1) ? wu : wg;
  const int j0 = chunk * 4 + (word & 1) * 2;
  P[(size_t)i * words_per_row + wword] =
      (uint32_t)w[(size_t)j0 * D + i] | ((uint32_t)w[(size_t)(j0 + 1) * D + i] << 16);
}

// W_down [D, F] -> channel-major [F, D]  (Sec. 3.1: y = sum_j s_j W_down[j,:]).  64 x 64 tiles (D % 128 == 0,
// F % 64 == 0), 16-byte loads and stores of whole 128-byte pieces on both sides; a thread turns 8 rows x 2
// columns around with byte permutes.  The 16-byte columns of row d are xor-ed with d / 8: both sides of the
// shared tile are free of bank conflicts.  Bound by HBM: 31 us for the 201 MB of a 4096 x 12288 layer, 6.4 TB/s.
__global__ void __launch_bounds__(256)
transpose_bf16_kernel(const uint16_t* __restrict__ in, uint16_t* __restrict__ out, int rows, int cols) {
  __shared__ __align__(16) uint32_t tile[64 * 32];
  const int t = threadIdx.x, c0 = blockIdx.x * 64, r0 = blockIdx.y * 64;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int r = (t >> 3) + 32 * k, v = t & 7;
    *reinterpret_cast<uint4*>(&tile[r * 32 + ((v ^ (r >> 3)) << 2)]) =
        __ldg(reinterpret_cast<const uint4*>(in + (size_t)(r0 + r) * cols + c0) + v);
  }
  __syncthreads();
  const int dv = t & 7, fp = t >> 3;                 // rows dv*8 .. dv*8+7, columns 2 fp and 2 fp + 1
  uint32_t w[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) w[e] = tile[(dv * 8 + e) * 32 + (fp ^ (dv << 2))];
  uint4 a, b;
  a.x = __byte_perm(w[0], w[1], 0x5410); a.y = __byte_perm(w[2], w[3], 0x5410);
  a.z = __byte_perm(w[4], w[5], 0x5410); a.w = __byte_perm(w[6], w[7], 0x5410);
  b.x = __byte_perm(w[0], w[1], 0x7632); b.y = __byte_perm(w[2], w[3], 0x7632);
  b.z = __byte_perm(w[4], w[5], 0x7632); b.w = __byte_perm(w[6], w[7], 0x7632);
  uint16_t* o = out + (size_t)(c0 + 2 * fp) * rows + r0 + dv * 8;
  *reinterpret_cast<uint4*>(o) = a;
  *reinterpret_cast<uint4*>(o + rows) = b;
}

}  // namespace prox
