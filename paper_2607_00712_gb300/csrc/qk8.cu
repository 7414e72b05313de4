// 8-bit queries and keys for the chunk attention (SageAttention's 8-bit Q K^T with 16-bit
// P V, which the paper cites in Sec. 3.4 for its attention kernels): e4m3 codes with one fp32
// scale per head.
//
//   head_amax_kernel + quant_heads_kernel + head_scale_kernel
//       x bf16 [n][H][d] -> codes [n][H][d], scale[h] = amax_h / 448 (1 for an all-zero head),
//       code = e4m3(x * (1 / scale_h)); the three launches run in stream order, the scale
//       array holding amax (as fp32 bits, reduced with integer atomicMax: non-negative fp32
//       values order like their bit patterns; per block in shared memory first) until the
//       last one converts it.
//   quant_q_blocks_kernel
//       queries: one scale per head and block of 128 tokens (one attention CTA), one pass.
//   quant_given_kernel
//       codes with given per-head scales (the chunk's keys with the ring's key scales).
//   append_qk8_kernel
//       appends frames to a ring whose keys are e4m3: K rows quantised with the ring's given
//       per-head scales into their slots, V rows (bf16) copied, or, for a ring whose values are e4m3
//       too, quantised d-major by further CTAs of the same launch.
//   quant_vt_kernel
//       values as d-major e4m3 codes [H][d][keys] with given per-head scales (the operand layout
//       of the 8-bit P V): the chunk's values.
// All are HBM streams of a few us, launched as programmatic dependents, with every load of a thread
// in flight before its first use.  At 4680 tokens x 12 heads x 128 (14.4 MB read, 7.2 written each, 3.2
// us at the copy rate), cold: queries 7.6 us, keys 6.4, d-major values 6.4, the append of both 11.4;
// 11.5, 7, 14 and 11 + 15 with 64-bit divisions, dependent loads and a byte-wise transpose.
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "internal.h"
#include "pdl.cuh"
#include "ptx.cuh"

namespace ispa {

namespace {

constexpr float kE4M3Max = 448.f;

__device__ __forceinline__ uint16_t e4m3x2(float x0, float x1) {   // x0 in the low byte
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(x1), "f"(x0));
  return r;
}

// 8 bf16 (one 16-byte word) times inv -> 8 codes (8 bytes)
__device__ __forceinline__ uint2 quant8(const uint4 v, float inv) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  uint32_t out[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint16_t lo = e4m3x2(__fmul_rn(__uint_as_float(w[2 * h] << 16), inv),
                               __fmul_rn(__uint_as_float(w[2 * h] & 0xFFFF0000u), inv));
    const uint16_t hi = e4m3x2(__fmul_rn(__uint_as_float(w[2 * h + 1] << 16), inv),
                               __fmul_rn(__uint_as_float(w[2 * h + 1] & 0xFFFF0000u), inv));
    out[h] = static_cast<uint32_t>(lo) | (static_cast<uint32_t>(hi) << 16);
  }
  return make_uint2(out[0], out[1]);
}

__device__ __forceinline__ float scale_of_amax(float amax) { return amax == 0.f ? 1.f : __fdiv_rn(amax, kE4M3Max); }
__device__ __forceinline__ float inv_of_scale(float s) { return __fdiv_rn(1.f, s); }

// One warp per (token, head) row of d bf16 (d % 8 == 0); amax_bits[h] must start at 0.
// Per-head maxima are gathered in shared memory (H <= kMaxHeadsSmem) and then merged into
// amax_bits with one atomic per head and block.
constexpr int kMaxHeadsSmem = 256;
__global__ void head_amax_kernel(const __nv_bfloat16* __restrict__ x, int64_t rows, int H, int d,
                                 unsigned int* __restrict__ amax_bits) {
  __shared__ unsigned int blk[kMaxHeadsSmem];
  for (int h = threadIdx.x; h < H; h += blockDim.x) blk[h] = 0u;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
  const int nw = d / 8;
  for (int64_t r = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); r < rows; r += warps) {
    const uint4* xr = reinterpret_cast<const uint4*>(x + r * d);
    float m = 0.f;
    for (int i = lane; i < nw; i += 32) {
      const uint4 v = xr[i];
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        m = fmaxf(m, fmaxf(fabsf(__uint_as_float(w[e] << 16)), fabsf(__uint_as_float(w[e] & 0xFFFF0000u))));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) atomicMax(blk + (r % H), __float_as_uint(m));
  }
  __syncthreads();
  for (int h = threadIdx.x; h < H; h += blockDim.x)
    if (blk[h]) atomicMax(amax_bits + h, blk[h]);
}

// Codes of every 16-byte word: grid-stride over n * H * d / 8 words.
__global__ void quant_heads_kernel(const uint4* __restrict__ x, int64_t n_words, int H, int d,
                                   const unsigned int* __restrict__ amax_bits, uint2* __restrict__ q) {
  const int wpr = d / 8;   // words per (token, head) row
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < n_words;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int h = static_cast<int>((i / wpr) % H);
    q[i] = quant8(x[i], inv_of_scale(scale_of_amax(__uint_as_float(amax_bits[h]))));
  }
}

__global__ void head_scale_kernel(float* __restrict__ s, int H) {
  const int h = blockIdx.x * blockDim.x + threadIdx.x;
  if (h < H) s[h] = scale_of_amax(s[h]);   // s holds amax until here
}

// Queries: one CTA per (block of 128 tokens, head); the block's rows (d / 8 16-byte words each,
// 16 WORDS words for a row at most) stay in registers between the max and the quantisation.
constexpr int QB = 128;
template <int WORDS>   // words per thread: d <= 16 WORDS
__global__ void __launch_bounds__(256) quant_q_blocks_kernel(const uint4* __restrict__ x, int64_t n, int H, int d,
                                                             uint2* __restrict__ q, float* __restrict__ scale) {
  pdl_wait();
  pdl_trigger();
  __shared__ float red[8];
  const int b = blockIdx.x, h = blockIdx.y;
  const int wpr = d / 8;
  const int64_t t0 = static_cast<int64_t>(b) * QB;
  const int rows = static_cast<int>(n - t0 < QB ? n - t0 : QB);
  const int words = rows * wpr;
  uint4 cache[WORDS];
  float m = 0.f;
#pragma unroll
  for (int c = 0; c < WORDS; ++c) {
    const int w = threadIdx.x + 256 * c;
    cache[c] = make_uint4(0, 0, 0, 0);
    if (w < words) cache[c] = x[((t0 + w / wpr) * H + h) * wpr + w % wpr];
  }
#pragma unroll
  for (int c = 0; c < WORDS; ++c) {
    const uint32_t v[4] = {cache[c].x, cache[c].y, cache[c].z, cache[c].w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      m = fmaxf(m, fmaxf(fabsf(__uint_as_float(v[e] << 16)), fabsf(__uint_as_float(v[e] & 0xFFFF0000u))));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  float amax = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) amax = fmaxf(amax, red[i]);
  const float sc = scale_of_amax(amax);
  const float inv = inv_of_scale(sc);
#pragma unroll
  for (int c = 0; c < WORDS; ++c) {
    const int w = threadIdx.x + 256 * c;
    if (w < words) q[((t0 + w / wpr) * H + h) * wpr + w % wpr] = quant8(cache[c], inv);
  }
  if (threadIdx.x == 0) scale[static_cast<int64_t>(h) * gridDim.x + b] = sc;
}

// Codes with given per-head scales: four 16-byte words a thread.  I: an index type that holds the
// word count (the divisions by the row length and the head count are 32-bit where they can be).
constexpr int G_WORDS = 4;
template <typename I>
__global__ void __launch_bounds__(256) quant_given_kernel(const uint4* __restrict__ x, I n_words, int H, int d,
                                                          const float* __restrict__ scale, uint2* __restrict__ q) {
  pdl_wait();
  pdl_trigger();
  const I wpr = d / 8;
  const I i0 = static_cast<I>(blockIdx.x) * (256 * G_WORDS) + threadIdx.x;
  uint4 v[G_WORDS];
#pragma unroll
  for (int u = 0; u < G_WORDS; ++u)
    if (i0 + 256 * u < n_words) v[u] = x[i0 + 256 * u];
#pragma unroll
  for (int u = 0; u < G_WORDS; ++u) {
    const I i = i0 + 256 * u;
    if (i < n_words) q[i] = quant8(v[u], inv_of_scale(scale[(i / wpr) % static_cast<I>(H)]));
  }
}

// d-major e4m3 values: out[h][c][key(t)] = e4m3(v[t][h][c] * (1 / scale_h)), key(t) = t, or
// slot[t / P] * P + t % P for appended frames (P % 4 == 0 keeps four tokens in one frame and their
// word aligned).  One CTA per (128 tokens, head): a thread quantises 8 channels of 4 tokens at a time and
// turns them into 8 words of one channel x 4 tokens in registers; through shared memory (word t4 of
// channel c at t4 ^ 2 (c / 8): no bank conflicts on either side) a warp then writes 128 contiguous
// bytes of a channel per store.
constexpr int VT_TOK = 128;
struct QuantVtParams {
  const uint4* v;        // bf16 [n][H][128]
  int64_t n;
  int32_t H;
  const float* scale;    // [H]
  uint8_t* out;          // [H][128][ld]
  int64_t ld;
  int32_t P, n_frames;   // n_frames == 0: key(t) = t
  int32_t slot[kMaxAppendFrames];
};

__device__ __forceinline__ void quant_vt_block(const QuantVtParams& p, int64_t t0, int h,
                                               uint32_t (*tile)[VT_TOK / 4]) {
  const int rows = static_cast<int>(p.n - t0 < VT_TOK ? p.n - t0 : VT_TOK);
  const int c8 = threadIdx.x & 15;
  uint4 x[2][4];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int t4 = (threadIdx.x >> 4) + 16 * i;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      x[i][r] = make_uint4(0, 0, 0, 0);
      if (4 * t4 + r < rows) x[i][r] = p.v[((t0 + 4 * t4 + r) * p.H + h) * 16 + c8];
    }
  }
  const float inv = inv_of_scale(p.scale[h]);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int t4 = (threadIdx.x >> 4) + 16 * i;
    uint2 q[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) q[r] = quant8(x[i][r], inv);
#pragma unroll
    for (int k = 0; k < 2; ++k) {   // 4 x 4 bytes: tokens x channels -> channels x tokens
      const uint32_t a0 = k ? q[0].y : q[0].x, a1 = k ? q[1].y : q[1].x;
      const uint32_t a2 = k ? q[2].y : q[2].x, a3 = k ? q[3].y : q[3].x;
      const uint32_t l0 = __byte_perm(a0, a1, 0x5140), l1 = __byte_perm(a2, a3, 0x5140);
      const uint32_t h0 = __byte_perm(a0, a1, 0x7362), h1 = __byte_perm(a2, a3, 0x7362);
      uint32_t* row = &tile[8 * c8 + 4 * k][t4 ^ (2 * c8)];
      row[0] = __byte_perm(l0, l1, 0x5410);
      row[VT_TOK / 4] = __byte_perm(l0, l1, 0x7632);
      row[2 * (VT_TOK / 4)] = __byte_perm(h0, h1, 0x5410);
      row[3 * (VT_TOK / 4)] = __byte_perm(h0, h1, 0x7632);
    }
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, t4 = threadIdx.x & 31;
  const int left = rows - 4 * t4;   // tokens of this lane's word that exist
  if (left <= 0) return;
  int64_t key = t0 + 4 * t4;
  if (p.n_frames > 0) {
    const int t = static_cast<int>(key), f = t / p.P;
    key = static_cast<int64_t>(p.slot[f]) * p.P + (t - f * p.P);
  }
  uint8_t* dst = p.out + (static_cast<int64_t>(h) * 128 + warp * 16) * p.ld + key;
#pragma unroll
  for (int j = 0; j < 16; ++j, dst += p.ld) {
    const int c = warp * 16 + j;
    const uint32_t w = tile[c][t4 ^ (2 * (c >> 3))];
    if (left >= 4) {
      *reinterpret_cast<uint32_t*>(dst) = w;
    } else {
      for (int i = 0; i < left; ++i) dst[i] = static_cast<uint8_t>(w >> (8 * i));
    }
  }
}

__global__ void __launch_bounds__(256) quant_vt_kernel(const __grid_constant__ QuantVtParams p) {
  __shared__ uint32_t tile[128][VT_TOK / 4];
  pdl_wait();
  pdl_trigger();
  quant_vt_block(p, static_cast<int64_t>(blockIdx.x) * VT_TOK, blockIdx.y, tile);
}

struct AppendQk8Params {
  int32_t n_frames, P, H, d;
  int32_t slot[kMaxAppendFrames];
  int64_t ring_tok;              // capacity_frames * P
  const uint4* k_src;            // bf16 [n_frames * P][H][d]
  const uint4* v_src;
  uint2* k_dst;                  // e4m3 [H][ring_tok][d]
  uint4* v_dst;                  // bf16 [H][ring_tok][d], or null: vt
  const float* k_scale;          // [H]
  int32_t k_blocks;              // CTAs of the keys; the others take blocks of vt, heads fastest
  QuantVtParams vt;
};

// Keys (and bf16 values): four 16-byte words (8 bf16) a thread.
template <typename I>
__global__ void __launch_bounds__(256) append_qk8_kernel(const __grid_constant__ AppendQk8Params p) {
  __shared__ uint32_t tile[128][VT_TOK / 4];
  pdl_wait();   // the new K / V may come from the kernel before this one, which may still read the ring
  pdl_trigger();
  if (static_cast<int>(blockIdx.x) >= p.k_blocks) {
    const int b = blockIdx.x - p.k_blocks;
    quant_vt_block(p.vt, static_cast<int64_t>(b / p.H) * VT_TOK, b % p.H, tile);
    return;
  }
  const I wpr = p.d / 8, H = p.H, P = p.P;
  const I total = static_cast<I>(p.n_frames) * P * H * wpr;
  const I i0 = static_cast<I>(blockIdx.x) * (256 * G_WORDS) + threadIdx.x;
  uint4 k[G_WORDS], v[G_WORDS];
#pragma unroll
  for (int u = 0; u < G_WORDS; ++u) {
    const I i = i0 + 256 * u;
    if (i < total) {
      k[u] = p.k_src[i];
      if (p.v_dst) v[u] = p.v_src[i];
    }
  }
#pragma unroll
  for (int u = 0; u < G_WORDS; ++u) {
    const I i = i0 + 256 * u;
    if (i >= total) break;
    const I row = i / wpr, w = i - row * wpr;      // row: token * H + head
    const I tok = row / H, h = row - tok * H;      // token of the appended frames
    const I f = tok / P;
    const int64_t dst_tok = static_cast<int64_t>(p.slot[f]) * p.P + (tok - f * P);
    const int64_t dst = (static_cast<int64_t>(h) * p.ring_tok + dst_tok) * wpr + w;
    p.k_dst[dst] = quant8(k[u], inv_of_scale(p.k_scale[h]));
    if (p.v_dst) p.v_dst[dst] = v[u];
  }
}

}  // namespace

cudaError_t launch_quant_heads(const void* x, int64_t n, int32_t H, int32_t d, uint8_t* q, float* scale,
                               cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(scale, 0, sizeof(float) * H, s);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t rows = n * H;
  const int64_t want = (rows + 7) / 8;
  const unsigned blocks = static_cast<unsigned>(want < sms * 16 ? want : sms * 16);
  head_amax_kernel<<<blocks, 256, 0, s>>>(static_cast<const __nv_bfloat16*>(x), rows, H, d,
                                           reinterpret_cast<unsigned int*>(scale));
  const int64_t words = rows * d / 8;
  const int64_t qb = (words + 255) / 256;
  quant_heads_kernel<<<static_cast<unsigned>(qb < sms * 16 ? qb : sms * 16), 256, 0, s>>>(
      static_cast<const uint4*>(x), words, H, d, reinterpret_cast<const unsigned int*>(scale),
      reinterpret_cast<uint2*>(q));
  head_scale_kernel<<<(H + 127) / 128, 128, 0, s>>>(scale, H);
  return cudaGetLastError();
}

static QuantVtParams vt_params(const void* x, int64_t n, int32_t H, const float* scale, uint8_t* out, int64_t ld,
                               int32_t P, int32_t n_frames, const int32_t* slots) {
  QuantVtParams p{};
  p.v = static_cast<const uint4*>(x);
  p.n = n;
  p.H = H;
  p.scale = scale;
  p.out = out;
  p.ld = ld;
  p.P = P;
  p.n_frames = n_frames;
  for (int f = 0; f < n_frames; ++f) p.slot[f] = slots[f];
  return p;
}

cudaError_t launch_append_qk8(const int32_t* slots, int32_t n_frames, int32_t P, int32_t H, int32_t d,
                              int64_t ring_tok, const void* k_src, const void* v_src, void* k_dst, void* v_dst,
                              const float* k_scale, const float* vt_scale, int64_t vt_ld, cudaStream_t s) {
  AppendQk8Params p{};
  p.n_frames = n_frames;
  p.P = P;
  p.H = H;
  p.d = d;
  for (int f = 0; f < n_frames; ++f) p.slot[f] = slots[f];
  p.ring_tok = ring_tok;
  p.k_src = static_cast<const uint4*>(k_src);
  p.v_src = static_cast<const uint4*>(v_src);
  p.k_dst = static_cast<uint2*>(k_dst);
  p.v_dst = vt_scale ? nullptr : static_cast<uint4*>(v_dst);
  p.k_scale = k_scale;
  const int64_t tokens = static_cast<int64_t>(n_frames) * P, total = tokens * H * d / 8;
  const int64_t kb = (total + 256 * G_WORDS - 1) / (256 * G_WORDS);
  int64_t vb = 0;
  if (vt_scale) {
    p.vt = vt_params(v_src, tokens, H, vt_scale, static_cast<uint8_t*>(v_dst), vt_ld, P, n_frames, slots);
    vb = (tokens + VT_TOK - 1) / VT_TOK * H;
  }
  if (kb + vb > INT32_MAX) return cudaErrorInvalidValue;
  p.k_blocks = static_cast<int32_t>(kb);
  const dim3 grid(static_cast<unsigned>(kb + vb));
  return total < (int64_t{1} << 31) - 1024 ? launch_pdl(append_qk8_kernel<uint32_t>, grid, dim3(256), 0, s, p)
                                           : launch_pdl(append_qk8_kernel<int64_t>, grid, dim3(256), 0, s, p);
}

cudaError_t launch_quant_vt(const void* x, int64_t n, int32_t H, const float* scale, uint8_t* out, int64_t ld,
                            cudaStream_t s) {
  const QuantVtParams p = vt_params(x, n, H, scale, out, ld, 0, 0, nullptr);
  const dim3 grid(static_cast<unsigned>((n + VT_TOK - 1) / VT_TOK), static_cast<unsigned>(H));
  return launch_pdl(quant_vt_kernel, grid, dim3(256), 0, s, p);
}

cudaError_t launch_quant_q_blocks(const void* x, int64_t n, int32_t H, int32_t d, uint8_t* q, float* scale,
                                  cudaStream_t s) {
  const dim3 grid(static_cast<unsigned>((n + QB - 1) / QB), static_cast<unsigned>(H));
  return launch_pdl(d <= 128 ? quant_q_blocks_kernel<8> : quant_q_blocks_kernel<16>, grid, dim3(256), 0, s,
                    static_cast<const uint4*>(x), n, static_cast<int>(H), static_cast<int>(d),
                    reinterpret_cast<uint2*>(q), scale);
}

cudaError_t launch_quant_given(const void* x, int64_t n, int32_t H, int32_t d, const float* scale, uint8_t* q,
                               cudaStream_t s) {
  const int64_t words = n * H * d / 8;
  const int64_t blocks = (words + 256 * G_WORDS - 1) / (256 * G_WORDS);
  if (blocks > INT32_MAX) return cudaErrorInvalidValue;
  const dim3 grid(static_cast<unsigned>(blocks));
  const uint4* xw = static_cast<const uint4*>(x);
  uint2* qw = reinterpret_cast<uint2*>(q);
  if (words < (int64_t{1} << 31) - 1024)
    return launch_pdl(quant_given_kernel<uint32_t>, grid, dim3(256), 0, s, xw, static_cast<uint32_t>(words),
                      static_cast<int>(H), static_cast<int>(d), scale, qw);
  return launch_pdl(quant_given_kernel<int64_t>, grid, dim3(256), 0, s, xw, words, static_cast<int>(H),
                    static_cast<int>(d), scale, qw);
}

}  // namespace ispa
