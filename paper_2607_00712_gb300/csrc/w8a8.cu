// W8A8 output projection on W + dW (Sec. 4, post-training quantisation; Sec. 3.2 for the
// injected weight): 8-bit e4m3 activations and weights on the tensor cores
// (tcgen05 kind::f8f6f4, fp32 accumulators in TMEM).
//
//   quant_rows_kernel    activations [T][D] bf16 -> e4m3 codes [T][D] + one fp32 scale per token
//   col_amax_kernel,     W (+ dW) fp32 [D][D_out] -> e4m3 codes [D_out][D] (K-major, i.e. the
//   quant_wt_kernel,     layout of a torch Linear weight) + one fp32 scale per output channel
//   col_scale_kernel
//   w8a8_gemm_kernel     out[t][n] = bf16(a_scale[t] * w_scale[n] * sum_k a[t][k] w[n][k])
//
// Quantisation arithmetic (fp32, rounded to nearest at every step, identical to the
// oracle's): amax = max |x|; inv = 448 / amax, scale = amax / 448 (both 1 for an all-zero
// group); code = e4m3(x * inv), round to nearest even with saturation at +-448.
//
// GEMM: persistent, one CTA per SM looping over 128 x BN output tiles (BN = 256, 192 or 128), or one pair of
// CTAs over 256 x 256 tiles (cta_group::2), whichever gives the shortest estimated run; both operands
// K-major with 128-byte swizzle (one 128-byte row = 128 codes = four K=32 UMMA steps), a
// 4-stage TMA ring (6 in a pair) that runs on across tile boundaries, two accumulator sets in TMEM so that
// the epilogue of one tile (both scales, bf16 store) overlaps the UMMAs of the next; with
// 128-column tiles each set has two accumulation chains that the k-steps alternate between.
// Warp 0 issues TMA, warp 1 allocates TMEM and issues UMMAs, warps 2-9 drain TMEM (warp w
// reads lanes 32 (w % 4) .. +31 and half of the columns), give the set back at once, and store
// through 32 x 32 blocks in shared memory and TMA.  (Stores from registers, a lane a row, were 32 cache lines an
// instruction: 64 KB of a tile took 2 us that nothing hid after a CTA's last tile and that slowed the others.)
// 4680 x 1536 -> 1536: 15.0 -> 11.5 us, -> 4608: 32.7 -> 24.8 us; 4680 x 5120 -> 5120: 79.6 -> 68.0 us (3.6
// PFLOP/s).  Every wait is bounded.
#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>

#include "internal.h"
#include "pdl.cuh"
#include "ptx.cuh"

namespace ispa {

namespace {

constexpr float kE4M3Max = 448.f;

// Two fp32 values -> two e4m3 codes (round to nearest even, saturating), x0 in the low byte.
__device__ __forceinline__ uint16_t e4m3x2(float x0, float x1) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(x1), "f"(x0));
  return r;
}

// One warp per row (grid-stride over rows); cols % 8 == 0.  Rows of up to 32 * CACHE
// 16-byte words (8 bf16 each) stay in registers between the max and the quantisation pass;
// of longer rows the rest is read twice.
template <int CACHE>
__global__ void __launch_bounds__(256, CACHE <= 4 ? 5 : CACHE <= 6 ? 4 : CACHE <= 8 ? 3 : 2)
    quant_rows_kernel(const __nv_bfloat16* __restrict__ x, int64_t rows, int cols, uint8_t* __restrict__ q,
                      float* __restrict__ scale) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x & 31;
  const int nw = cols / 8;   // 16-byte words of bf16 per row
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (blockDim.x >> 5);
  for (int64_t r = static_cast<int64_t>(blockIdx.x) * (blockDim.x >> 5) + (threadIdx.x >> 5); r < rows; r += warps) {
    const uint4* xr = reinterpret_cast<const uint4*>(x + r * cols);
    uint4 cache[CACHE];
    float amax = 0.f;
#pragma unroll
    for (int c = 0; c < CACHE; ++c) {
      const int i = lane + 32 * c;
      cache[c] = i < nw ? xr[i] : make_uint4(0, 0, 0, 0);
    }
    for (int i = lane + 32 * CACHE; i < nw; i += 32) {
      const uint4 v = xr[i];
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        amax = fmaxf(amax, fmaxf(fabsf(__uint_as_float(w[e] << 16)), fabsf(__uint_as_float(w[e] & 0xFFFF0000u))));
    }
#pragma unroll
    for (int c = 0; c < CACHE; ++c) {
      const uint32_t w[4] = {cache[c].x, cache[c].y, cache[c].z, cache[c].w};
#pragma unroll
      for (int e = 0; e < 4; ++e)
        amax = fmaxf(amax, fmaxf(fabsf(__uint_as_float(w[e] << 16)), fabsf(__uint_as_float(w[e] & 0xFFFF0000u))));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    const float inv = amax == 0.f ? 1.f : __fdiv_rn(kE4M3Max, amax);
    uint2* qr = reinterpret_cast<uint2*>(q + r * cols);
    auto quant8 = [&](const uint4& v) {
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
    };
#pragma unroll
    for (int c = 0; c < CACHE; ++c) {
      const int i = lane + 32 * c;
      if (i < nw) qr[i] = quant8(cache[c]);
    }
    for (int i = lane + 32 * CACHE; i < nw; i += 32) qr[i] = quant8(xr[i]);
    if (lane == 0) scale[r] = amax == 0.f ? 1.f : __fdiv_rn(amax, kE4M3Max);
  }
}

__device__ __forceinline__ float w_plus_dw(const float* W, const float* dW, int64_t i) {
  return dW ? __fadd_rn(W[i], dW[i]) : W[i];
}

// Per-column max |W + dW| into amax[D_out].  Block (32, 8) per 32 columns.
__global__ void col_amax_kernel(const float* __restrict__ W, const float* __restrict__ dW, int D, int Dout,
                                float* __restrict__ amax) {
  __shared__ float red[8][33];
  const int n = blockIdx.x * 32 + threadIdx.x;
  float m = 0.f;
  if (n < Dout)
    for (int k = threadIdx.y; k < D; k += 8) m = fmaxf(m, fabsf(w_plus_dw(W, dW, static_cast<int64_t>(k) * Dout + n)));
  red[threadIdx.y][threadIdx.x] = m;
  __syncthreads();
  if (threadIdx.y == 0 && n < Dout) {
#pragma unroll
    for (int i = 1; i < 8; ++i) m = fmaxf(m, red[i][threadIdx.x]);
    amax[n] = m;
  }
}

// codes[n][k] = e4m3((W + dW)[k][n] * inv_n) through a 32 x 32 shared-memory transpose.
// Block (32, 8); grid (ceil(D / 32), ceil(Dout / 32)).
__global__ void quant_wt_kernel(const float* __restrict__ W, const float* __restrict__ dW, int D, int Dout,
                                const float* __restrict__ amax, uint8_t* __restrict__ q_t) {
  __shared__ uint8_t tile[32][36];
  const int k0 = blockIdx.x * 32, n0 = blockIdx.y * 32;
  const int n = n0 + threadIdx.x;
  const float am = n < Dout ? amax[n] : 0.f;
  const float inv = am == 0.f ? 1.f : __fdiv_rn(kE4M3Max, am);
  for (int j = threadIdx.y; j < 32; j += 8) {
    const int k = k0 + j;
    uint8_t c = 0;
    if (k < D && n < Dout) {
      const float v = __fmul_rn(w_plus_dw(W, dW, static_cast<int64_t>(k) * Dout + n), inv);
      c = static_cast<uint8_t>(e4m3x2(v, 0.f) & 0xFF);
    }
    tile[j][threadIdx.x] = c;   // [k][n]
  }
  __syncthreads();
  for (int j = threadIdx.y; j < 32; j += 8) {
    const int nn = n0 + j, k = k0 + threadIdx.x;
    if (nn < Dout && k < D) q_t[static_cast<int64_t>(nn) * D + k] = tile[threadIdx.x][j];
  }
}

__global__ void col_scale_kernel(float* __restrict__ s, int Dout) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n < Dout) s[n] = s[n] == 0.f ? 1.f : __fdiv_rn(s[n], kE4M3Max);
}

// ------------------------------------------------------------ GEMM
constexpr int QM = 128;        // output rows (tokens) per tile
constexpr int QK = 128;        // K (bytes = codes) per stage: one 128-byte swizzled row
constexpr int Q_EPI = 8;         // read-back warps: two per TMEM lane quarter, half of the columns each
constexpr int Q_BLOCK = 32 * 64;
constexpr int Q_THREADS = 64 + 32 * Q_EPI;
constexpr uint64_t Q_DRAIN_NS = 200ull * 1000 * 1000;

template <int BN, bool PAIR>
struct QCfg {
  // Persistent: one CTA per SM loops over output tiles.  Two accumulator sets in TMEM let the
  // epilogue of one tile overlap the UMMAs of the next; with 128-column tiles each set holds
  // two accumulation chains (k-steps alternate between them), with 192- and 256-column tiles one.
  static_assert(BN == 128 || BN == 192 || BN == 256, "tile width");
  static constexpr int CHAINS = BN == 128 ? 2 : 1;
  static constexpr int SET = CHAINS * BN;         // TMEM columns per accumulator set
  static constexpr int QST = PAIR ? 6 : 4;
  static constexpr int CTAS = PAIR ? 2 : 1;
  static constexpr int BR = BN / CTAS;            // this CTA's rows of B
  static constexpr int A_BYTES = QM * QK;         // 16 KB
  static constexpr int B_BYTES = BR * QK;         // 32, 24 or 16 KB, half of that in a pair
  static constexpr int STAGE = A_BYTES + B_BYTES;
  static constexpr int OFF_OUT = QST * STAGE;     // two blocks of 32 x 32 bf16 per read-back warp
  static constexpr int OFF_BAR = OFF_OUT + Q_EPI * 2 * Q_BLOCK;
  static constexpr int N_BAR = 2 * QST + 4 + 1;   // full/empty per stage, set full/empty x2, drain
  static constexpr int SMEM = OFF_BAR + N_BAR * 8 + 16;
  // more than half of an SM's shared memory: one CTA per SM, so the 512-column TMEM
  // allocation never waits for another CTA
  static_assert(SMEM > 116 * 1024 && SMEM <= 232448 && STAGE % 1024 == 0, "shared memory layout");
  static constexpr uint32_t IDESC = idesc_e4m3(QM * CTAS, BN);
  static constexpr uint32_t TMEM_COLS = 512;      // the allocation (a power of two)
  static_assert(2 * SET <= 512, "two accumulator sets fit in TMEM");
};

struct GemmParams {
  int32_t T, D, Dout, n_kb;
  int32_t n_mt, n_tiles;   // row tiles (of 256 rows for pairs); all tiles (tile t: rows (t % n_mt), columns (t / n_mt))
  int32_t split;           // CTAs that share a tile's k-blocks (SPLIT)
  const float* a_scale;
  const float* w_scale;
  __nv_bfloat16* out;
  int* status;
  uint64_t wait_limit_ns;
};

template <int BN, bool PAIR, bool SPLIT>
__global__ void __launch_bounds__(Q_THREADS, 1)
    w8a8_gemm_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_w,
                     const __grid_constant__ CUtensorMap tm_out, const GemmParams p) {
  using C = QCfg<BN, PAIR>;
  constexpr int QST = C::QST;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = smem_raw;
  const uint32_t sbase = smem_u32(smem);
  if (sbase & 1023u) {
    if (threadIdx.x == 0) record_error(p.status, DEVERR_LAYOUT, 0, sbase, 0, 2);
    return;
  }
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::OFF_BAR);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + C::N_BAR);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  uint32_t* issued = tmem_slot + 2;   // PAIR: k-blocks loaded by this CTA's producer; the other CTA's word
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * QST, accf0 = empty0 + 8 * QST,
                 acce0 = accf0 + 16, drain_bar = acce0 + 16;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = PAIR ? static_cast<int>(cluster_ctarank()) : 0;
  // one CTA, pair or (SPLIT) cluster per output tile
  const int ctas = SPLIT ? p.split : C::CTAS, unit = blockIdx.x / ctas, units = gridDim.x / ctas;
  // this CTA's k-blocks: of a split tile its share, else all
  const int part = SPLIT ? static_cast<int>(cluster_ctarank()) : 0;
  const int kb0 = SPLIT ? p.n_kb * part / p.split : 0, kb1 = SPLIT ? p.n_kb * (part + 1) / p.split : p.n_kb;
  // A pair's rank 0 issues the UMMAs: its full barriers count both CTAs' bytes, its set-empty barriers both
  // CTAs' epilogue warps.  The stage-empty, set-full and drain barriers are each CTA's own,
  // arrived at by commits that go to both.

  if (threadIdx.x == 0) {
    for (int i = 0; i < QST; ++i) {
      mbar_init(full0 + 8 * i, 1);
      mbar_init(empty0 + 8 * i, 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(accf0 + 8 * i, 1);
      mbar_init(acce0 + 8 * i, Q_EPI * C::CTAS);
    }
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if constexpr (PAIR) cluster_sync();   // both CTAs run and their barriers exist
  if (warp == 1) {
    if constexpr (PAIR) {
      tmem_alloc_pair(smem_u32(tmem_slot), C::TMEM_COLS);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(smem_u32(tmem_slot), C::TMEM_COLS);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();   // the codes and scales may come from the kernel before this one
  pdl_trigger();
  const WaitCtx wc{abort_flag, p.status, p.wait_limit_ns};
  auto commit = [](uint32_t bar) {
    if constexpr (PAIR) tc_commit_pair(bar);
    else tc_commit(bar);
  };

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      int g = 0;   // k-blocks issued over all tiles of this CTA
      bool ok = true;
      for (int t = unit; ok && t < p.n_tiles; t += units) {
        const int m0 = ((t % p.n_mt) * C::CTAS + rank) * QM, n0 = (t / p.n_mt) * BN;
        for (int kb = kb0; kb < kb1; ++kb, ++g) {
          const int st = g % QST;
          if (!mbar_wait(empty0 + 8 * st, ((g / QST) & 1) ^ 1, wc, 31, g)) {
            ok = false;
            break;
          }
          if (rank == 0) mbar_arrive_expect_tx(full0 + 8 * st, C::CTAS * C::STAGE);
          const uint32_t sa = sbase + st * C::STAGE;
          if constexpr (PAIR) {
            const uint32_t bar = cluster_map(full0 + 8 * st, 0);
            tma_load_2d_pair(sa, &tm_a, bar, kb * QK, m0);
            tma_load_2d_pair(sa + C::A_BYTES, &tm_w, bar, kb * QK, n0 + rank * C::BR);
          } else {
            tma_load_2d(sa, &tm_a, full0 + 8 * st, kb * QK, m0);
            tma_load_2d(sa + C::A_BYTES, &tm_w, full0 + 8 * st, kb * QK, n0);
          }
        }
      }
      if constexpr (PAIR) {
        issued[0] = static_cast<uint32_t>(g);   // a pair drains at its end
      } else {
        for (int i = g > QST ? g - QST : 0; i < g; ++i)
          mbar_wait_drain(full0 + 8 * (i % QST), (i / QST) & 1, Q_DRAIN_NS);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ UMMA issuer
    if (lane == 0 && rank == 0) {
      int g = 0, i = 0;
      bool ok = true;
      for (int t = unit; ok && t < p.n_tiles; t += units, ++i) {
        const int set = i & 1;
        // the epilogue has drained this set's previous tile (tile i - 2)
        if (!mbar_wait(acce0 + 8 * set, ((i >> 1) & 1) ^ 1, wc, 34, i)) break;
        tc_fence_after();
        const uint32_t acc = tmem + set * C::SET;
        for (int kb = kb0; kb < kb1; ++kb, ++g) {
          const int st = g % QST;
          if (!mbar_wait(full0 + 8 * st, (g / QST) & 1, wc, 32, g)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = sbase + st * C::STAGE, sb = sa + C::A_BYTES;
          // four K=32 steps inside the 128-byte swizzle row (alternating chains for BN 128)
#pragma unroll
          for (int k = 0; k < QK / 32; ++k) {
            const uint32_t d = acc + (C::CHAINS == 2 ? (k & 1) * BN : 0), more = (kb > kb0 || k >= C::CHAINS) ? 1u : 0u;
            const uint64_t da = sw128_desc(sa + 32 * k, 16, 1024), db = sw128_desc(sb + 32 * k, 16, 1024);
            if constexpr (PAIR) umma_f8_pair(d, da, db, C::IDESC, more);
            else umma_f8(d, da, db, C::IDESC, more);
          }
          commit(empty0 + 8 * st);
        }
        if (!ok) break;
        commit(accf0 + 8 * set);
      }
      commit(drain_bar);
    }
    if (lane == 0) mbar_wait_drain(drain_bar, 0, rank == 0 ? Q_DRAIN_NS : p.wait_limit_ns + 2 * Q_DRAIN_NS);
    __syncwarp();
  } else {
    // ------------------------------------------------------------ epilogue (warps 2-9)
    constexpr int HC = BN / 64;   // 32-column chunks of this warp's half
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    uint8_t* block = smem + C::OFF_OUT + (warp - 2) * 2 * Q_BLOCK;
    int first = 0;   // block of the tile's first store: they alternate on across tiles, also when a tile has three
    int i = 0;
    for (int t = unit; t < p.n_tiles; t += units, ++i) {
      const int set = i & 1;
      const int m0 = ((t % p.n_mt) * C::CTAS + rank) * QM, n0 = (t / p.n_mt) * BN + half * (BN / 2);
      const int row = m0 + quarter * 32 + lane;
      // the scales are here before the sums are
      const float sa = row < p.T ? p.a_scale[row] : 0.f;
      float sw[HC];   // of column 32 c + lane
#pragma unroll
      for (int c = 0; c < HC; ++c) sw[c] = p.w_scale[n0 + 32 * c + lane];
      if (!__all_sync(0xffffffffu, mbar_wait(accf0 + 8 * set, (i >> 1) & 1, wc, 33, i))) break;
      tc_fence_after();
      const uint32_t taddr = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + set * C::SET + half * (BN / 2);
      // all loads out together, then the set goes back at once
      uint32_t v[C::CHAINS * HC][32];
#pragma unroll
      for (int c = 0; c < HC; ++c) {
        tmem_ld32(taddr + 32 * c, v[c]);
        if constexpr (C::CHAINS == 2) tmem_ld32(taddr + BN + 32 * c, v[HC + c]);
      }
#pragma unroll
      for (int c = 0; c < C::CHAINS * HC; ++c) tmem_wait_ld32(v[c]);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if constexpr (PAIR) mbar_arrive_cluster(cluster_map(acce0 + 8 * set, 0));
        else mbar_arrive(acce0 + 8 * set);
      }
      if constexpr (SPLIT) {
        // the partial sums into the stages, which have been read: 16-byte word q of row r at q ^ (r & 7)
        float4* x = reinterpret_cast<float4*>(smem) + (quarter * 32 + lane) * (BN / 4);
#pragma unroll
        for (int c = 0; c < HC; ++c)
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            float s4[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              s4[e] = __uint_as_float(v[c][4 * q + e]);
              if constexpr (C::CHAINS == 2) s4[e] += __uint_as_float(v[HC + c][4 * q + e]);
            }
            x[(half * (BN / 8) + 8 * c + q) ^ (lane & 7)] = make_float4(s4[0], s4[1], s4[2], s4[3]);
          }
        break;   // a split tile's CTA has no other
      }
      if (m0 + quarter * 32 >= p.T) continue;   // uniform over the warp; rows past T inside the block are clipped
#pragma unroll
      for (int c = 0; c < HC; ++c) {
        uint8_t* b = block + ((first + c) & 1) * Q_BLOCK;
        if (lane == 0) bulk_wait_read<1>();   // the store before last, this block's last, has read it
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint32_t pk[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float s0 = __uint_as_float(v[c][8 * q + 2 * e]), s1 = __uint_as_float(v[c][8 * q + 2 * e + 1]);
            if constexpr (C::CHAINS == 2) {
              s0 += __uint_as_float(v[HC + c][8 * q + 2 * e]);
              s1 += __uint_as_float(v[HC + c][8 * q + 2 * e + 1]);
            }
            pk[e] = pack_bf16x2(__fmul_rn(__fmul_rn(s0, sa), __shfl_sync(0xffffffffu, sw[c], 8 * q + 2 * e)),
                                __fmul_rn(__fmul_rn(s1, sa), __shfl_sync(0xffffffffu, sw[c], 8 * q + 2 * e + 1)));
          }
          // 64-byte swizzle: 16-byte word q of row r at word q ^ (r / 2 mod 4)
          *reinterpret_cast<uint4*>(b + lane * 64 + (q ^ ((lane >> 1) & 3)) * 16) =
              make_uint4(pk[0], pk[1], pk[2], pk[3]);
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          tma_store_2d(&tm_out, smem_u32(b), n0 + 32 * c, m0 + quarter * 32);
          bulk_commit_group();
        }
      }
      first ^= HC & 1;
    }
    if (lane == 0) bulk_wait_all();
    __syncwarp();
  }

  tc_fence_before();
  __syncthreads();
  if constexpr (SPLIT) {
    cluster_sync();   // every CTA's partial sums are in its shared memory
    static_assert(!SPLIT || BN == 128, "a row is four columns a lane");
    const int m0 = unit % p.n_mt * QM, n0 = unit / p.n_mt * BN + 4 * lane;
    const float4 sw = *reinterpret_cast<const float4*>(p.w_scale + n0);
    // one warp per row of this CTA's share
    for (int r = QM * part / p.split + warp; r < QM * (part + 1) / p.split && m0 + r < p.T; r += Q_THREADS / 32) {
      const uint32_t x = sbase + (r * (BN / 4) + (lane ^ (r & 7))) * 16;
      float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int i = 0; i < p.split; ++i) {
        const float4 v = cluster_ld4(cluster_map(x, i));
        o.x += v.x;
        o.y += v.y;
        o.z += v.z;
        o.w += v.w;
      }
      const float sa = p.a_scale[m0 + r];
      *reinterpret_cast<uint2*>(p.out + static_cast<size_t>(m0 + r) * p.Dout + n0) =
          make_uint2(pack_bf16x2(__fmul_rn(__fmul_rn(o.x, sa), sw.x), __fmul_rn(__fmul_rn(o.y, sa), sw.y)),
                     pack_bf16x2(__fmul_rn(__fmul_rn(o.z, sa), sw.z), __fmul_rn(__fmul_rn(o.w, sa), sw.w)));
    }
    cluster_sync();   // no CTA leaves while another still reads its shared memory
  }
  if constexpr (PAIR) {
    // Without a timeout rank 0's UMMA thread has waited for every load.  After one the two producers may have
    // stopped at different k-blocks, and rank 1's loads count on rank 0's barriers: the CTAs tell each other how far
    // they got, rank 0 waits for what is in flight, and neither leaves before that.
    constexpr uint32_t kAborted = 1u << 31;
    const uint32_t mine = issued[0] | (*abort_flag ? kAborted : 0u);
    if (threadIdx.x == 0) cluster_st1(cluster_map(smem_u32(issued + 1), rank ^ 1), mine);
    cluster_sync();   // neither CTA's TMEM, barriers or shared memory is used by the other's roles any more
    const uint32_t other = issued[1];
    if ((mine | other) & kAborted) {
      if (rank == 0 && threadIdx.x == 0) {
        const int g0 = static_cast<int>(mine & ~kAborted), g1 = static_cast<int>(other & ~kAborted), g = max(g0, g1);
        for (int i = max(g - QST, 0); i < g; ++i) {   // the last round of every stage
          const uint32_t bar = full0 + 8 * (i % QST);
          if (i >= g0) mbar_arrive_expect_tx(bar, C::STAGE);   // rank 1's half only
          if (i >= g1) mbar_complete_tx(bar, C::STAGE);        // rank 1's half was never asked for
          mbar_wait_drain(bar, (i / QST) & 1, Q_DRAIN_NS);
        }
      }
      cluster_sync();
    }
  }
  if (warp == 1) {
    tc_fence_after();
    if constexpr (PAIR) tmem_dealloc_pair(tmem, C::TMEM_COLS);
    else tmem_dealloc(tmem, C::TMEM_COLS);
  }
}

template <int BN, bool PAIR, bool SPLIT = false>
cudaError_t launch_gemm_bn(int split, const uint8_t* a_q, const float* a_scale, const uint8_t* w_q,
                           const float* w_scale, int32_t T, int32_t D, int32_t Dout, __nv_bfloat16* out, int* status,
                           uint64_t wait_limit_ns, cudaStream_t s) {
  using C = QCfg<BN, PAIR>;
  int dev = 0;
  cudaGetDevice(&dev);
  {
    const cudaError_t e =
        set_smem_limit_once(reinterpret_cast<const void*>(w8a8_gemm_kernel<BN, PAIR, SPLIT>), C::SMEM);
    if (e != cudaSuccess) return e;
  }
  CUtensorMap ta, tw, to;
  if (!encode_tmap_2d_u8(&ta, a_q, D, T, D, QK, QM) || !encode_tmap_2d_u8(&tw, w_q, D, Dout, D, QK, C::BR) ||
      !encode_tmap_2d_sw64(&to, out, Dout, T, 2 * static_cast<uint64_t>(Dout), 32, 32))
    return cudaErrorInvalidValue;
  GemmParams p;
  p.T = T;
  p.D = D;
  p.Dout = Dout;
  p.n_kb = D / QK;
  p.split = split;
  p.out = out;
  p.n_mt = (T + QM * C::CTAS - 1) / (QM * C::CTAS);
  p.n_tiles = p.n_mt * (Dout / BN);
  p.a_scale = a_scale;
  p.w_scale = w_scale;
  p.status = status;
  p.wait_limit_ns = wait_limit_ns;
  int dev_sms = 152;
  cudaDeviceGetAttribute(&dev_sms, cudaDevAttrMultiProcessorCount, dev);
  const int ctas = SPLIT ? split : C::CTAS, units = SPLIT ? p.n_tiles : std::min(p.n_tiles, dev_sms / ctas);
  return launch_pdl_cluster(w8a8_gemm_kernel<BN, PAIR, SPLIT>, dim3(units * ctas), dim3(Q_THREADS), C::SMEM, ctas, s,
                            ta, tw, to, p);
}

}  // namespace

cudaError_t launch_quant_rows(const void* x, int64_t rows, int32_t cols, uint8_t* q, float* scale, cudaStream_t s) {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t want = (rows + 7) / 8;   // one warp per row, 8 warps per block
  const int64_t blocks = want < static_cast<int64_t>(sms) * 16 ? want : static_cast<int64_t>(sms) * 16;
  // No more registers than the row needs: latency bounds this kernel, and with fewer of them all rows are in flight
  // at once.  4680 x 1536: 4.4 -> 3.2 us, 9400 x 1024: 7.0 -> 4.0 (against 12 words a lane for every row).  Rows of
  // more than 3072 values keep 12 and read the rest twice: with 20 only 8 warps a SM fit, 8.1 -> 10.2 us at 5120.
  const int words = (cols / 8 + 31) / 32;
  const auto kernel = words <= 4   ? quant_rows_kernel<4>
                      : words <= 6 ? quant_rows_kernel<6>
                      : words <= 8 ? quant_rows_kernel<8>
                                   : quant_rows_kernel<12>;
  return launch_pdl(kernel, dim3(static_cast<unsigned>(blocks)), dim3(256), 0, s,
                    static_cast<const __nv_bfloat16*>(x), rows, static_cast<int>(cols), q, scale);
}

cudaError_t launch_quant_weight(const float* W, const float* dW, int32_t D, int32_t Dout, uint8_t* q_t, float* scale,
                                cudaStream_t s) {
  col_amax_kernel<<<(Dout + 31) / 32, dim3(32, 8), 0, s>>>(W, dW, D, Dout, scale);
  quant_wt_kernel<<<dim3((D + 31) / 32, (Dout + 31) / 32), dim3(32, 8), 0, s>>>(W, dW, D, Dout, scale, q_t);
  col_scale_kernel<<<(Dout + 255) / 256, 256, 0, s>>>(scale, Dout);
  return cudaGetLastError();
}

cudaError_t launch_w8a8_gemm(const uint8_t* a_q, const float* a_scale, const uint8_t* w_q, const float* w_scale,
                             int32_t T, int32_t D, int32_t Dout, void* out, int* status, uint64_t wait_limit_ns,
                             cudaStream_t s) {
  __nv_bfloat16* o = static_cast<__nv_bfloat16*>(out);
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // Estimated run (ns): waves of tiles x (k-blocks x time of one + a tile's fixed part) + launch and fill, all
  // fitted to measured runs of 40 to 9400 tokens and 512 to 8960 features (within 15 %).  One CTA is
  // bound by its shared memory: a k-block's (128 + BN) x 128 bytes are written by TMA and read by
  // the UMMAs at 128 bytes per clock, so wider tiles cost less per MAC.  A pair halves B's
  // part, 325 against 366 ns at 256 columns, but its tiles are twice as high and both CTAs have to meet
  // before the first load: it needs several waves.  Pairs with 128 or 192 columns were never faster than
  // one CTA with the same columns (4680 x 1536 x 1536: 13.1 against 11.5 us with 192).
  struct Shape {
    int bn, ctas, kblock_ns, start_ns;
  };
  static constexpr Shape kShapes[4] = {
      {256, 2, 325, 4800}, {256, 1, 366, 3000}, {192, 1, 325, 3000}, {128, 1, 308, 3000}};
  const int64_t m_tiles = (static_cast<int64_t>(T) + QM - 1) / QM;
  int best = -1;
  int64_t best_cost = 0;
  for (int i = 0; i < 4; ++i) {
    const Shape& f = kShapes[i];
    if (Dout % f.bn != 0 || sms < f.ctas) continue;
    const int64_t rows = QM * f.ctas, units = sms / f.ctas;
    const int64_t tiles = (T + rows - 1) / rows * (Dout / f.bn);
    const int64_t cost = (tiles + units - 1) / units * (D / QK * f.kblock_ns + 360) + f.start_ns;
    if (best < 0 || cost < best_cost) {
      best = i;
      best_cost = cost;
    }
  }
  // Few tiles and many k-blocks: clusters of `split` CTAs share a tile's k-blocks and merge their sums through
  // distributed shared memory, 2.6 to 2.9 us more for two cluster barriers and the merge.  64 x 5120 -> 640: 14.3 ->
  // 6.3 us, 256 x 5120 -> 1536: 14.7 -> 8.6, 40 x 1536 -> 1536: 6.4 -> 6.0; 512 x 2048 -> 2048 stays whole (7.97
  // against 8.54).  As many clusters as run at once: of four or eight CTAs that is taken as four fifths of the chip
  // (any more would run later: an estimate, not a limit).
  int split = 1;
  for (const int c : {2, 4, 8}) {
    const int64_t tiles = m_tiles * (Dout / 128);
    if (D / QK < c || tiles * c * (c > 2 ? 5 : 4) > 4 * static_cast<int64_t>(sms)) break;
    const int64_t cost = (D / QK + c - 1) / c * 308 + 360 + 3000 + 2500 + 50 * c;
    if (cost < best_cost) {
      split = c;
      best_cost = cost;
    }
  }
  if (split > 1)
    return launch_gemm_bn<128, false, true>(split, a_q, a_scale, w_q, w_scale, T, D, Dout, o, status, wait_limit_ns, s);
  const auto run = best == 0 ? launch_gemm_bn<256, true> : best == 1 ? launch_gemm_bn<256, false>
                 : best == 2 ? launch_gemm_bn<192, false> : launch_gemm_bn<128, false>;
  return run(1, a_q, a_scale, w_q, w_scale, T, D, Dout, o, status, wait_limit_ns, s);
}

}  // namespace ispa
