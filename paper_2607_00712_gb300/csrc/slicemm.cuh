// Products of fp64-grade matrices on the bf16 tensor cores, by exact slices.
//
// A number x of a row whose largest magnitude is below 2^E is the fixed-point integer
// xi = x * 2^(63-E), and xi is split into seven signed 8-bit digits, d_0 .. d_6 in [-128, 128],
//   x ~= 2^E * sum_p d_p 2^(-7-8p),
// what is left over being below 2^-56 of the row's largest magnitude (E is the row's own power of
// two).  A product of two such rows is sum_s 2^(-14-8s) v_s with v_s = sum_{p+q=s} <d_p, d'_q>, s = 0 .. 7
// (the pairs beyond weigh less than the digits' own remainder; without s = 7 the solve's error on
// well-conditioned systems, 3e-16 of dW against 1e-15 in fp64 arithmetic, was up to twice as large).  Digits are bf16
// numbers, their products integers up to 2^14, and over 128 products of at most 7 pairs a v_s stays below
// 2^24: the fp32 accumulators of the tensor cores hold it exactly.  So every 128 products the
// accumulators are read back and added up as 64-bit integers, and a whole contraction is exact
// but for the digits dropped, in a fixed-point word of 2^-70 of the two rows' scales.  This is the
// error-free splitting of Ozaki, Ogita, Oishi and Rump (Numer. Algorithms 59, 2012).
//
// Why: GB300 has 1.25 TFLOP/s of fp64 against 2250 of dense bf16, so 34 bf16 products for one
// fp64 product are still an order of magnitude faster.
//
// Operand layout ("op").  Rows of a matrix with the contraction index k contiguous, cut into tiles
// of 64 rows and chunks of 32 k:  [k / 32][row / 64][slice 7][(row / 8) % 8][(k % 32) / 8][row % 8][k % 8]
// bf16, i.e. 28 KB per (chunk, tile), each 8 x 8 block a 128-byte UMMA core matrix (K-major, no
// swizzle).  The columns' seven slices arrive by ONE bulk copy, without a tensor map, and slices q,
// q + 1, ... of it form one operand of 128, 192, ... columns; the rows' come as fourteen copies of 4 KB that put
// two tiles' slice p together.  So the same op serves as rows (128 of them) and as columns (64).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"
#include "pdl.cuh"
#include "ptx.cuh"

namespace ispa {

constexpr int SL = 7;                       // slices
constexpr int SL_K = 32;                    // k per chunk (one pipeline stage)
constexpr int SL_BLOCK = 64 * SL_K * 2;     // bytes of 64 rows x 32 k of one slice
constexpr int SL_TILE = SL * SL_BLOCK;      // of all seven
constexpr int SL_NAN = 1 << 28;             // exponent of a row that holds a NaN or an infinity

// ---------------------------------------------------------------- digits
// Fixed-point image of |x| < 2^E with 63 fraction bits, rounded to nearest; integer arithmetic
// only (the fp64 pipe converts 2 numbers per clock and SM).
__device__ __forceinline__ int64_t fix63(uint64_t mant, int shift, bool neg) {   // mant * 2^shift
  uint64_t v;
  if (shift >= 0) v = mant << (shift & 63);   // below 64 for all but zero
  else v = shift > -63 ? (mant + (1ull << (-shift - 1))) >> -shift : 0ull;
  return neg ? -static_cast<int64_t>(v) : static_cast<int64_t>(v);
}

template <typename T>
struct SliceSrc;
template <>
struct SliceSrc<float> {
  using Mag = uint32_t;
  static __device__ Mag mag(float x) { return __float_as_uint(x) & 0x7FFFFFFFu; }
  static __device__ int exp_of(Mag m) {
    const int e = static_cast<int>(m >> 23);
    return m == 0 ? 0 : (e == 255 ? SL_NAN : e - 126);
  }
  static __device__ int64_t fixed(float x, int E) {
    const uint32_t m = mag(x);
    const int e = static_cast<int>(m >> 23);
    const uint64_t mant = (m & 0x7FFFFFu) | (e ? 0x800000u : 0u);
    return fix63(mant, 63 - E + (e ? e : 1) - 150, __float_as_uint(x) >> 31);
  }
};
template <>
struct SliceSrc<double> {
  using Mag = unsigned long long;
  static __device__ Mag mag(double x) { return __double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFll; }
  static __device__ int exp_of(Mag m) {
    const int e = static_cast<int>(m >> 52);
    return m == 0 ? 0 : (e == 2047 ? SL_NAN : (e ? e - 1022 : -1022));
  }
  static __device__ int64_t fixed(double x, int E) {
    const Mag m = mag(x);
    const int e = static_cast<int>(m >> 52);
    const uint64_t mant = (m & 0xFFFFFFFFFFFFFull) | (e ? 1ull << 52 : 0ull);
    return fix63(mant, 63 - E + (e ? e : 1) - 1075, __double_as_longlong(x) < 0);
  }
};
template <>
struct SliceSrc<int64_t> {   // fixed point already, 63 fraction bits
  using Mag = unsigned long long;
  static __device__ Mag mag(int64_t x) { return x < 0 ? 0ull - static_cast<Mag>(x) : static_cast<Mag>(x); }
  static __device__ int exp_of(Mag m) { return m == 0 ? 0 : 1 - __clzll(static_cast<long long>(m)); }
  static __device__ int64_t fixed(int64_t x, int E) { return static_cast<int64_t>(static_cast<uint64_t>(x) << -E); }
};

// Bytes from an op's start to row r's eight values k .. k + 7 (k % 8 == 0) of slice 0.
__device__ __forceinline__ int64_t sl_offset(int64_t chunk, int n_t, int r, int kc) {
  return (chunk * n_t + (r >> 6)) * SL_TILE + ((r >> 3) & 7) * 512 + kc * 128 + (r & 7) * 16;
}

// The digits of eight fixed-point numbers as bf16, stored at dst + SL_BLOCK * slice (16 bytes each).
// A number is rounded to 56 bits; with 128 added at every digit but the first its bytes are the digits plus 128
// (the first keeps its sign and range [-128, 128]), so that a digit costs a byte permute and an addition: byte b under
// the exponent of 2^23 is the fp32 number 2^23 + b.  Rounding and subtracting 64-bit digits one after another took five
// times as many instructions: with fixed_to_double's funnel shifts a 1536 x 1536 solve went from 3.07 to 2.93 ms,
// 5120 x 5120 from 28.4 to 27.5.
__device__ __forceinline__ void store_digits8(const int64_t* xi, uint8_t* dst) {
  constexpr float kBias = 8388608.f + 128.f;
  uint32_t lo[8], hi[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint64_t z = static_cast<uint64_t>(((xi[i] >> 7) + 1) >> 1) + 0x808080808080ull;   // no overflow at the top
    lo[i] = static_cast<uint32_t>(z);
    hi[i] = static_cast<uint32_t>(z >> 32);
  }
#pragma unroll
  for (int s = 0; s < SL; ++s) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      uint32_t d;   // 2^23 + 128 + the digit
      if (s == 0) d = 0x4B000080u + static_cast<uint32_t>(static_cast<int32_t>(hi[i]) >> 16);
      else d = __byte_perm(s < 3 ? hi[i] : lo[i], 0x4B000000u, 0x7650u | static_cast<uint32_t>((6 - s) & 3));
      const uint32_t b = __float_as_uint(__uint_as_float(d) - kBias);   // exact in bf16
      w[i >> 1] = (i & 1) ? __byte_perm(w[i >> 1], b, 0x7632) : b;
    }
    *reinterpret_cast<uint4*>(dst + SL_BLOCK * s) = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

// What a slice kernel takes: grid.y segments z of `rows` rows x `ks` k.  Segments either follow each other
// along k (L's block columns: z_k chunks apart in the op, exponents per segment) or are blocks down a
// diagonal (z_rows rows apart, in the same chunks).
struct SliceParams {
  const void* src;
  int64_t ld;          // elements between rows (k-contiguous source) or between k (row-contiguous source)
  int64_t z_src;       // elements between the segments' first values
  int32_t rows, ks;    // valid rows and k of a segment
  int32_t rows_total, ks_total;   // if not 0: segment z has at most rows_total - z z_rows rows (those past
                                  // them are not written), ks_total - z (z_k or z_rows) k
  int32_t k_pad;       // k written: a multiple of 32, zeros past the valid ones (z_k segments: only those)
  int32_t z_rows;      // op rows between segments
  int32_t z_k;         // k between segments in the op: 0 or k_pad
  int32_t z_exp;       // exponents between segments
  int32_t win;         // z_k segments: if not 0, only the rows of the segment's own window of so many rows, and
                       // a window's segments start again at the op's first chunk
  int32_t lower;       // z_k segments: 1: only the rows past the segment's k, -1: only those before them
  int32_t n_t;         // tiles of 64 rows of the op
  const int32_t* k_exp;   // SCALED: value k of a row is taken times 2^(k_sign k_exp[k]); k_sign is 1 or -1
  int32_t k_sign;
  const int32_t* r_max;   // SCALED, row-contiguous source: the rows' exponents (SL_NONE, SL_NAN as SliceMax takes them)
  uint8_t* op;
  int32_t* exps;
};
__device__ __forceinline__ int sl_rows(const SliceParams& p, int z) {
  return p.rows_total ? min(p.rows, p.rows_total - z * p.z_rows) : p.rows;
}
__device__ __forceinline__ int sl_ks(const SliceParams& p, int z) {
  return p.ks_total ? min(p.ks, p.ks_total - z * (p.z_k ? p.z_k : p.z_rows)) : p.ks;
}
__device__ __forceinline__ int sl_z(const SliceParams& p, int z) { return p.win ? z % (p.win / p.z_k) : z; }
__device__ __forceinline__ int sl_row0(const SliceParams& p, int z) { return p.win ? z * p.z_k / p.win * p.win : 0; }
__device__ __forceinline__ int sl_pad(const SliceParams& p, int ks) {
  return p.z_k ? (ks + SL_K - 1) / SL_K * SL_K : p.k_pad;
}
// The largest magnitude of a row, and its exponent.  SCALED compares exponents instead: a power of two for each value
// makes the magnitudes leave their type, and the row's exponent is all that is taken from them.
constexpr int SL_NONE = -(1 << 30);   // no value yet, or all zero
template <typename T, bool SCALED>
struct SliceMax {
  using V = typename SliceSrc<T>::Mag;
  static constexpr V none = 0;
  static __device__ V of(T x, int) { return SliceSrc<T>::mag(x); }
  static __device__ int exp_of(V v) { return SliceSrc<T>::exp_of(v); }
};
template <typename T>
struct SliceMax<T, true> {
  using V = int;
  static constexpr V none = SL_NONE;
  static __device__ V of(T x, int scale) {
    const typename SliceSrc<T>::Mag m = SliceSrc<T>::mag(x);
    return m == 0 ? SL_NONE : SliceSrc<T>::exp_of(m) + scale;
  }
  static __device__ int exp_of(V v) { return v == SL_NONE ? 0 : (v > SL_NAN / 2 ? SL_NAN : v); }
};
// The scales of values k .. k + 7 (k % 8 == 0; k_exp is 16-byte aligned and goes up to k_pad).
template <bool SCALED>
__device__ __forceinline__ void sl_scales8(const SliceParams& p, int k, int (&s)[8]) {
  int4 a = make_int4(0, 0, 0, 0), b = a;
  if constexpr (SCALED) {
    a = reinterpret_cast<const int4*>(p.k_exp + k)[0];
    b = reinterpret_cast<const int4*>(p.k_exp + k)[1];
  }
  s[0] = p.k_sign * a.x, s[1] = p.k_sign * a.y, s[2] = p.k_sign * a.z, s[3] = p.k_sign * a.w;
  s[4] = p.k_sign * b.x, s[5] = p.k_sign * b.y, s[6] = p.k_sign * b.z, s[7] = p.k_sign * b.w;
}

// Which of a segment's values are there (the others are taken as zero): all, k <= row, or k >= row.
enum SlTri : int { SL_FULL, SL_LOWER, SL_UPPER };
template <int TRI>
__device__ __forceinline__ bool sl_there(int row, int k) {
  return TRI == SL_FULL || (TRI == SL_LOWER ? k <= row : k >= row);
}

// Source with k contiguous.  One CTA (8 warps, 16 for long rows) per 8 rows (blockIdx.x) and segment
// (blockIdx.y): first a warp or two find a row's exponent, then the warps take the segment's chunks in turn, a
// thread 8 k of one row, a warp 8 rows x 32 k, so that each slice of it is one contiguous 512-byte
// store.  (Loading once, in the second pass's order, and reducing over the CTA is slower, 10.1 us
// against 9.1 on average in a 5120 x 5120 solve: each of those loads touches 32 sectors.)
template <typename T, int TRI, bool SCALED>
__global__ void __launch_bounds__(512) slice_rows_kernel(const SliceParams p) {
  using S = SliceSrc<T>;
  using M = SliceMax<T, SCALED>;
  pdl_wait();
  pdl_trigger();
  __shared__ typename M::V red[2][8];
  const int z = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warp = blockDim.x >> 5;
  const int zc = sl_z(p, z), r0 = sl_row0(p, z) + blockIdx.x * 8;
  if (p.lower > 0 && r0 < (z + 1) * p.k_pad) return;
  if (p.lower < 0 && r0 >= z * p.k_pad) return;
  const int rows = sl_rows(p, z), ks = sl_ks(p, z), k_pad = sl_pad(p, ks);
  if (p.rows_total && r0 >= rows) return;
  const T* src = static_cast<const T*>(p.src) + z * p.z_src + r0 * p.ld;
  typename M::V m = M::none;
  {
    const int r = warp & 7;
    const T* row = src + r * p.ld;
    if (r0 + r < rows) {
      for (int k = lane + 32 * (warp >> 3); k < ks; k += 4 * n_warp)
        if (sl_there<TRI>(r0 + r, k)) m = max(m, M::of(row[k], SCALED ? p.k_sign * p.k_exp[k] : 0));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) red[warp >> 3][r] = m;
  }
  __syncthreads();
  const int r = lane & 7, kc = lane >> 3;
  m = n_warp > 8 ? max(red[0][r], red[1][r]) : red[0][r];
  const int E = M::exp_of(m);
  if (threadIdx.x < 8) p.exps[zc * p.z_exp + z * p.z_rows + r0 + r] = E;
  const bool live = r0 + r < rows && E != SL_NAN;
  const T* row = src + r * p.ld;
  for (int c = warp; c < k_pad / SL_K; c += n_warp) {
    int64_t xi[8];
    int scale[8];
    sl_scales8<SCALED>(p, c * SL_K + kc * 8, scale);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = c * SL_K + kc * 8 + i;
      xi[i] = live && k < ks && sl_there<TRI>(r0 + r, k) ? S::fixed(row[k], E - scale[i]) : 0;
    }
    store_digits8(xi, p.op + sl_offset(zc * (p.z_k / SL_K) + c, p.n_t, z * p.z_rows + r0 + r, kc));
  }
}

// Source with rows contiguous (k strided).  One CTA (8 warps, 32 for long segments) per 32 rows and
// segment; lane = row, so every load is a contiguous run of the source and every slice store four
// 128-byte runs.  Where that leaves SMs idle the stores are split over blockIdx.z, each CTA finding the exponents
// for itself (SCALED: they are given, six times over the search took as long as the stores).
template <typename T, int TRI, bool SCALED>
__global__ void __launch_bounds__(1024) slice_cols_kernel(const SliceParams p) {
  using S = SliceSrc<T>;
  using M = SliceMax<T, SCALED>;
  pdl_wait();
  pdl_trigger();
  __shared__ typename M::V red[32][32];
  const int z = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warp = blockDim.x >> 5;
  const int zc = sl_z(p, z), r0 = sl_row0(p, z) + blockIdx.x * 32, r = r0 + lane;
  if (p.lower > 0 && r0 < (z + 1) * p.k_pad) return;
  if (p.lower < 0 && r0 >= z * p.k_pad) return;
  const int rows = sl_rows(p, z), ks = sl_ks(p, z), k_pad = sl_pad(p, ks);
  if (p.rows_total && r0 >= rows) return;
  const T* src = static_cast<const T*>(p.src) + z * p.z_src + r;
  const bool in = r < rows;
  typename M::V m = M::none;
  if constexpr (SCALED) {
    if (in) m = p.r_max[r];
  } else {
    if (in) {
      for (int q = warp; 8 * q < ks; q += n_warp) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int k = 8 * q + i;
          if (k < ks && sl_there<TRI>(r, k)) m = max(m, M::of(src[k * p.ld], 0));
        }
      }
    }
    red[warp][lane] = m;
    __syncthreads();
    for (int w = 0; w < n_warp; ++w) m = max(m, red[w][lane]);
  }
  const int E = M::exp_of(m);
  if (z * p.z_rows + r >= p.n_t * 64) return;
  if (warp == 0 && blockIdx.z == 0) p.exps[zc * p.z_exp + z * p.z_rows + r] = E;
  const bool live = in && E != SL_NAN;
  for (int q = warp + n_warp * blockIdx.z; q < k_pad / 8; q += n_warp * gridDim.z) {
    int64_t xi[8];
    int scale[8];
    sl_scales8<SCALED>(p, 8 * q, scale);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int k = 8 * q + i;
      xi[i] = live && k < ks && sl_there<TRI>(r, k) ? S::fixed(src[k * p.ld], E - scale[i]) : 0;
    }
    store_digits8(xi, p.op + sl_offset(zc * (p.z_k / SL_K) + (q >> 2), p.n_t, z * p.z_rows + r, q & 3));
  }
}

// ---------------------------------------------------------------- product
enum SlMode : int {
  SL_STORE,   // out[col][row] = product * 2^-row_exp[row]   (row_exp null: 1)
  SL_SUB,     // out[col][row] -= product
  SL_CHOL,    // lower tiles: fixed[col][row] -= product, 62 fraction bits
  SL_DOT      // lower tiles: *dot += sum_{i >= j} (i > j ? 2 : 1) product_ij sym[j][i]
};

struct SlGemm {
  const uint8_t* a;       // op of the rows, at its first chunk
  const uint8_t* b;       // op of the columns
  int64_t a_chunk, b_chunk;   // bytes between chunks
  const int32_t* ea;      // exponents of the rows / columns
  const int32_t* eb;
  int32_t row0, col0;     // first row and column (multiples of 8)
  int32_t n_mt, n_nt;     // tiles of 128 rows, of 64 columns (SL_STORE, SL_SUB)
  int32_t n_tiles;        // all tiles
  int32_t n_chunks;       // chunks of 32 k
  int32_t n_split;        // SL_DOT: pieces that the chunks of a tile are cut into (whole flushes); else 1
  int32_t row_end;        // rows and columns stored stay below these
  int32_t col_end;
  int64_t ld;             // elements between columns of out / fixed / rows of sym
  void* out;
  const int32_t* row_exp;
  const float* sym;
  double* dot;
  int* status;
  int* flag;              // bit 1: a device wait ran out
  uint64_t wait_limit_ns;
};

constexpr int SG_EPI = 16;             // read-back warps: four per TMEM lane quarter, 16 columns each
constexpr int SG_COLS = 64 / (SG_EPI / 4);
constexpr int SG_THREADS = 64 + 32 * SG_EPI;   // warp 0 bulk copies, warp 1 UMMA, then the read-back warps
constexpr int SG_ST = 2;
constexpr int SG_A = 2 * SL_TILE;              // 128 rows, [slice][tile]: 56 KB
constexpr int SG_B = SL_TILE;                  // 64 rows: 28 KB
constexpr int SG_STAGE = SG_A + SG_B;
constexpr int SG_OFF_BAR = SG_ST * SG_STAGE;
constexpr int SG_N_BAR = 2 * SG_ST + 6 + 1;    // stages full / empty, groups full x3 / free x3, drain
constexpr int SG_S = 8;                        // sums v_0 .. v_7
// in groups that are read back one after another: s = 0 .. 2, 3 .. 4, 5 .. 7
__host__ __device__ constexpr int sg_s0(int h) { return h == 0 ? 0 : (h == 1 ? 3 : (h == 2 ? 5 : SG_S)); }
constexpr int SG_SMEM = SG_OFF_BAR + SG_N_BAR * 8 + 16;
static_assert(SG_SMEM > 116 * 1024 && SG_SMEM <= 232448, "one CTA per SM");
constexpr int SG_FLUSH = 4;                    // chunks (128 k) between read-backs: v_s < 2^24
constexpr uint64_t SG_DRAIN_NS = 200ull * 1000 * 1000;

// K-major operand without swizzle: 128-byte core matrices, `lbo` bytes apart along k, `sbo` along rows.
__device__ __forceinline__ uint64_t core_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return static_cast<uint64_t>((addr & 0x3FFFFu) >> 4) | (static_cast<uint64_t>(lbo >> 4) << 16) |
         (static_cast<uint64_t>(sbo >> 4) << 32) | (1ull << 46);
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}

// (hi 2^32 + lo) 2^e rounded to nearest, without the fp64 pipe (2 operations per clock and SM); e is a row's and a
// column's exponent and a few tens: normal results only need the integer path, in 32-bit words and funnel shifts, the
// rest goes through ldexp.
__device__ __forceinline__ double fixed_to_double(int64_t hi, uint32_t lo, int e) {
  const uint32_t sign = static_cast<uint32_t>(static_cast<uint64_t>(hi) >> 32) & 0x80000000u;
  const uint32_t neg = static_cast<uint32_t>(static_cast<int32_t>(sign) >> 31);   // all ones for a negative number
  // magnitude: complement and add one
  const uint32_t w0 = (lo ^ neg) - neg;
  const uint64_t up = (static_cast<uint64_t>(hi) ^ (static_cast<uint64_t>(neg) << 32 | neg)) + (neg & (w0 == 0));
  uint32_t x2 = static_cast<uint32_t>(up >> 32), x1 = static_cast<uint32_t>(up), x0 = w0;
  int ex = 1023 + 95 + e;
  if (x2 == 0) {   // the leading word first
    x2 = x1;
    x1 = x0;
    x0 = 0;
    ex -= 32;
    if (x2 == 0) {
      x2 = x1;
      x1 = 0;
      ex -= 32;
      if (x2 == 0) return 0.0;
    }
  }
  const int lz = __clz(x2);
  ex -= lz;
  const uint32_t m1 = __funnelshift_l(x1, x2, lz), m0 = __funnelshift_l(x0, x1, lz);   // the leading 64 bits
  // 53 bits; a carry out raises the exponent by itself
  const uint64_t m = (static_cast<uint64_t>(m1 >> 11) << 32 | __funnelshift_r(m0, m1, 11)) + ((m0 >> 10) & 1);
  if (ex < 1 || ex > 2045) return ldexp(sign ? -static_cast<double>(m) : static_cast<double>(m), ex - 1023 - 52);
  const uint32_t top = (static_cast<uint32_t>(ex - 1) << 20) + static_cast<uint32_t>(m >> 32) + sign;
  return __hiloint2double(static_cast<int>(top), static_cast<int>(static_cast<uint32_t>(m)));
}

__device__ __forceinline__ double pow2d(int e) {   // 2^e; 0 below the normal range, inf above it
  return e < -1022 ? 0.0 : __longlong_as_double(static_cast<long long>(e > 1023 ? 2047 : e + 1023) << 52);
}

__device__ __forceinline__ void sg_tile(const SlGemm& p, bool tri, int t, int& row, int& col) {
  if (tri) {   // row tile i holds the 2 (i + 1) column tiles on or below the diagonal
    int i = static_cast<int>((sqrtf(4.f * t + 1.f) - 1.f) * 0.5f);
    while (i * (i + 1) > t) --i;
    while ((i + 1) * (i + 2) <= t) ++i;
    row = p.row0 + i * 128;
    col = p.col0 + (t - i * (i + 1)) * 64;
  } else {   // row tiles vary fastest: the CTAs of a wave share the columns' op
    row = p.row0 + (t % p.n_mt) * 128;
    col = p.col0 + (t / p.n_mt) * 64;
  }
}

// Work item t: its tile and its chunks [c0, c1).
__device__ __forceinline__ void sg_item(const SlGemm& p, bool tri, int t, int& row, int& col, int& c0, int& c1) {
  const int tile = t / p.n_split, piece = t - tile * p.n_split;
  const int n_flush = (p.n_chunks + SG_FLUSH - 1) / SG_FLUSH;
  sg_tile(p, tri, tile, row, col);
  c0 = n_flush * piece / p.n_split * SG_FLUSH;
  c1 = min(n_flush * (piece + 1) / p.n_split * SG_FLUSH, p.n_chunks);
}

// The UMMAs of one chunk of 32 k (operands at da and db) into the eight sums, flush f: `first` and `last` chunk of it.
__device__ __forceinline__ bool sg_umma_chunk(uint32_t tmem, uint64_t da, uint64_t db, bool first, bool last,
                                              uint32_t gfull0, uint32_t gfree0, int f, const WaitCtx& wc) {
#pragma unroll
  for (int h = 0; h < 3; ++h) {
    // the group's sums of the flush before have been read
    if (first && !mbar_wait(gfree0 + 8 * h, (f & 1) ^ 1, wc, 43 + h, f)) return false;
    tc_fence_after();
#pragma unroll
    for (int ks = 0; ks < SL_K / 16; ++ks)
#pragma unroll
      for (int i = 0; i < (h < 2 ? sg_s0(h + 1) : SL); ++i) {
        // slice q of the rows with the columns' slices s0 .. s1 - 1 in one UMMA: sums q + s0 .. q + s1 - 1.
        // The first one of a group starts all of its sums; in the last group that is q = 1 (q = 0 has none for s = 7)
        const int q = h == 2 && i < 2 ? 1 - i : i;
        const int s0 = sg_s0(h) > q ? sg_s0(h) - q : 0, s1 = sg_s0(h + 1) - q < SL ? sg_s0(h + 1) - q : SL;
        umma_ss(tmem + 64 * (q + s0), da + (q * 2 * SL_BLOCK + ks * 256) / 16, db + (s0 * SL_BLOCK + ks * 256) / 16,
                idesc_bf16(128, 64 * (s1 - s0), false, false), (!first || ks > 0 || i > 0) ? 1u : 0u);
      }
    if (last) tc_commit(gfull0 + 8 * h);
  }
  return true;
}

// Flush f's sums of this thread's row and SG_COLS columns (TMEM address tbase), added to hi 2^32 + lo in units of
// 2^-70 of the rows' scales.  The whole warp calls it.
__device__ __forceinline__ bool sg_read_sums(int64_t (&hi)[SG_COLS], uint32_t (&lo)[SG_COLS], uint32_t tbase, int lane,
                                             uint32_t gfull0, uint32_t gfree0, int f, const WaitCtx& wc) {
#pragma unroll
  for (int h = 0; h < 3; ++h) {
    if (!__all_sync(0xffffffffu, mbar_wait(gfull0 + 8 * h, f & 1, wc, 46 + h, f))) return false;
    tc_fence_after();
    const int ns = sg_s0(h + 1) - sg_s0(h);
#pragma unroll
    for (int c = 0; c < SG_COLS / 8; ++c) {
      uint32_t v[3][8];
#pragma unroll
      for (int s = 0; s < ns; ++s) tmem_ld8(tbase + 64 * (sg_s0(h) + s) + 8 * c, v[s]);
#pragma unroll
      for (int s = 0; s < ns; ++s) tmem_wait_ld8(v[s]);
      if (c == SG_COLS / 8 - 1) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(gfree0 + 8 * h);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int u0 = __float2int_rn(__uint_as_float(v[0][i])), u1 = __float2int_rn(__uint_as_float(v[1][i]));
        const int u2 = ns > 2 ? __float2int_rn(__uint_as_float(v[2][i])) : 0;
        if (h == 0) {
          // |u0| <= 2^21
          hi[8 * c + i] += static_cast<int64_t>(u0 * 256 + u1) * 65536 + static_cast<int64_t>(u2) * 256;
        } else {
          if (h == 1) hi[8 * c + i] += u0;
          const int64_t l = h == 1 ? static_cast<int64_t>(u1) * (1 << 24)
                                   : static_cast<int64_t>(u0) * 65536 + static_cast<int64_t>(u1) * 256 + u2;
          const uint64_t sum = static_cast<uint64_t>(lo[8 * c + i]) + static_cast<uint32_t>(l);
          lo[8 * c + i] = static_cast<uint32_t>(sum);
          hi[8 * c + i] += (l >> 32) + static_cast<int64_t>(sum >> 32);
        }
      }
    }
  }
  return true;
}

// 128 x 64 output tiles; TMEM holds the eight v_s of a tile (8 x 64 columns, s after s).  A stage is 32 k
// of all 14 slices (84 KB), used for all 34 pairs: about 40 bytes per clock of operand traffic, where
// one pair at a time would need 128.  An UMMA of 128 x 64 x 16 takes as long as one of 128 x 128 x 16 (64
// clocks, measured), so one slice of the rows meets two or three adjacent slices of the columns in one
// UMMA of 128 or 192 columns, whose sums are adjacent v_s.
// The v_s are read back in three groups, each handed over as soon as its last UMMA of the flush is
// in the stream, so that a read-back runs under the other groups' UMMAs.
template <int MODE>
__global__ void __launch_bounds__(SG_THREADS, 1) slice_gemm_kernel(const SlGemm p) {
  constexpr bool TRI = MODE == SL_CHOL || MODE == SL_DOT;
  extern __shared__ __align__(1024) uint8_t smem[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SG_OFF_BAR);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + SG_N_BAR);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const uint32_t sbase = smem_u32(smem);
  const uint32_t full0 = smem_u32(bars), empty0 = full0 + 8 * SG_ST, gfull0 = empty0 + 8 * SG_ST, gfree0 = gfull0 + 24,
                 drain_bar = gfree0 + 24;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < SG_ST; ++i) {
      mbar_init(full0 + 8 * i, 1);
      mbar_init(empty0 + 8 * i, 1);
    }
    for (int i = 0; i < 3; ++i) {
      mbar_init(gfull0 + 8 * i, 1);
      mbar_init(gfree0 + 8 * i, SG_EPI);
    }
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();
  pdl_trigger();
  const WaitCtx wc{abort_flag, p.status, p.wait_limit_ns};

  if (warp == 0) {
    if (lane == 0) {
      int g = 0;
      bool ok = true;
      for (int t = blockIdx.x; ok && t < p.n_tiles; t += gridDim.x) {
        int row, col, k0, k1;
        sg_item(p, TRI, t, row, col, k0, k1);
        const uint8_t* a = p.a + static_cast<int64_t>(row >> 6) * SL_TILE;
        const uint8_t* b = p.b + static_cast<int64_t>(col >> 6) * SL_TILE;
        for (int c = k0; c < k1; ++c, ++g) {
          const int st = g % SG_ST;
          if (!mbar_wait(empty0 + 8 * st, ((g / SG_ST) & 1) ^ 1, wc, 41, g)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(full0 + 8 * st, SG_STAGE);
          for (int i = 0; i < 2 * SL; ++i)   // slice i >> 1 of row tile i & 1
            bulk_load(sbase + st * SG_STAGE + i * SL_BLOCK, a + c * p.a_chunk + (i & 1) * SL_TILE + (i >> 1) * SL_BLOCK,
                      SL_BLOCK, full0 + 8 * st);
          bulk_load(sbase + st * SG_STAGE + SG_A, b + c * p.b_chunk, SG_B, full0 + 8 * st);
        }
      }
      for (int i = g > SG_ST ? g - SG_ST : 0; i < g; ++i)
        mbar_wait_drain(full0 + 8 * (i % SG_ST), (i / SG_ST) & 1, SG_DRAIN_NS);
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      int g = 0, f = 0;   // stages used, flushes begun
      bool ok = true;
      for (int t = blockIdx.x; ok && t < p.n_tiles; t += gridDim.x) {
        int row, col, k0, k1;
        sg_item(p, TRI, t, row, col, k0, k1);
        for (int c0 = k0; ok && c0 < k1; c0 += SG_FLUSH, ++f) {
          const int c1 = min(c0 + SG_FLUSH, k1);
          for (int c = c0; ok && c < c1; ++c, ++g) {
            const int st = g % SG_ST;
            if (!mbar_wait(full0 + 8 * st, (g / SG_ST) & 1, wc, 42, g)) {
              ok = false;
              break;
            }
            const uint64_t da = core_desc(sbase + st * SG_STAGE, 128, 512);
            const uint64_t db = core_desc(sbase + st * SG_STAGE + SG_A, 128, 512);
            ok = sg_umma_chunk(tmem, da, db, c == c0, c == c1 - 1, gfull0, gfree0, f, wc);
            if (ok) tc_commit(empty0 + 8 * st);
          }
        }
      }
      tc_commit(drain_bar);
      mbar_wait_drain(drain_bar, 0, SG_DRAIN_NS);
    }
    __syncwarp();
  } else {
    // TMEM lanes 32 quarter .. + 31 (the tile's rows), columns SG_COLS part .. + SG_COLS - 1 of every sum
    const int quarter = warp & 3, part = (warp - 2) >> 2;
    const uint32_t tbase = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + SG_COLS * part;
    double dot = 0.0;
    int f = 0;
    bool ok = true;
#pragma unroll 1
    for (int t = blockIdx.x; ok && t < p.n_tiles; t += gridDim.x) {
      // hi 2^32 + lo, in units of 2^-70 of the rows' scales
      int64_t hi[SG_COLS];
      uint32_t lo[SG_COLS];
#pragma unroll
      for (int i = 0; i < SG_COLS; ++i) hi[i] = lo[i] = 0;
      int row, col, k0, k1;
      sg_item(p, TRI, t, row, col, k0, k1);
#pragma unroll 1
      for (int c0 = k0; c0 < k1; c0 += SG_FLUSH, ++f) {
        ok = sg_read_sums(hi, lo, tbase, lane, gfull0, gfree0, f, wc);
        if (!ok) break;
      }
      if (!ok) break;
      row += quarter * 32 + lane;
      col += SG_COLS * part;
      if (row < p.row_end) {
        const int ea = p.ea[row];
        if constexpr (MODE == SL_CHOL) {
          int64_t* out = static_cast<int64_t*>(p.out) + row;
#pragma unroll
          for (int i = 0; i < SG_COLS; ++i) {
            const int sh = 8 - (ea + p.eb[min(col + i, row)]);   // exponents of factor rows are never above 0
            const uint32_t rest = lo[i] >> min(sh, 31) >> (sh == 32);
            hi[i] = sh <= 32 ? static_cast<int64_t>(static_cast<uint64_t>(hi[i]) << (32 - sh)) + rest
                             : hi[i] >> min(sh - 32, 63);
          }
          int64_t o[SG_COLS];   // all in flight at once; nothing above the diagonal
#pragma unroll
          for (int i = 0; i < SG_COLS; ++i) o[i] = col + i <= row ? out[static_cast<int64_t>(col + i) * p.ld] : 0;
#pragma unroll
          for (int i = 0; i < SG_COLS; ++i)
            if (col + i <= row) out[static_cast<int64_t>(col + i) * p.ld] = o[i] - hi[i];
        } else {
          constexpr double kNan = __builtin_nan("");
          auto value = [&](int i, int c, int de) {   // NaN where the row or the column holds one
            const int e = ea + p.eb[c];
            return e > SL_NAN / 2 ? kNan : fixed_to_double(hi[i], lo[i], e - 70 + de);
          };
          if constexpr (MODE == SL_DOT) {
#pragma unroll
            for (int i = 0; i < SG_COLS; ++i) {
              const int c = col + i;
              if (c > row) break;
              dot = fma(value(i, c, row != c), static_cast<double>(p.sym[static_cast<int64_t>(c) * p.ld + row]), dot);
            }
          } else if constexpr (MODE == SL_STORE) {
            double* out = static_cast<double*>(p.out) + row;
            const int er = p.row_exp ? p.row_exp[row] : 0;
#pragma unroll
            for (int i = 0; i < SG_COLS; ++i)
              if (col + i < p.col_end) out[static_cast<int64_t>(col + i) * p.ld] = value(i, col + i, -er);
          } else {
            double* out = static_cast<double*>(p.out) + row;
            double x[SG_COLS], o[SG_COLS];
#pragma unroll
            for (int i = 0; i < SG_COLS; ++i) x[i] = col + i < p.col_end ? value(i, col + i, 0) : 0.0;
#pragma unroll
            for (int i = 0; i < SG_COLS; ++i)   // all in flight at once
              o[i] = col + i < p.col_end ? out[static_cast<int64_t>(col + i) * p.ld] : 0.0;
#pragma unroll
            for (int i = 0; i < SG_COLS; ++i)
              if (col + i < p.col_end) out[static_cast<int64_t>(col + i) * p.ld] = o[i] - x[i];
          }
        }
      }
    }
    if constexpr (MODE == SL_DOT) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
      // the stages are free: a warp is done once all of this CTA's sums have been read
      if (lane == 0) reinterpret_cast<double*>(smem)[warp - 2] = dot;
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (MODE == SL_DOT) {
    // one addition a CTA: each rounds the whole sum, and one a warp cost eps as many bits as all else
    if (threadIdx.x == 0) {
      double sum = 0.0;
      for (int i = 0; i < SG_EPI; ++i) sum += reinterpret_cast<const double*>(smem)[i];
      atomicAdd(p.dot, sum);
    }
  }
  if (threadIdx.x == 0 && *abort_flag) atomicOr(p.flag, 2);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

template <int MODE>
cudaError_t launch_slice_gemm(const SlGemm& p, int sms, cudaStream_t s) {
  const cudaError_t e = set_smem_limit_once(reinterpret_cast<const void*>(slice_gemm_kernel<MODE>), SG_SMEM);
  if (e != cudaSuccess) return e;
  const unsigned grid = static_cast<unsigned>(p.n_tiles < sms ? p.n_tiles : sms);
  return launch_pdl(slice_gemm_kernel<MODE>, dim3(grid), dim3(SG_THREADS), SG_SMEM, s, p);
}

}  // namespace ispa
