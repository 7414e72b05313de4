// Closed-form absorption solve (Sec. 3.2, Eq. 5-6), fp64-grade, on the tensor cores.
//
//   M  = G + lambda I                      (G symmetrised from its upper tiles)
//   L  = chol(M)                           (right-looking, panels of 64 columns)
//   Y  = L^{-1} (X W)                      (forward substitution in blocks of 128 rows)
//   dW = L^{-T} Y                          (back substitution)
//   eps = tr(W^T S W) - ||Y||_F^2 - lambda ||dW||_F^2
// The eps expression is Eq. 6 expanded with the normal equations
// (G + lambda I) dW = X W, which give tr(dW^T G dW) = ||Y||^2 - lambda||dW||^2
// and tr(dW^T X W) = ||Y||^2.
//
// Every cubic part is a product, and every product goes through slicemm.cuh (34 exact bf16 products
// for one fp64 one): X W, the trailing updates of the factorisation and of both substitutions, the
// products with the inverses of L's 128 x 128 diagonal blocks, and tr(W^T S W) = sum_ij S_ij (W W^T)_ij, half
// the work of S W and nothing to store.  Plain fp64 code ran all of it at 1.09 TFLOP/s, the chip's
// fp64 rate: 782 ms at hidden 5120 and 33 ms at 1536 (where the panels' launches and latency counted
// too), against 27.7 and 2.94 ms.  What bounds it now: at 5120 the products' tensor time and read-back (21
// of 28 ms), at 1536 the chain of 24 panels (45 us each) and 24 block steps, one after another.
// dW's error against 80-bit arithmetic, read before its rounding to fp32, at dim 384 (plain fp64 code's in brackets):
// features of one size or spread by exp(2 N(0, 1)) 3e-16 (1e-15); sums of half as many tokens as features 6e-11
// (1.2e-10), near-duplicate pairs 9e-11 (3.4e-10), rank 20 plus 1 % noise 2.4e-11 (3.5e-10), singular values falling to
// 1e-4 1.3e-12 (1.5e-11).  Errors are relative to the largest rows of the scaled solution: a row 1e-6 of them, of
// features that share no token with theirs, had 6e-11 of itself, where fp64 code had 7e-16.
//
// The factorisation runs in fixed point.  Row and column i are scaled by a power of two (exactly)
// so that M_ii lies in [1/4, 1); then every |M_ij|, every element of every Schur complement and
// every |L_ij| of a positive definite M is below 1, and 64-bit words with 62 (M) and 63 (L) fraction bits
// hold them with an absolute error of 2^-62, where fp64 has 2^-54 near 1.  The trailing update is then
// an integer subtraction, and a panel runs on the integer pipe.  A word that leaves its range shows
// that M is not positive definite, like a pivot that isn't positive.
//
// All of it is stored by columns (element (i, j) at [j][i]): a tile's epilogue thread owns a row,
// so its warp's accesses run along a column.
#include <cuda_runtime.h>
#include <stdint.h>

#include "internal.h"
#include "slicemm.cuh"

namespace ispa {

namespace {

constexpr int NB = 64;     // panel of the factorisation
constexpr int TB = 128;    // block of the substitutions
// Window of a large problem's substitutions.  Each block of 128 rows updates only the rows of its own
// window at once; the others get one product with K = 512 for the window's four blocks, a quarter of the
// read-modify-writes of B and of the pipeline fills: 30.7 -> 28.5 ms at 5120 x 5120 (the
// updates alone 10.3 -> 8.1).  It costs two launches a window and small products that fill few SMs, so it starts
// where the average update has 512 tiles: 3072 x 3072 (576 tiles) 10.11 -> 9.91 ms, 4096 x 4096 18.5 -> 17.65;
// at 400 tiles (2560 x 2560) 7.28 -> 7.29, at 144 (1536 x 1536) 3.13 -> 3.19.
constexpr int SB = 512;
constexpr size_t SB_TILES = 512;
constexpr int PR = 32;     // panel rows per CTA
constexpr int FLAG_NOT_SPD = 1;

// t_i: the power of two with M_ii 2^(-2 t_i) in [1/4, 1).  Rows past D (padding) get 0.
// u, ew: where col_exp_kernel's maxima start.
constexpr int U_NONE = -(1 << 20);   // a column of zeros: its weights count for nothing
__global__ void __launch_bounds__(256) equil_kernel(const float* __restrict__ gram, int D, int Dp, double lambda,
                                                    int32_t* __restrict__ t, int32_t* __restrict__ u, int n,
                                                    int32_t* __restrict__ ew, int* flag) {
  pdl_wait();
  pdl_trigger();
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i < n) ew[i] = SL_NONE;
  if (i >= Dp) return;
  int e = 0;
  if (i < D) {
    const double v = static_cast<double>(gram[static_cast<int64_t>(i) * (2 * D) + i]) + lambda;
    if (v > 0.0 && v <= 1.7976931348623157e308) {
      e = (SliceSrc<double>::exp_of(SliceSrc<double>::mag(v)) + 1) >> 1;
    } else {
      atomicOr(flag, FLAG_NOT_SPD);
    }
  }
  t[i] = e;
  u[i] = U_NONE;
}

// out[j] = max(out[j], exponent of max_i |m[i][j]| 2^(sign add[i])) for the columns of an fp32 matrix.  NANS: SL_NAN
// for a column that isn't finite (else such values are passed over).  A CTA takes 64 columns x 64 rows.
//
// It gives u_j, the power of two with max_i |X_ij| 2^(-t_i - u_j) in [1/2, 1), and the columns' exponents of
// 2^(u_j) W_jk.  X W is formed from X_ij 2^(-u_j) and W_jk 2^(u_j): both operands keep 56 bits below the largest value
// of a row or a column, so what counts is that the features j meet there at one size.  Without it a W that undoes
// large differences between features (W_j ~ 1 / f_j) lost as many bits as they differ by: dW's error at dim 384 was
// 7e-11 with f = exp(3 N(0, 1)) and 1e-7 with exp(4 N(0, 1)), where it is 4e-16 now and fp64 code has 1e-15.  The two
// launches and the scales cost 11 us of 2.91 ms at 1536 x 1536, 85 us of 27.5 ms at 5120 x 5120.
constexpr int U_COLS = 64, U_ROWS = 64, U_PART = U_ROWS / (256 / U_COLS);
template <bool NANS>
__global__ void __launch_bounds__(256) col_exp_kernel(const float* __restrict__ m, int64_t ld, int rows, int cols,
                                                      const int32_t* __restrict__ add, int sign,
                                                      int32_t* __restrict__ out) {
  pdl_wait();
  pdl_trigger();
  __shared__ int red[256];
  const int j = blockIdx.x * U_COLS + threadIdx.x % U_COLS;
  const int i0 = blockIdx.y * U_ROWS + threadIdx.x / U_COLS * U_PART;
  int e = SL_NONE;
#pragma unroll
  for (int n = 0; n < U_PART; ++n) {
    const int i = i0 + n;
    if (i >= rows || j >= cols) continue;
    const uint32_t mag = SliceSrc<float>::mag(m[i * ld + j]);
    const int xe = SliceSrc<float>::exp_of(mag);
    if (mag != 0 && (NANS || xe != SL_NAN)) e = max(e, xe == SL_NAN ? SL_NAN : xe + sign * add[i]);
  }
  red[threadIdx.x] = e;
  __syncthreads();
  if (threadIdx.x >= U_COLS || j >= cols) return;
#pragma unroll
  for (int n = 1; n < 256 / U_COLS; ++n) e = max(e, red[threadIdx.x + n * U_COLS]);
  if (e != SL_NONE) atomicMax(out + j, e);
}

// fix[j][i] (i >= j) = M_ij 2^(-t_i - t_j) with 62 fraction bits, from G's upper triangle (row j of G is column
// j here); the padding is the identity / 2.
__global__ void __launch_bounds__(256) form_kernel(const float* __restrict__ gram, int D, int Dp, double lambda,
                                                   const int32_t* __restrict__ t, int64_t* __restrict__ fix,
                                                   int* flag) {
  pdl_wait();
  pdl_trigger();
  const int j = blockIdx.x;
  const int i = blockIdx.y * 256 + threadIdx.x;
  if (i < j || i >= Dp) return;
  int64_t v = 0;
  if (i >= D) {
    v = i == j ? int64_t{1} << 61 : 0;
  } else {
    const float g = gram[static_cast<int64_t>(j) * (2 * D) + i];
    const int e = t[i] + t[j];
    bool bad;
    if (i == j) {
      const double d = static_cast<double>(g) + lambda;
      bad = !(d > 0.0 && d <= 1.7976931348623157e308);
      v = bad ? int64_t{1} << 61 : SliceSrc<double>::fixed(d, e + 1);
    } else {
      const uint32_t m = SliceSrc<float>::mag(g);
      const int ge = SliceSrc<float>::exp_of(m);   // |g| < 2^ge
      bad = m != 0 && ge - e > 1;                  // |M_ij| >= 1 (or not finite): not positive definite
      if (!bad && m != 0) {
        v = SliceSrc<float>::fixed(g, e + 1);
        bad = v >= (int64_t{1} << 62) || v <= -(int64_t{1} << 62);
      }
      if (bad) v = 0;
    }
    if (bad) atomicOr(flag, FLAG_NOT_SPD);
  }
  fix[static_cast<int64_t>(j) * Dp + i] = v;
}

// 1 / sqrt of the pivot d (62 fraction bits): y 2^e, y in [1, 2] with 62 fraction bits.  The fp32
// estimate m 2^-23 and one third-order Newton step in fixed point: y += y (err / 2 + 3/8 err^2),
// err = 1 - v y^2 below 2^-21.
__device__ __forceinline__ void pivot_rsqrt(int64_t d, uint64_t& y, int& e) {
  const int s = __clzll(d) & ~1;
  const uint64_t u = static_cast<uint64_t>(d) << s;   // v = u 2^-64 in [1/4, 1), d = v 2^(2 - s)
  e = (s - 2) >> 1;
  const float v = __uint2float_rn(static_cast<uint32_t>(u >> 32));
  float yf;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(v));   // 2^-16 v^(-1/2)
  const uint32_t m = min(max(__float2uint_rn(yf * 549755813888.f), 1u << 23), 1u << 24);   // 2^39
  const uint64_t t = __umul64hi(u, static_cast<uint64_t>(m) * m << 14);   // v y^2, 60 fraction bits
  const int64_t err = static_cast<int64_t>((1ull << 60) - t);
  const int e20 = static_cast<int>(err >> 20);
  const int64_t corr = (err >> 1) + ((3 * ((static_cast<int64_t>(e20) * e20) >> 20)) >> 3);
  y = (static_cast<uint64_t>(m) << 39) + static_cast<uint64_t>((static_cast<int64_t>(m) * corr) >> 21);
}

// An element of L as the panel's dot products take it: x 2^-30 + y 2^-58, rounded, y signed (28 bits).  A multiply-add
// is then three 32 x 32 + 64 bit ones without any shift or carry (a 64-bit multiply-high takes 21 issue slots, these
// 12); the middle sums of 64 products of rows whose norm is at most 1 stay below 2^62.  What is lost is half of 2^-58
// of the other factor a term and the product of the two y, 2^-62 at most, both either way, where fp64 rounds the
// running sum to 2^-54 of itself.  A square's y^2 is never negative: its mean goes into the rounding (a square of 0
// stays 0).  With y cut off and unsigned the diagonal of L L^T was 6e-18 too large, and eps of ill-conditioned systems
// 3e-14 of its terms off (here 2e-15, plain fp64 code 8e-15 to 4e-14); a fourth product for the two y gave the same
// as this but 6 us a panel.
__device__ __forceinline__ int2 pack_l(int64_t l) {   // 60 fraction bits
  return make_int2(static_cast<int>((l + 2 + (1 << 29)) >> 30),
                   static_cast<int>((static_cast<uint32_t>(l) + 2) << 2) >> 4);
}
struct Dot {
  int64_t hi = 0, mid = 0;
  __device__ __forceinline__ void add(const int2 a, const int2 b) {
    hi += static_cast<int64_t>(a.x) * b.x;
    mid += static_cast<int64_t>(a.x) * b.y;
    mid += static_cast<int64_t>(a.y) * b.x;
  }
  // 62 fraction bits
  __device__ __forceinline__ int64_t sum(int round = 1 << 25) const { return (hi << 2) + ((mid + round) >> 26); }
  __device__ __forceinline__ int64_t square() const { return sum((1 << 25) + (1 << 26) / 3); }
};

// c (62 fraction bits) times y 2^e with 63 fraction bits; a magnitude of 1 or more sets `over`.  pk: the same for the
// dot products.
__device__ __forceinline__ int64_t scale_col(int64_t c, uint64_t y, int e, bool& over, int2& pk) {
  const int64_t c1 = static_cast<int64_t>(static_cast<uint64_t>(c) << (e + 1));
  const __int128 p = static_cast<__int128>(c1) * static_cast<int64_t>(y >> 1);
  const int64_t hi = static_cast<int64_t>(p >> 64);   // 60 fraction bits
  over |= (c1 >> (e + 1)) != c || static_cast<uint64_t>(hi + (int64_t{1} << 60)) >= (uint64_t{1} << 61);
  pk = pack_l(hi);
  return static_cast<int64_t>(p >> 61);
}

struct PanelParams {
  int64_t* fix;       // [Dp][Dp] by columns: M, overwritten by L below the diagonal blocks
  int64_t* diag;      // [Dp / 64][64][64] by columns: L of the diagonal blocks
  int32_t Dp, k0;
  uint8_t* op;        // slices of the panel's rows (2 chunks of 32 columns)
  int32_t n_t;
  int32_t* exps;      // their exponents
  int* flag;
  int* status;
  uint64_t wait_limit_ns;
};

// One panel: every CTA factors the 64 x 64 diagonal block for itself (the same work on every SM, and
// no launch between it and the rows that need it) together with 32 rows below it, whose slices it writes.
// Column by column, four lanes a row (k mod 4 of its dot product).  What bounds it is the chain of the
// diagonal block's 64 columns: l of the last column -> the pivot and its reciprocal root -> the column's
// scaling.  So one warp keeps the diagonal up to date and does nothing but pivots, two scale, and eight take
// the next column's dot products, all but their last term, in the meantime.  The rows below the block
// aren't on the chain: their four warps follow at their own pace, an mbarrier per column.  (All rows in step
// took 1800 clocks a column, 63 us a panel, and one right-looking column at a time 3900.)
constexpr int PROWS = NB + PR;          // rows in shared memory
constexpr int PLD = NB + 1;
constexpr int PL = 4;                   // lanes per row
constexpr int P_DOT = PL * NB;          // threads of the diagonal block's dot products,
constexpr int P_SCALE = P_DOT + NB;     // its scaling up to here,
constexpr int P_CHAIN = P_SCALE + 32;   // the pivots' warp up to here,
constexpr int P_THREADS = P_CHAIN + PL * PR;   // and the rows below
constexpr int PANEL_SMEM = (2 * PROWS * PLD + 3 * NB) * 8 + NB * 4 + 16;
static_assert(P_THREADS <= 1024, "panel roles");
__device__ __forceinline__ void chain_sync() { asm volatile("bar.sync 1, %0;" ::"n"(P_CHAIN) : "memory"); }

__global__ void __launch_bounds__(P_THREADS) panel_kernel(const PanelParams p) {
  extern __shared__ int64_t psm[];
  int64_t* a = psm;                                               // [row][PLD]: M, then L
  int2* pk = reinterpret_cast<int2*>(psm + PROWS * PLD);           // L for the dot products
  uint64_t* ys = reinterpret_cast<uint64_t*>(psm + 2 * PROWS * PLD);   // the pivots' reciprocal roots
  int64_t* cs = reinterpret_cast<int64_t*>(ys + NB);               // column j before its scaling
  uint64_t* done = reinterpret_cast<uint64_t*>(cs + NB);           // mbarrier j: column j of the block is complete
  int* es = reinterpret_cast<int*>(done + NB);
  volatile int* abort_flag = es + NB;
  pdl_wait();
  pdl_trigger();
  const int tid = threadIdx.x, lane = tid & 31;
  const int r0 = p.k0 + NB + blockIdx.x * PR;   // this CTA's first row below the diagonal block
  const bool rows = r0 < p.Dp;
  bool over = false;   // a pivot that isn't positive, or an element of L not below 1: not positive definite
  {
    const int64_t* col0 = p.fix + static_cast<int64_t>(p.k0) * p.Dp;
    // all of a thread's loads in flight at once
    constexpr int ND = (NB * NB + P_THREADS - 1) / P_THREADS, NX = (NB * PR + P_THREADS - 1) / P_THREADS;
    int64_t d[ND], x[NX];
#pragma unroll
    for (int i = 0; i < ND; ++i) {
      const int e = tid + i * P_THREADS, c = e >> 6, r = e & 63;
      d[i] = e < NB * NB && r >= c ? col0[static_cast<int64_t>(c) * p.Dp + p.k0 + r] : 0;
    }
#pragma unroll
    for (int i = 0; i < NX; ++i) {
      const int e = tid + i * P_THREADS;
      x[i] = e < NB * PR && rows ? col0[static_cast<int64_t>(e >> 5) * p.Dp + r0 + (e & 31)] : 0;
    }
#pragma unroll
    for (int i = 0; i < ND; ++i) {
      const int e = tid + i * P_THREADS;
      if (e < NB * NB) a[(e & 63) * PLD + (e >> 6)] = d[i];
    }
#pragma unroll
    for (int i = 0; i < NX; ++i) {
      const int e = tid + i * P_THREADS;
      if (e < NB * PR) a[(NB + (e & 31)) * PLD + (e >> 5)] = x[i];
    }
    if (tid < NB) mbar_init(smem_u32(done + tid), 1);
    if (tid == 0) *abort_flag = 0;
  }
  __syncthreads();
  if (tid < P_DOT) {
    const int r = tid / PL, h = tid % PL;
    const int2* row = pk + r * PLD;
    Dot acc;              // this lane's share of column j's dot product
    const int first = (tid >> 5) * (32 / PL);   // the warp's first row
#pragma unroll 1
    for (int j = 0; j < NB; ++j) {
      Dot next;
      if (r > j) {
        if (j > 0 && (j - 1) % PL == h) acc.add(row[j - 1], pk[j * PLD + j - 1]);
        const int past = PL * (j + 1 - first);   // lanes of the rows up to j
        const unsigned live = past > 0 ? 0xFFFFFFFFu << past : 0xFFFFFFFFu;
        int64_t sum = acc.sum();
#pragma unroll
        for (int o = PL / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(live, sum, o);
        if (h == 0) cs[r] = a[r * PLD + j] - sum;
        if (j + 1 < NB) {
          const int2* ln = pk + (j + 1) * PLD;
#pragma unroll 4
          for (int k = h; k < j; k += PL) next.add(row[k], ln[k]);
        }
      }
      acc = next;
      chain_sync();   // pivot j
      chain_sync();   // column j
    }
  } else if (tid < P_SCALE) {
    const int r = tid - P_DOT;
#pragma unroll 1
    for (int j = 0; j < NB; ++j) {
      chain_sync();   // pivot j
      if (r > j) {
        a[r * PLD + j] = scale_col(cs[r], ys[j], es[j], over, pk[r * PLD + j]);
      }
      chain_sync();   // column j
    }
  } else if (tid < P_CHAIN) {
    int64_t d0 = a[lane * PLD + lane], d1 = a[(lane + 32) * PLD + lane + 32];   // diagonal elements lane, lane + 32
#pragma unroll 1
    for (int j = 0; j < NB; ++j) {
      if (j > 0) {
        Dot q0, q1;
        const int2 l0 = pk[lane * PLD + j - 1], l1 = pk[(lane + 32) * PLD + j - 1];
        q0.add(l0, l0);
        q1.add(l1, l1);
        d0 -= lane >= j ? q0.square() : 0;
        d1 -= lane + 32 >= j ? q1.square() : 0;
      }
      int64_t d = __shfl_sync(0xffffffffu, j < 32 ? d0 : d1, j & 31);
      if (d <= 0) {
        over = true;
        d = int64_t{1} << 61;   // keep the remaining arithmetic in range; the caller reports NOT_SPD
      }
      uint64_t y;
      int e;
      pivot_rsqrt(d, y, e);
      if (lane == 0) {
        ys[j] = y;
        es[j] = e;
      }
      chain_sync();   // pivot j
      // sqrt(d) = d / sqrt(d); the chain reads no diagonal element of L
      if (lane == 0) a[j * PLD + j] = static_cast<int64_t>((static_cast<__int128>(d) * y) >> (61 - e));
      chain_sync();   // column j
      if (lane == 0) mbar_arrive(smem_u32(done + j));
    }
  } else {
    const int t = tid - P_CHAIN, h = t % PL, r = NB + t / PL;
    int2* row = pk + r * PLD;
    const WaitCtx wc{abort_flag, p.status, p.wait_limit_ns};
#pragma unroll 1
    for (int j = 0; j < NB; ++j) {
      if (!__all_sync(0xffffffffu, mbar_wait(smem_u32(done + j), 0, wc, 61, j))) break;
      const int2* ln = pk + j * PLD;
      Dot acc;
#pragma unroll 4
      for (int k = h; k < j; k += PL) acc.add(row[k], ln[k]);
      int64_t sum = acc.sum();
#pragma unroll
      for (int o = PL / 2; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      int2 packed;
      const int64_t l = scale_col(a[r * PLD + j] - sum, ys[j], es[j], over, packed);
      __syncwarp();
      if (h == 0) {
        row[j] = packed;
        a[r * PLD + j] = l;
      }
      __syncwarp();
    }
  }
  __syncthreads();
  if (tid == 0 && *abort_flag) atomicOr(p.flag, 2);
  if (over) atomicOr(p.flag, FLAG_NOT_SPD);
  if (blockIdx.x == 0) {
    int64_t* dst = p.diag + static_cast<int64_t>(p.k0 / NB) * (NB * NB);   // by columns
    for (int e = tid; e < NB * NB; e += P_THREADS) dst[e] = (e & 63) >= (e >> 6) ? a[(e & 63) * PLD + (e >> 6)] : 0;
  }
  if (!rows) return;
  for (int e = tid; e < NB * PR; e += P_THREADS)
    p.fix[static_cast<int64_t>(p.k0 + (e >> 5)) * p.Dp + r0 + (e & 31)] = a[(NB + (e & 31)) * PLD + (e >> 5)];
  if (tid < 256) {
    // slices: warp w takes the 8 columns 8 w .. of the 32 rows; a row's exponent from all 64
    const int kc = tid >> 5;
    const int64_t* row = a + (NB + lane) * PLD;
    uint64_t mx = 0;
#pragma unroll 16
    for (int k = 0; k < NB; ++k) mx |= static_cast<uint64_t>(SliceSrc<int64_t>::mag(row[k]));   // top bit of the max
    const int E = SliceSrc<int64_t>::exp_of(mx);
    if (kc == 0) p.exps[r0 + lane] = E;
    int64_t xi[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) xi[i] = SliceSrc<int64_t>::fixed(row[kc * 8 + i], E);
    store_digits8(xi, p.op + sl_offset(kc >> 2, p.n_t, r0 + lane, kc & 3));
  }
}

// Inverse I of L's 128 x 128 diagonal blocks, fp64.  The factor is stored by columns and leaves the other half of
// its array free: I_ij goes to [i][j], where column i has no L (the 64 x 64 blocks on the diagonal are
// L's in `diag`).  One CTA per 8 columns of a block; thread (column, row group): right-looking substitution with its
// rows in registers.  The CTAs of all blocks' first columns, which have the longest chains, come first, and load only
// what they need: 117 -> 62 us at 1536, 257 -> 151 at 5120.
constexpr int IC = 8;
constexpr int IG = 256 / IC;   // row groups
constexpr int INV_SMEM = (TB * (TB + 1) + 2 * IC + TB) * 8;
__global__ void __launch_bounds__(256) inverse_kernel(const int64_t* fix, const int64_t* __restrict__ diag,
                                                      int Dp, double* inv) {
  extern __shared__ double sm[];
  double* l = sm;                        // by columns, [c][TB + 1]
  double* xs = sm + TB * (TB + 1);       // the current row of the solution, twice
  double* rd = xs + 2 * IC;                  // reciprocals of the diagonal
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.x, c0 = blockIdx.y * IC, tid = threadIdx.x;   // the first columns, most of the work, first
  constexpr double k63 = 1.0842021724855044e-19;   // 2^-63
  for (int e = tid; e < TB * TB; e += 256) {
    const int c = e >> 7, r = e & 127;
    if (r < c || c < c0) continue;
    int64_t v;
    if ((c >> 6) == (r >> 6)) v = diag[(static_cast<int64_t>(2 * b + (c >> 6)) << 12) + ((c & 63) << 6) + (r & 63)];
    else v = fix[static_cast<int64_t>(b * TB + c) * Dp + b * TB + r];
    const double d = static_cast<double>(v) * k63;
    l[c * (TB + 1) + r] = d;
    if (c == r) rd[c] = 1.0 / d;
  }
  __syncthreads();
  const int col = tid % IC, g = tid / IC;
  double x[TB / IG];
#pragma unroll
  for (int m = 0; m < TB / IG; ++m) x[m] = g + IG * m == c0 + col ? 1.0 : 0.0;
#pragma unroll
  for (int k = 0; k < TB; ++k) {
    if (k < c0) continue;
    double* xk = xs + (k & 1) * IC;   // alternating: one barrier a step
    if (g == k % IG) {
      x[k / IG] *= rd[k];
      xk[col] = x[k / IG];
    }
    __syncthreads();
    const double v = xk[col];
#pragma unroll
    for (int m = k / IG; m < TB / IG; ++m)
      if (g + IG * m > k) x[m] = fma(-l[k * (TB + 1) + g + IG * m], v, x[m]);
  }
#pragma unroll
  for (int m = 0; m < TB / IG; ++m) {
    const int i = g + IG * m, j = c0 + col;
    if (i >= j) inv[static_cast<int64_t>(b * TB + i) * Dp + b * TB + j] = x[m];
  }
}

// *out += sum x^2
__device__ __forceinline__ void block_add(double s, double* out) {
  __shared__ double red[8];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int i = 1; i < 8; ++i) s += red[i];
    atomicAdd(out, s);
  }
}

__global__ void __launch_bounds__(256) sumsq_kernel(const double* __restrict__ x, int64_t n, double* out) {
  pdl_wait();
  pdl_trigger();
  double s = 0.0;
  const int64_t step = static_cast<int64_t>(gridDim.x) * 256;
  for (int64_t e = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x; e < n; e += step) s = fma(x[e], x[e], s);
  block_add(s, out);
}

// dW[i][j] = z[j][i] 2^(-t_i), through 32 x 32 tiles, a CTA every gridDim.y-th of its rows; *out += ||dW||^2 (before
// the fp32 rounding).
__global__ void __launch_bounds__(256) finish_kernel(const double* __restrict__ z, int D, int Dp, int n,
                                                     const int32_t* __restrict__ t, float* __restrict__ dW,
                                                     double* out) {
  __shared__ float tile[32][33];
  pdl_wait();
  pdl_trigger();
  const int i0 = blockIdx.x * 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double s = 0.0;
  for (int j0 = blockIdx.y * 32; j0 < n; j0 += gridDim.y * 32) {
    for (int jj = w; jj < 32; jj += 8) {
      double v = 0.0;
      if (j0 + jj < n && i0 + lane < D) v = z[static_cast<int64_t>(j0 + jj) * Dp + i0 + lane] * pow2d(-t[i0 + lane]);
      s = fma(v, v, s);
      tile[jj][lane] = static_cast<float>(v);
    }
    __syncthreads();
    for (int ii = w; ii < 32; ii += 8)
      if (i0 + ii < D && j0 + lane < n) dW[static_cast<int64_t>(i0 + ii) * n + j0 + lane] = tile[lane][ii];
    __syncthreads();
  }
  block_add(s, out);
}

size_t align256(size_t b) { return (b + 255) & ~static_cast<size_t>(255); }

struct SolveWs {
  int32_t Dp, np, kn;      // D to 128, d_out to 64 and to 32
  int32_t win;             // rows of a window of the substitutions
  int32_t t_d, t_n;        // 64-row tiles of the ops over D (one spare: a 128-row tile may start with the
                           // last) and over d_out
  uint8_t *op_a, *op_b;    // op_b (W) and the factor share their memory: X W is formed first
  int64_t* fix;
  double* B;               // by columns [d_out][Dp]: X W, then Y, then Z
  uint8_t *op_panel, *op_s, *op_n, *op_i, *op_it;
  int64_t* diag;
  int32_t *t, *u, *ew, *ea, *en, *eb, *es, *ei, *eit;
  double* scal;            // [0] ||Y||^2, [1] ||dW||^2, [2] tr(W^T S W)
  int* flag;
  size_t bytes;
};

SolveWs carve(void* ws, int D, int d_out) {
  SolveWs w;
  w.Dp = (D + TB - 1) / TB * TB;
  w.np = (d_out + 63) / 64 * 64;
  w.kn = (d_out + 31) / 32 * 32;
  w.t_d = w.Dp / 64 + 1;
  w.t_n = w.np / 64;
  uint8_t* p = static_cast<uint8_t*>(ws);
  auto take = [&](size_t bytes) {
    uint8_t* r = p;
    p += align256(bytes);
    return r;
  };
  const size_t Dp = w.Dp, chunk_d = static_cast<size_t>(w.t_d) * SL_TILE;
  const size_t chunk_n = static_cast<size_t>(w.t_n) * SL_TILE;
  const size_t ka = Dp > static_cast<size_t>(w.kn) ? Dp : w.kn;
  w.op_a = take(ka / SL_K * chunk_d);
  const size_t opb = Dp / SL_K * chunk_n, fix = Dp * Dp * 8;
  w.op_b = take(opb > fix ? opb : fix);
  w.fix = reinterpret_cast<int64_t*>(w.op_b);
  w.B = reinterpret_cast<double*>(take(Dp * static_cast<size_t>(d_out) * 8));
  w.op_panel = take(NB / SL_K * chunk_d);
  w.win = w.Dp > SB && Dp / 256 * static_cast<size_t>(w.t_n) >= SB_TILES ? SB : w.Dp;
  const bool one = w.win == w.Dp;
  w.op_s = take((one ? TB : SB) / SL_K * chunk_n);
  w.op_n = one ? w.op_a : take(SB / SL_K * chunk_d);
  w.op_i = take(TB / SL_K * chunk_d);
  w.op_it = take(TB / SL_K * chunk_d);
  w.diag = reinterpret_cast<int64_t*>(take(Dp * NB * 8));
  w.t = reinterpret_cast<int32_t*>(take(Dp * 4));
  w.u = reinterpret_cast<int32_t*>(take(Dp * 4));
  w.ew = reinterpret_cast<int32_t*>(take(static_cast<size_t>(d_out) * 4));
  w.ea = reinterpret_cast<int32_t*>(take((Dp + w.win - 1) / w.win * Dp * 4));
  w.en = reinterpret_cast<int32_t*>(take(w.win / TB * Dp * 4));
  w.eb = reinterpret_cast<int32_t*>(take(static_cast<size_t>(w.np) * 4));
  w.es = reinterpret_cast<int32_t*>(take(static_cast<size_t>(w.np) * 4));
  w.ei = reinterpret_cast<int32_t*>(take(Dp * 4));
  w.eit = reinterpret_cast<int32_t*>(take(Dp * 4));
  w.scal = reinterpret_cast<double*>(take(256));
  w.flag = reinterpret_cast<int*>(w.scal + 4);
  w.bytes = static_cast<size_t>(p - static_cast<uint8_t*>(ws));
  return w;
}

// One segment: rows x ks values, k padded to k_pad with zeros.
SliceParams slice(const void* src, int64_t ld, int rows, int ks, int k_pad, int n_t, uint8_t* op, int32_t* exps) {
  SliceParams p{};
  p.src = src;
  p.ld = ld;
  p.rows = rows;
  p.ks = ks;
  p.k_pad = k_pad;
  p.n_t = n_t;
  p.op = op;
  p.exps = exps;
  return p;
}

// grid_rows: rows of a segment in the op (multiples of 8, those past the valid ones are zeroed).
template <typename T, int TRI = SL_FULL, bool SCALED = false>
cudaError_t slice_rows(const SliceParams& p, int grid_rows, int n_seg, cudaStream_t s) {
  const dim3 grid(grid_rows / 8, n_seg);
  return launch_pdl(slice_rows_kernel<T, TRI, SCALED>, grid, dim3(p.k_pad > 512 ? 512 : 256), 0, s, p);
}

template <typename T, int TRI = SL_FULL, bool SCALED = false>
cudaError_t slice_cols(const SliceParams& p, int grid_rows, int n_seg, int sms, cudaStream_t s) {
  dim3 grid((grid_rows + 31) / 32, n_seg);
  const int warps = p.k_pad > 128 ? 32 : 8, most = p.k_pad / 8 / warps;   // parts with work for every warp
  const int fill = 2 * sms / static_cast<int>(grid.x * grid.y);
  grid.z = fill < 1 || most < 1 ? 1 : (fill < most ? fill : most);
  return launch_pdl(slice_cols_kernel<T, TRI, SCALED>, grid, dim3(32 * warps), 0, s, p);
}

}  // namespace

size_t ls_solve_ws_bytes(int32_t D, int32_t d_out) { return carve(nullptr, D, d_out).bytes; }

ispa_status run_ls_solve(int32_t D, const float* gram, const float* W, int32_t d_out, double lambda,
                         float* dW, double* eps_out, void* ws, cudaStream_t s) {
  const SolveWs w = carve(ws, D, d_out);
  const int Dp = w.Dp, nb = Dp / TB;
  const int64_t ldg = 2 * static_cast<int64_t>(D);
  const int64_t chunk_d = static_cast<int64_t>(w.t_d) * SL_TILE, chunk_n = static_cast<int64_t>(w.t_n) * SL_TILE;
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
#define ISPA_CK(x)                            \
  do {                                        \
    if ((x) != cudaSuccess) return ISPA_ERR_CUDA; \
  } while (0)
  SlGemm base{};
  base.status = device_status_ptr();
  if (!base.status) return ISPA_ERR_CUDA;
  base.flag = w.flag;
  base.wait_limit_ns = wait_limit_ns();
  base.n_split = 1;
  ISPA_CK(set_smem_limit_once(reinterpret_cast<const void*>(inverse_kernel), INV_SMEM));
  ISPA_CK(set_smem_limit_once(reinterpret_cast<const void*>(panel_kernel), PANEL_SMEM));
  ISPA_CK(cudaMemsetAsync(w.scal, 0, 256, s));
  ISPA_CK(launch_pdl(equil_kernel, dim3(((Dp > d_out ? Dp : d_out) + 255) / 256), dim3(256), 0, s, gram, D, Dp, lambda,
                     w.t, w.u, d_out, w.ew, w.flag));
  auto col_grid = [&](int cols) { return dim3((cols + U_COLS - 1) / U_COLS, (D + U_ROWS - 1) / U_ROWS); };
  ISPA_CK(launch_pdl(col_exp_kernel<false>, col_grid(D), dim3(256), 0, s, gram + D, ldg, D, D,
                     static_cast<const int32_t*>(w.t), -1, w.u));
  ISPA_CK(launch_pdl(col_exp_kernel<true>, col_grid(d_out), dim3(256), 0, s, W, static_cast<int64_t>(d_out), D, d_out,
                     static_cast<const int32_t*>(w.u), 1, w.ew));

  // tr(W^T S W) = sum_ij S_ij (W W^T)_ij: W's rows sliced over d_out
  ISPA_CK(slice_rows<float>(slice(W, d_out, D, d_out, w.kn, w.t_d, w.op_a, w.ea), Dp, 1, s));
  {
    SlGemm p = base;
    p.a = p.b = w.op_a;
    p.a_chunk = p.b_chunk = chunk_d;
    p.ea = p.eb = w.ea;
    // the sum over the contraction index too can be cut, into up to eight pieces of at least two flushes; with eight
    // waves of tiles the last one's idle SMs are a small part of the whole anyway
    const int mt = Dp / 128, chunks = w.kn / SL_K, pieces = chunks / (2 * SG_FLUSH);
    p.n_split = pieces < 1 || mt * (mt + 1) > 8 * sms ? 1 : (pieces > 8 ? 8 : pieces);
    p.n_tiles = mt * (mt + 1) * p.n_split;
    p.n_chunks = chunks;
    p.row_end = D;
    p.ld = ldg;
    p.sym = gram + static_cast<int64_t>(D) * ldg + D;
    p.dot = w.scal + 2;
    ISPA_CK(launch_slice_gemm<SL_DOT>(p, sms, s));
  }
  // B = 2^-t X W = 2^-t (X 2^-u) (2^u W)
  {
    SliceParams x = slice(gram + D, ldg, D, D, Dp, w.t_d, w.op_a, w.ea);
    SliceParams y = slice(W, d_out, d_out, D, Dp, w.t_n, w.op_b, w.eb);
    x.k_exp = y.k_exp = w.u;
    x.k_sign = -1;
    y.k_sign = 1;
    y.r_max = w.ew;
    ISPA_CK((slice_rows<float, SL_FULL, true>(x, Dp, 1, s)));
    ISPA_CK((slice_cols<float, SL_FULL, true>(y, w.np, 1, sms, s)));
  }
  {
    SlGemm p = base;
    p.a = w.op_a;
    p.b = w.op_b;
    p.a_chunk = chunk_d;
    p.b_chunk = chunk_n;
    p.ea = w.ea;
    p.eb = w.eb;
    p.n_mt = Dp / 128;
    p.n_nt = w.np / 64;
    p.n_tiles = p.n_mt * p.n_nt;
    p.n_chunks = Dp / SL_K;
    p.row_end = Dp;
    p.col_end = d_out;
    p.ld = Dp;
    p.out = w.B;
    p.row_exp = w.t;
    ISPA_CK(launch_slice_gemm<SL_STORE>(p, sms, s));
  }
  // Cholesky
  ISPA_CK(launch_pdl(form_kernel, dim3(Dp, (Dp + 255) / 256), dim3(256), 0, s, gram, D, Dp, lambda,
                     static_cast<const int32_t*>(w.t), w.fix, w.flag));
  for (int k0 = 0; k0 < Dp; k0 += NB) {
    const int rest = Dp - k0 - NB;
    const PanelParams pp{w.fix, w.diag, Dp, k0, w.op_panel, w.t_d, w.ea, w.flag, base.status, base.wait_limit_ns};
    ISPA_CK(launch_pdl(panel_kernel, dim3(rest > 0 ? rest / PR : 1), dim3(P_THREADS), PANEL_SMEM, s, pp));
    if (rest <= 0) break;
    SlGemm p = base;
    p.a = p.b = w.op_panel;
    p.a_chunk = p.b_chunk = chunk_d;
    p.ea = p.eb = w.ea;
    p.row0 = p.col0 = k0 + NB;
    const int mt = (rest + 127) / 128;
    p.n_tiles = mt * (mt + 1);
    p.n_chunks = NB / SL_K;
    p.row_end = Dp;
    p.ld = Dp;
    p.out = w.fix;
    ISPA_CK(launch_slice_gemm<SL_CHOL>(p, sms, s));
  }
  double* inv = reinterpret_cast<double*>(w.fix);
  ISPA_CK(launch_pdl(inverse_kernel, dim3(nb, TB / IC), dim3(256), INV_SMEM, s, static_cast<const int64_t*>(w.fix),
                     static_cast<const int64_t*>(w.diag), Dp, inv));
  const int64_t ld = Dp;
  {
    // I for the forward steps (rows i), I^T for the backward ones (rows j)
    SliceParams q = slice(inv, ld, TB, TB, TB, w.t_d, w.op_i, w.ei);
    q.z_src = TB * (ld + 1);
    q.z_rows = TB;
    ISPA_CK((slice_rows<double, SL_LOWER>(q, TB, nb, s)));
    q.op = w.op_it;
    q.exps = w.eit;
    ISPA_CK((slice_cols<double, SL_UPPER>(q, TB, nb, sms, s)));
  }

  // B's rows [r0, r0 + n) sliced, over all columns
  auto slice_b = [&](int r0, int n) {
    return slice_rows<double>(slice(w.B + r0, Dp, d_out, n, n, w.t_n, w.op_s, w.es), w.np, 1, s);
  };
  SlGemm sub = base;
  sub.b = w.op_s;
  sub.a_chunk = chunk_d;
  sub.b_chunk = chunk_n;
  sub.eb = w.es;
  sub.n_nt = w.np / 64;
  sub.col_end = d_out;
  sub.ld = Dp;
  sub.out = w.B;
  auto rows = [](SlGemm p, const uint8_t* op, const int32_t* exps, int r0, int r1, int k) {
    p.a = op;
    p.ea = exps;
    p.row0 = r0;
    p.row_end = r1;
    p.n_mt = (r1 - r0) / 128;
    p.n_tiles = p.n_mt * p.n_nt;
    p.n_chunks = k / SL_K;
    return p;
  };
  // One block step of a substitution: block row k of B becomes inv(L_kk) (or its transpose) times itself, and
  // rows [r0, r1) of its window lose their product with it.
  auto step = [&](int k, const uint8_t* op_i, const int32_t* e_i, int r0, int r1) -> cudaError_t {
    cudaError_t e = slice_b(k * TB, TB);
    if (e == cudaSuccess) e = launch_slice_gemm<SL_STORE>(rows(sub, op_i, e_i, k * TB, (k + 1) * TB, TB), sms, s);
    if (e != cudaSuccess || r0 >= r1) return e;
    if ((e = slice_b(k * TB, TB)) != cudaSuccess) return e;
    const int zc = k % (w.win / TB);
    return launch_slice_gemm<SL_SUB>(rows(sub, w.op_n + static_cast<int64_t>(zc) * (TB / SL_K) * chunk_d,
                                          w.en + static_cast<int64_t>(zc) * Dp, r0, r1, TB), sms, s);
  };
  // Rows [r0, r1) outside of window z lose their product with all of it.
  auto far = [&](int z, int r0, int r1) -> cudaError_t {
    const int n = Dp - z * w.win < w.win ? Dp - z * w.win : w.win;
    const cudaError_t e = slice_b(z * w.win, n);
    if (e != cudaSuccess) return e;
    return launch_slice_gemm<SL_SUB>(rows(sub, w.op_a + static_cast<int64_t>(z) * (w.win / SL_K) * chunk_d,
                                          w.ea + static_cast<int64_t>(z) * Dp, r0, r1, n), sms, s);
  };
  // L's values for both: blocks of 128 columns (forward; rows: backward) within the windows, the window's width outside
  const int n_win = (Dp + w.win - 1) / w.win;
  SliceParams near_l = slice(w.fix, ld, Dp, TB, TB, w.t_d, w.op_n, w.en);
  SliceParams far_l = slice(w.fix, ld, Dp, w.win, w.win, w.t_d, w.op_a, w.ea);
  near_l.rows_total = far_l.ks_total = Dp;
  near_l.z_k = TB;
  near_l.win = far_l.z_k = w.win;
  near_l.z_exp = far_l.z_exp = Dp;
  // forward
  near_l.lower = far_l.lower = 1;
  near_l.z_src = TB * ld;
  far_l.z_src = w.win * ld;
  if (nb > 1) ISPA_CK(slice_cols<int64_t>(near_l, w.win, nb, sms, s));
  if (n_win > 1) ISPA_CK(slice_cols<int64_t>(far_l, Dp, n_win - 1, sms, s));
  for (int z = 0; z < n_win; ++z) {
    const int k1 = (z + 1) * (w.win / TB) < nb ? (z + 1) * (w.win / TB) : nb;
    for (int k = z * (w.win / TB); k < k1; ++k) ISPA_CK(step(k, w.op_i, w.ei, (k + 1) * TB, k1 * TB));
    if (k1 < nb) ISPA_CK(far(z, k1 * TB, Dp));
  }
  const int64_t nB = static_cast<int64_t>(Dp) * d_out;
  const unsigned dot_grid = static_cast<unsigned>(nB / 2048 < 1 ? 1 : (nB / 2048 < 8 * sms ? nB / 2048 : 8 * sms));
  ISPA_CK(launch_pdl(sumsq_kernel, dim3(dot_grid), dim3(256), 0, s, static_cast<const double*>(w.B), nB, w.scal));
  // backward
  near_l.lower = far_l.lower = -1;
  near_l.z_src = TB;
  far_l.z_src = w.win;
  if (nb > 1) ISPA_CK(slice_rows<int64_t>(near_l, w.win, nb, s));
  if (n_win > 1) ISPA_CK(slice_rows<int64_t>(far_l, Dp, n_win, s));
  for (int z = n_win - 1; z >= 0; --z) {
    const int k1 = (z + 1) * (w.win / TB) < nb ? (z + 1) * (w.win / TB) : nb;
    for (int k = k1 - 1; k >= z * (w.win / TB); --k) ISPA_CK(step(k, w.op_it, w.eit, z * w.win, k * TB));
    if (z > 0) ISPA_CK(far(z, 0, z * w.win));
  }
  // no more CTAs than fill the chip: each adds to the one sum
  const unsigned fx = (D + 31) / 32, fy = (d_out + 31) / 32, fmax = fx < 8u * sms ? 8u * sms / fx : 1u;
  ISPA_CK(launch_pdl(finish_kernel, dim3(fx, fy < fmax ? fy : fmax), dim3(256), 0, s,
                     static_cast<const double*>(w.B), D, Dp, d_out, static_cast<const int32_t*>(w.t), dW, w.scal + 1));
  struct {
    double scal[4];
    int flag;
  } h;
  ISPA_CK(cudaMemcpyAsync(&h, w.scal, 4 * sizeof(double) + sizeof(int), cudaMemcpyDeviceToHost, s));
  ISPA_CK(cudaStreamSynchronize(s));
#undef ISPA_CK
  if (eps_out) *eps_out = h.scal[2] - h.scal[0] - lambda * h.scal[1];
  if (h.flag & 2) return ISPA_ERR_TIMEOUT;
  return h.flag ? ISPA_ERR_NOT_SPD : ISPA_OK;
}

}  // namespace ispa
