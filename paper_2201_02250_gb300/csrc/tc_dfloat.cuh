// Double-float tile products on the tensor cores: A(128 x 64) B(64 x 64) of double-float values, computed with
// BF16 x BF16 -> FP32 tcgen05 MMAs.
//
// Method (an error-free splitting in the manner of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix multiplication and its
// applications", Numer. Algorithms 2012): every row of A is scaled by a power of two 2^eA_r >= its
// largest magnitude, every column of B by 2^eB_c, and each scaled value y in [-1, 1] is written as seven
// base-256 digits, y = sum_s t_s 256^-(s+1) with integers |t_0| <= 256, |t_s| <= 128 (s > 0), obtained by
// repeated rounding to the nearest integer (each step is exact in double-float arithmetic).  Digit s
// is stored as the BF16 value t_s 2^(-8 s), which is exact (at most 8 significant bits).  The product
// of digit i of A and digit j of B then has the natural weight 2^(-8 (i + j)), and the 28 digit pairs
// with i + j <= 6 are accumulated by the tensor cores in seven FP32 accumulator blocks, one per weight.
// Block d sums d + 1 pairs over 64 terms, at most 9 x 2^20 units of its weight, below 2^24, so FP32
// accumulates every block exactly whatever the order.  The result, 2^(eA_r + eB_c - 16) times the sum
// of the blocks, is formed in double-float.  Its error is about 2^-52 of max_k |A_rk| max_k |B_kc|
// (seven digits: the dropped pairs weigh 2^-56 and less), which stays below the double-float product's
// error bound of a few 2^-47 (|A| |B|)_rc unless the largest entries of the row and of the column sit
// at different k and exceed their partners by more than about 2^5.
//
// Shared memory: A digits 7 x 16 KiB, B digits 7 x 8 KiB (168 KiB), K-major canonical layout
// (tc_sm100.cuh).  TMEM: 7 accumulator blocks x 64 columns (512 columns allocated: one CTA per SM).
#pragma once

#include <cuda_bf16.h>

#include "dfloat.cuh"
#include "tc_sm100.cuh"

namespace a2ls {
namespace tcdf {

constexpr int TM = 128, TN = 64, TK = 64;   // tile shape
constexpr int NDIG = 7;                      // base-256 digits per value
constexpr int NBLK = NDIG;                   // exact accumulator blocks, one per digit weight 0 .. 6
constexpr uint32_t A_DIGIT_BYTES = TM * TK * 2;
constexpr uint32_t B_DIGIT_BYTES = TN * TK * 2;
constexpr size_t SMEM_BYTES = (size_t)NDIG * (A_DIGIT_BYTES + B_DIGIT_BYTES);   // 172032
constexpr uint32_t TMEM_COLS = 512;
constexpr int THREADS = 512;                 // of the CTA that calls the functions of a tile below
constexpr long WAIT_LIMIT = 1L << 26;        // polls of the completion barrier before giving up

// 2^k as a float for k in [-126, 127]
__device__ __forceinline__ float pow2f(int k) { return __uint_as_float((uint32_t)(k + 127) << 23); }

// x 2^k for any k a sum of two scale exponents can be: two exact multiplications by powers of two (ldexpf
// takes a score of instructions, and the digit kernels need it for every value)
__device__ __forceinline__ dfloat df_scale(dfloat x, int k) {
  const int k1 = min(max(k, -126), 127), k2 = min(max(k - k1, -126), 127);
  const float f1 = pow2f(k1), f2 = pow2f(k2);
  return dfloat(__fmul_rn(__fmul_rn(x.hi, f1), f2), __fmul_rn(__fmul_rn(x.lo, f1), f2));
}

// The NDIG digits of y = x / 2^e (|y| <= 1), as the values t_s 2^(-8 s), exact in BF16.  y 2^56 as a 64-bit
// integer (the pair's two parts convert separately) plus 128 at every digit but the first has the digits
// plus 128 as its bytes, the first signed above them; a byte becomes a float by way of 2^23's mantissa.
// About 40 instructions where rounding digit by digit in double-float takes 90, and the split of an
// operand is on the critical chain of every block of the triangular solves (k_tcsolve.cu).
// A NaN or an infinity makes the first digit NaN, and with it every product of its row or column, so that the
// Rayleigh-Ritz step's test of its matrix sees it.
__device__ __forceinline__ void df_digits(dfloat x, int e, float (&d)[NDIG]) {
  const dfloat y = df_scale(x, 56 - e);
  const long long v = __float2ll_rn(y.hi) + __float2ll_rn(y.lo) + 0x0000808080808080ll;
  const uint32_t lo = (uint32_t)v, mid = (uint32_t)((unsigned long long)v >> 32);
  d[0] = __fmaf_rn(x.hi, 0.f, (float)(int)(v >> 48));   // NaN where x is not finite, which no integer can show
#pragma unroll
  for (int s = 1; s < NDIG; ++s) {
    const uint32_t byte = s < 3 ? (mid >> (8 * (2 - s))) & 0xffu : (lo >> (8 * (6 - s))) & 0xffu;
    d[s] = __fmul_rn(__fsub_rn(__uint_as_float(0x4b000000u | byte), 8388736.f), 1.f / (float)(1ull << (8 * s)));
  }
}

// digit s of eight consecutive values as 16 bytes of BF16
__device__ __forceinline__ uint4 pack_digits(const float (&d)[8][NDIG], int s) {
  __nv_bfloat162 p0 = __floats2bfloat162_rn(d[0][s], d[1][s]), p1 = __floats2bfloat162_rn(d[2][s], d[3][s]),
                 p2 = __floats2bfloat162_rn(d[4][s], d[5][s]), p3 = __floats2bfloat162_rn(d[6][s], d[7][s]);
  uint4 w;
  w.x = *reinterpret_cast<uint32_t*>(&p0);
  w.y = *reinterpret_cast<uint32_t*>(&p1);
  w.z = *reinterpret_cast<uint32_t*>(&p2);
  w.w = *reinterpret_cast<uint32_t*>(&p3);
  return w;
}

// exponent e with |v| < 2^e (0 for v = 0), at least -100: smaller values keep the digits above 2^-156
__device__ __forceinline__ int scale_exponent(float maxabs) {
  int e = 0;
  if (maxabs > 0.f) frexpf(maxabs, &e);
  return max(e, -100);
}

// The sum of the seven accumulator blocks: a_d is an integer of at most 9 x 2^20 times 2^(-8 d).  a_0 plus
// a_1 rounded to an integer is exact, so is what a_1 leaves plus a_2 (multiples of 2^-16 below 2^8); a_3
// joins with its rounding error, and the last three, in FP32, weigh 2^-32 of the first and less.  The pair
// is not normalised (|lo| may exceed ulp(hi) / 2).
__device__ __forceinline__ dfloat sum_blocks(float a0, float a1, float a2, float a3, float a4, float a5, float a6) {
  const float t1 = rintf(a1);
  const dfloat q = df_two_sum(__fadd_rn(__fsub_rn(a1, t1), a2), a3);
  const dfloat v = df_two_sum(__fadd_rn(a0, t1), q.hi);
  return dfloat(v.hi, __fadd_rn(v.lo, __fadd_rn(q.lo, __fadd_rn(a4, __fadd_rn(a5, a6)))));
}

struct Ctx {
  unsigned char* smem;   // SMEM_BYTES, 16-byte aligned
  uint64_t* bar;         // completion mbarrier (initialised with count 1)
  uint32_t tmem;         // TMEM base address (TMEM_COLS columns)
  uint32_t phase;        // parity of the next completion
  int* eA;               // shared, TM row exponents
  int* eB;               // shared, TN column exponents (of the B written last)
};

// A digits: rows [0, TM) x k [0, TK) of A(m, k) = fa(m, k) (zero outside): four threads per row.
template <class FA>
__device__ __forceinline__ void split_a(Ctx& c, FA fa) {
  const int tid = threadIdx.x, r = tid >> 2, h = tid & 3;
  dfloat v[16];
  float mx = 0.f;
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    v[q] = fa(r, h * 16 + q);
    mx = fmaxf(mx, fabsf(v[q].hi));
  }
  mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
  mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
  const int e = scale_exponent(mx);
  if (h == 0) c.eA[r] = e;
#pragma unroll
  for (int q8 = 0; q8 < 2; ++q8) {
    float dg[8][NDIG];
#pragma unroll
    for (int q = 0; q < 8; ++q) df_digits(v[q8 * 8 + q], e, dg[q]);
    const uint32_t off = tc::operand_offset(r, h * 16 + q8 * 8, TK);
#pragma unroll
    for (int s = 0; s < NDIG; ++s) *reinterpret_cast<uint4*>(c.smem + s * A_DIGIT_BYTES + off) = pack_digits(dg, s);
  }
}

// B digits: k [0, TK) x columns [0, TN) of B(k, n) = fb(k, n), stored as the K-major operand (n, k); column
// n = tid % 64, k eighth tid / 64.  red: shared scratch of 8 x TN floats.  In two parts, so that the loads can be
// in flight during the MMAs of another tile: load_b, and write_b once the B region is free.
template <class FB>
__device__ __forceinline__ void load_b(FB fb, dfloat (&v)[8]) {
  const int tid = threadIdx.x, n = tid & (TN - 1), qk = tid >> 6;
#pragma unroll
  for (int q = 0; q < 8; ++q) v[q] = fb(qk * 8 + q, n);
}
__device__ __forceinline__ void write_b(Ctx& c, const dfloat (&v)[8], float* red) {
  const int tid = threadIdx.x, n = tid & (TN - 1), qk = tid >> 6;
  float mx = 0.f;
#pragma unroll
  for (int q = 0; q < 8; ++q) mx = fmaxf(mx, fabsf(v[q].hi));
  red[qk * TN + n] = mx;
  __syncthreads();
  mx = 0.f;
#pragma unroll
  for (int q = 0; q < 8; ++q) mx = fmaxf(mx, red[q * TN + n]);
  const int e = scale_exponent(mx);
  if (qk == 0) c.eB[n] = e;
  float dg[8][NDIG];
#pragma unroll
  for (int q = 0; q < 8; ++q) df_digits(v[q], e, dg[q]);
  const uint32_t off = tc::operand_offset(n, qk * 8, TK);
#pragma unroll
  for (int s = 0; s < NDIG; ++s) *reinterpret_cast<uint4*>(c.smem + NDIG * A_DIGIT_BYTES + s * B_DIGIT_BYTES + off) = pack_digits(dg, s);
}

// After split_a and write_b by all threads (and their last product8 of an earlier tile): the 40 MMAs of the 28
// digit pairs, issued by thread 0.  Contains a barrier.
__device__ __forceinline__ void issue(Ctx& c) {
  tc::fence_proxy_async();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (threadIdx.x == 0) {
    const uint32_t a0 = tc::smem_u32(c.smem), b0 = a0 + NDIG * A_DIGIT_BYTES;
    // descriptors of the first K-chunk of digit plane 0; the others differ only in the start address
    // field (address / 16, low bits), which no offset here carries out of
    const uint64_t ad0 = tc::smem_desc(a0, 128, TK * 16), bd0 = tc::smem_desc(b0, 128, TK * 16);
    // The B digit planes are consecutive 64-row groups of one K-major operand, so an MMA with A digit i
    // and B digits j0 .. j0 + nj - 1 (N = 64 nj <= 256) writes pair (i, j) into block i + j, the
    // block of its weight.  The two MMAs of digit 0 write all seven blocks first; the others add.
#pragma unroll
    for (int i = 0; i < NDIG; ++i)
#pragma unroll
      for (int j0 = 0; j0 < NDIG - i; j0 += 4) {
        const int nj = (NDIG - i - j0) < 4 ? (NDIG - i - j0) : 4;
        const uint32_t idesc = tc::idesc_bf16_f32(TM, TN * nj);
#pragma unroll
        for (int kk = 0; kk < TK / 16; ++kk)
          tc::mma_bf16(c.tmem + (i + j0) * TN, ad0 + ((i * A_DIGIT_BYTES + kk * 256) >> 4),
                       bd0 + ((j0 * B_DIGIT_BYTES + kk * 256) >> 4), idesc, (i == 0 && kk == 0) ? 0u : 1u);
      }
    tc::commit(c.bar);
  }
  __syncwarp();
}

// A bounded wait by every thread for the MMAs issued last.  Returns false (on every thread) if they did not
// complete.
__device__ __forceinline__ bool wait(Ctx& c) {
  const bool ok = tc::mbar_wait_bounded(c.bar, c.phase, WAIT_LIMIT);
  c.phase ^= 1u;
  tc::fence_after_sync();
  return __syncthreads_and(ok) != 0;
}

// Columns [col, col + 8) of the tile product for this thread's row 32 (warp % 4) + lane, handed to put(column,
// value) unnormalised; eB: the column exponents of the tile's B.  A single multiplication by the power of two
// where it has one (df_scale's result, in a third of its instructions).
template <class F>
__device__ __forceinline__ void product8(const Ctx& c, const int* eB, int col, F put) {
  const int w4 = (threadIdx.x >> 5) & 3;
  const int em = c.eA[w4 * 32 + (threadIdx.x & 31)] - 16;
  const uint32_t addr = c.tmem + ((uint32_t)(w4 * 32) << 16) + col;
  __syncwarp();   // the loads are warp-wide, and the values' scaling and put may have diverged
  float acc[NBLK][8];
#pragma unroll
  for (int g = 0; g < NBLK; ++g) tc::tmem_ld8(addr + g * TN, acc[g]);
  tc::tmem_wait_ld();
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const dfloat sum = sum_blocks(acc[0][q], acc[1][q], acc[2][q], acc[3][q], acc[4][q], acc[5][q], acc[6][q]);
    const int e = em + eB[col + q];
    if (e >= -126 && e <= 127) {
      const float f = pow2f(e);
      put(col + q, dfloat(__fmul_rn(sum.hi, f), __fmul_rn(sum.lo, f)));
    } else {
      put(col + q, df_scale(sum, e));
    }
  }
}

// A tile product is turned from one row a thread into one row a warp for its memory accesses in a staging
// buffer of TM rows x 32 columns.
constexpr int SUB_LD = 33;   // staging row stride in double-float values (odd: spreads the banks)
constexpr size_t STAGE_BYTES = (size_t)TM * SUB_LD * sizeof(dfloat);
__device__ __forceinline__ void stage_half(const Ctx& c, const int* eB, int half, dfloat* S) {
  const int warp = threadIdx.x >> 5, m = (warp & 3) * 32 + (threadIdx.x & 31);
  product8(c, eB, half * 32 + (warp >> 2) * 8, [&](int col, dfloat v) { S[m * SUB_LD + col - half * 32] = v; });
}

}  // namespace tcdf
}  // namespace a2ls
