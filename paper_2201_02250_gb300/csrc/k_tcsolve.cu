// Double-float block triangular solves of the local eigensolves on the tensor cores.
//
// The operator of the local eigenproblem (Eq. 3.1) is applied through the double-float LU of the
// splitting A~_ii: X <- inv(U) inv(L) X for a block of p <= 32 columns.  In the block-inverted storage
// both sweeps are sequences of 64 x 64 tile products (k_dense.cu).  Here each product runs as
// BF16 x BF16 -> FP32 tcgen05 MMAs on base-256 digit expansions (the scheme of tc_dfloat.cuh):
//   * after the factorisation every 64 x 64 factor tile a sweep reads (the off-diagonal tiles inside
//     the envelope of L and U, and the two inverted triangles of each diagonal tile) is split once
//     into seven BF16 digit planes with one power-of-two scale per row (k_factor_digits);
//   * a sweep keeps, for every finished 64-row block of X, its seven digit planes with one scale per
//     column in a scratch array, so that each later block reads digits instead of splitting again;
//   * per 64-row block: the tile products of its panel, X_b - panel, then the product with the inverted
//     diagonal triangle, whose result is X_b.
//
// MMA shape.  Two digit planes of A (rows of the factor tile) are adjacent and form one operand of M = 128
// rows, the digit planes of B are adjacent groups of 32 rows (columns of X), and the accumulator blocks
// of 32 TMEM columns are adjacent by weight: with A planes 2t, 2t + 1 and B planes 0 .. 7 - 2t, one MMA of
// N = 64 (4 - t) puts the pairs (2t, j) into TMEM lanes 0-63 of block 2t + j, their weight, and the pairs
// (2t + 1, j) into lanes 64-127 of the same block, one weight less than theirs.  16 MMAs (four t, four
// K-chunks) make a tile; the eighth planes are zero.  The two lane halves are folded by different warps
// into partial sums of their own, which meet once a block.
//
// Pipeline.  One CTA per subdomain (largest first): eight folding warps and a control lane in a ninth.  The
// control lane walks the sweep's list of products: it loads the operands of the next one into the other of
// two stages with bulk copies while the current one's MMAs run, and issues the MMAs into one of two TMEM
// buffers while the warps fold the other.  The digits of the block just finished are multiplied from
// where they were split (the first product of the next block), and reach the scratch array by a bulk store
// beside it.  What bounds it: with all SMs busy the digits' way from HBM (57 KB a product, 4.9 TB/s), and
// per block the chain fold, split, diagonal product, fold, split.  In step through loads, 112 MMAs of
// N = 32 and folds with ldexpf, one CTA took 8800 cycles a panel product and 32000 a diagonal one; now 3600
// (1540 of them the fold) and 12800.  A sweep over 512 subdomains of about 2400 rows 3.92 -> 1.63 ms, over
// 64 of 1250 rows 0.59 -> 0.23 ms.
// 197 KB of stages; 512 TMEM columns.
#include "a2ls_internal.cuh"
#include "tc_dfloat.cuh"

#include <algorithm>

namespace a2ls {
namespace tcs {

constexpr int M = 64, NC = 32, K = 64, NDIG = tcdf::NDIG;
constexpr uint32_t A_PLANE = M * K * 2;            // 8 KiB
constexpr uint32_t B_PLANE = NC * K * 2;           // 4 KiB
constexpr uint32_t A_TILE = NDIG * A_PLANE + M * 4;   // digit planes, then int32 row exponents
constexpr uint32_t B_TILE = NDIG * B_PLANE;
constexpr uint32_t A_BYTES = NDIG * A_PLANE, B_BYTES = NDIG * B_PLANE;   // the digit planes alone
constexpr uint32_t STAGE_A = 8 * A_PLANE, STAGE = STAGE_A + 8 * B_PLANE; // in shared memory: eight planes each
constexpr int S_LD = NC + 1;                       // row stride of S: rows fall on different banks
constexpr uint32_t S_BYTES = M * S_LD * 8;         // 64 x 32 double-float values
// dynamic shared memory: two stages, S, and the column factors of every block of X (nb of the largest)
constexpr size_t smem_bytes(int nb) { return 2 * (size_t)STAGE + S_BYTES + (size_t)nb * NC * 4; }
constexpr uint32_t BUF_COLS = 8 * NC;              // TMEM columns of one accumulator buffer
constexpr uint32_t TMEM_COLS = 512;
constexpr int THREADS = 256;                       // the folding threads (and k_factor_digits)
constexpr int ALL_THREADS = THREADS + 32;
static_assert(A_TILE % 16 == 0 && B_TILE % 16 == 0 && STAGE % 128 == 0, "16-byte copies");
static_assert(2 * BUF_COLS <= TMEM_COLS, "two accumulator buffers");

// kinds of digit tiles
enum { KIND_OFF = 0, KIND_DIAG_LOWER = 1, KIND_DIAG_UPPER = 2 };

// ---------------------------------------------------------------------------------------------
// digits of the factor tiles: one CTA per tile (i, b, c, kind) -> fdig + index * A_TILE
// ---------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(THREADS) k_factor_digits(const int4* __restrict__ jobs, const int* ni,
                                                           const int* ld, const int64_t* foff,
                                                           const dfloat* __restrict__ fac,
                                                           unsigned char* __restrict__ fdig) {
  const int4 jb = jobs[blockIdx.x];
  const int i = jb.x, b = jb.y, c = jb.z, kind = jb.w;
  const int n = ni[i];
  const int64_t L = ld[i];
  const dfloat* A = fac + foff[i];
  unsigned char* out = fdig + (size_t)blockIdx.x * A_TILE;
  const int t = threadIdx.x, r = t >> 2, q = t & 3;   // row r, k-quarter q (16 columns)
  const int gr = b * M + r;
  dfloat v[16];
  float mx = 0.f;
#pragma unroll
  for (int u = 0; u < 16; ++u) {
    const int k = q * 16 + u, gc = c * K + k;
    dfloat x(0.f, 0.f);
    if (gr < n && gc < n) {
      if (kind == KIND_OFF) x = A[(int64_t)gr * L + gc];
      else if (kind == KIND_DIAG_LOWER) x = (k < r) ? A[(int64_t)gr * L + gc] : (k == r ? dfloat(1.f, 0.f) : x);
      else x = (k >= r) ? A[(int64_t)gr * L + gc] : x;
    }
    v[u] = x;
    mx = fmaxf(mx, fabsf(x.hi));
  }
  mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
  mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
  const int e = tcdf::scale_exponent(mx);
  if (q == 0) reinterpret_cast<int*>(out + NDIG * A_PLANE)[r] = e;
#pragma unroll
  for (int h8 = 0; h8 < 2; ++h8) {
    float dg[8][NDIG];
#pragma unroll
    for (int u = 0; u < 8; ++u) tcdf::df_digits(v[h8 * 8 + u], e, dg[u]);
    const uint32_t off = tc::operand_offset(r, q * 16 + h8 * 8, K);
#pragma unroll
    for (int s = 0; s < NDIG; ++s) *reinterpret_cast<uint4*>(out + s * A_PLANE + off) = tcdf::pack_digits(dg, s);
  }
}

// the factor digits stream through L2 once per sweep (evicted first); the digits of X's finished
// blocks are read again by every later block of the sweep (kept)
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
// bulk copies (sizes multiples of 16, addresses 16-byte aligned): global -> shared with the bytes counted on
// bar; shared -> global in the thread's bulk group
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
          tc::smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(tc::smem_u32(bar)), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(tc::smem_u32(src)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// every store of the thread has been written; later bulk loads see it
__device__ __forceinline__ void bulk_stores_done() {
  asm volatile("cp.async.bulk.wait_group 0;\n\tfence.proxy.async;" ::: "memory");
}
__device__ __forceinline__ void expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(bar)) : "memory");
}
// barrier of the folding threads
__device__ __forceinline__ void fold_sync() { asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory"); }

// Digits of a 64 x 32 block as the N x K operand (column j is operand row j, the block's row index is K), one
// scale per column: v holds rows 8g .. 8g + 7 of column j (j = tid % 32, g = tid / 32).  scale[j] receives
// 2^(e_j - 8), the column's factor in the fold; red: 8 x 32 floats of scratch.  The folding threads; the
// digits become visible to the tensor cores and bulk copies once every thread has passed its next barrier.
__device__ __forceinline__ void split_columns(const dfloat (&v)[8], unsigned char* dst, float* scale, float* red) {
  const int t = threadIdx.x, j = t & 31, g = t >> 5;
  float mx = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) mx = fmaxf(mx, fabsf(v[k].hi));
  red[g * NC + j] = mx;
  fold_sync();
  mx = 0.f;
#pragma unroll
  for (int u = 0; u < 8; ++u) mx = fmaxf(mx, red[u * NC + j]);
  const int e = tcdf::scale_exponent(mx);
  if (g == 0) scale[j] = tcdf::pow2f(e - 8);
  float dg[8][NDIG];
#pragma unroll
  for (int k = 0; k < 8; ++k) tcdf::df_digits(v[k], e, dg[k]);
  const uint32_t off = tc::operand_offset(j, g * 8, K);
#pragma unroll
  for (int s = 0; s < NDIG; ++s) *reinterpret_cast<uint4*>(dst + s * B_PLANE + off) = tcdf::pack_digits(dg, s);
  tc::fence_proxy_async();
}

// The 16 MMAs of one tile product (A planes at a, B planes at b, eight each) into TMEM buffer `buf`, by one
// thread, which commits them to bar.  The first of t = 0 overwrites all eight blocks, the others add.
__device__ __forceinline__ void issue_mmas(uint32_t tmem, int buf, const unsigned char* a, const unsigned char* bsm,
                                           uint64_t* bar) {
  // descriptors of the first K-chunk of plane 0; the others differ only in the start address field
  const uint64_t ad0 = tc::smem_desc(tc::smem_u32(a), 128, K * 16), bd0 = tc::smem_desc(tc::smem_u32(bsm), 128, K * 16);
#pragma unroll
  for (int t = 0; t < 4; ++t)
#pragma unroll
    for (int kk = 0; kk < K / 16; ++kk)
      tc::mma_bf16(tmem + buf * BUF_COLS + 2 * t * NC, ad0 + ((2 * t * A_PLANE + kk * 256) >> 4), bd0 + ((kk * 256) >> 4),
                   tc::idesc_bf16_f32(2 * M, 2 * NC * (4 - t)), (t == 0 && kk == 0) ? 0u : 1u);
  tc::commit(bar);
}

// acc[0..15] += the product in TMEM buffer `buf`, for the thread's TMEM lane (a row of the tile with factor fr;
// the upper lanes hold the pairs of odd A planes, whose weights start one lower) and its 16 columns from
// h * 16 with factors fc.  acc is not normalised.
__device__ __forceinline__ void fold(uint32_t tmem, int buf, bool upper, int h, float fr, const float* fc,
                                     dfloat (&acc)[16]) {
  const uint32_t base = tmem + ((uint32_t)(((threadIdx.x >> 5) & 3) * 32) << 16) + buf * BUF_COLS + h * 16;
#pragma unroll
  for (int c8 = 0; c8 < 16; c8 += 8) {
    float a[NDIG][8];
#pragma unroll
    for (int g = 0; g < NDIG; ++g) tc::tmem_ld8(base + g * NC + c8, a[g]);
    tc::tmem_wait_ld();
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const dfloat s = tcdf::sum_blocks(a[0][q], a[1][q], a[2][q], a[3][q], a[4][q], a[5][q], upper ? 0.f : a[6][q]);
      const float f = fc[h * 16 + c8 + q];
      dfloat& o = acc[c8 + q];
      const dfloat z = df_two_sum(o.hi, __fmul_rn(__fmul_rn(s.hi, fr), f));
      o = dfloat(z.hi, __fadd_rn(o.lo, __fadd_rn(z.lo, __fmul_rn(__fmul_rn(s.lo, fr), f))));
    }
  }
}

// ---------------------------------------------------------------------------------------------
// one sweep (forward with L, or backward with U) over the subdomains with 1 <= p <= 32
// ---------------------------------------------------------------------------------------------
// items: the sweep's products of every subdomain in order, ioff[i] .. ioff[i + 1]: {factor digit tile, block c
// of X} for a panel product, {tile, -1} for the product with a block's inverted diagonal triangle, which
// ends the block.  The panel product with the block finished last comes first in its block.
// A wait that runs out (wait_limit polls) sets abort_flag, after which no wait waits: the folding warps pass
// through their remaining products without reading TMEM, and the control lane waits (up to WAIT_LIMIT polls
// each) for the MMAs, stores and loads that it has begun, so that nothing of the CTA is in flight when it gives
// its TMEM back.
__global__ void __launch_bounds__(ALL_THREADS, 1) k_block_solve_tc(
    const int* ni, const int* sched, const int* active, const int* pvec, dfloat* X, const int64_t* xoff, int col0,
    int ldx, const int64_t* ioff, const int2* __restrict__ items, const unsigned char* __restrict__ fdig,
    unsigned char* xdig, const int64_t* xdoff, int forward, long wait_limit, int* st) {
  extern __shared__ __align__(128) unsigned char sm[];
  // full: operands of a stage loaded; done: MMAs of a TMEM buffer completed; folded: a TMEM buffer read;
  // sdig, xdig_rdy: the digits of X_b - panel, of X_b, split; stored: those of X_b in the scratch array
  __shared__ __align__(8) uint64_t full[2], done[2], folded[2], sdig, xdig_rdy, stored;
  __shared__ uint32_t tbase;
  __shared__ float red[8 * NC];
  __shared__ float facS[NC];
  __shared__ volatile int abort_flag;
  const int i = sched[blockIdx.x];
  if (active && !active[i]) return;
  const int p = pvec[i];
  if (p < 1 || p > NC) return;
  const int n = ni[i], nb = (n + M - 1) / M;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int u = 0; u < 2; ++u) {
      tc::mbar_init(&full[u], 1);
      tc::mbar_init(&done[u], 1);
      tc::mbar_init(&folded[u], THREADS / 32);
    }
    tc::mbar_init(&sdig, THREADS);
    tc::mbar_init(&xdig_rdy, THREADS);
    tc::mbar_init(&stored, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    tc::tmem_alloc(&tbase, TMEM_COLS);
    tc::tmem_relinquish();
  }
  // the eighth planes of both stages stay zero
  for (int e = tid; e < 2 * (int)(A_PLANE + B_PLANE) / 16; e += ALL_THREADS) {
    const int s2 = e / (int)((A_PLANE + B_PLANE) / 16), r = e % (int)((A_PLANE + B_PLANE) / 16) * 16;
    unsigned char* z = sm + s2 * STAGE + (r < (int)A_PLANE ? A_BYTES + r : STAGE_A + B_BYTES + (r - A_PLANE));
    *reinterpret_cast<uint4*>(z) = make_uint4(0u, 0u, 0u, 0u);
  }
  tc::fence_proxy_async();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tbase;
  const int2* it = items + ioff[i];
  const int nitems = (int)(ioff[i + 1] - ioff[i]);
  unsigned char* xd = xdig + xdoff[i];
  const int dir = forward ? 1 : -1, b0 = forward ? 0 : nb - 1;
  auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
    for (long it2 = 0; it2 < wait_limit && !abort_flag; ++it2)
      if (tc::mbar_try_wait(bar, parity)) return true;
    abort_flag = 1;
    return false;
  };

  if (warp == THREADS / 32) {
    // ---- the control lane
    if (lane == 0) {
      const uint64_t pol_stream = policy_evict_first(), pol_keep = policy_evict_last();
      bool ok = true, storing = false, late_b = false;
      int2 late = {0, 0};      // the product whose B part is held back
      int b = b0, loads = 0, issued = 0;   // the current product's block; full- and done-barrier phases begun
      // operands of product m: A, and B unless it is a diagonal product or taken in place (direct)
      auto load_a = [&](int m, int2 x, bool direct) {
        uint64_t* bar = &full[m & 1];
        expect_tx(bar, A_BYTES + (x.y >= 0 && !direct ? B_BYTES : 0));
        bulk_load(sm + (m & 1) * STAGE, fdig + (size_t)x.x * A_TILE, A_BYTES, bar, pol_stream);
        ++loads;
      };
      auto load_b = [&](int m, int2 x) {
        bulk_load(sm + (m & 1) * STAGE + STAGE_A, xd + (size_t)x.y * B_TILE, B_BYTES, &full[m & 1], pol_keep);
      };
      int2 cur = it[0], nxt = cur;
      bool prev_diag = false;          // product m - 1 ended a block
      int last = -1;                   // the block finished last
      load_a(0, cur, false);           // the first product is a diagonal one
      for (int m = 0; m < nitems && ok; ++m) {
        const bool diag = cur.y < 0, direct = !diag && prev_diag && cur.y == last;
        // stage (m + 1) & 1 is free once product m - 1 has run
        if (m > 0) ok = wait(&done[(m - 1) & 1], ((m - 1) >> 1) & 1);
        if (!ok) break;
        tc::fence_after_sync();
        if (storing) {                 // X digits of an earlier block: written, and their stage free
          bulk_stores_done();
          arrive(&stored);
          storing = false;
        }
        if (late_b) {                  // product m's B part, held back while its stage held X digits
          load_b(m, late);
          late_b = false;
        }
        if (m + 1 < nitems) {
          nxt = it[m + 1];
          // product m + 1 is direct if product m ends a block and m + 1 multiplies that block
          const bool ndirect = diag && nxt.y == b;
          load_a(m + 1, nxt, ndirect);
          if (nxt.y >= 0 && !ndirect) {
            // the B slot of its stage holds X digits if product m - 1 was a diagonal one: product m multiplies
            // them, or they are still to be stored
            if (prev_diag) {
              late_b = true;
              late = nxt;
            } else {
              load_b(m + 1, nxt);
            }
          }
        }
        const int blk = (b - b0) * dir;                       // blocks finished before this one
        ok = wait(&full[m & 1], (m >> 1) & 1);
        if (ok && m >= 2) ok = wait(&folded[m & 1], ((m - 2) >> 1) & 1);
        if (ok && diag) ok = wait(&sdig, blk & 1);
        if (ok && prev_diag) ok = wait(&xdig_rdy, (blk - 1) & 1);
        if (!ok) break;
        tc::fence_after_sync();
        const unsigned char* A = sm + (m & 1) * STAGE;
        issue_mmas(tmem, m & 1, A, sm + ((direct ? m - 1 : m) & 1) * STAGE + STAGE_A, &done[m & 1]);
        issued = m + 1;
        if (prev_diag) {
          // the digits of the block just finished, from the stage of its diagonal product
          bulk_store(xd + (size_t)last * B_TILE, sm + ((m - 1) & 1) * STAGE + STAGE_A, B_BYTES);
          bulk_commit();
          storing = true;
        }
        prev_diag = diag;
        if (diag) {
          last = b;
          b += dir;
        }
        cur = nxt;
      }
      // nothing of this CTA may be in flight when it leaves: the MMAs, the stores, the loads begun (of which the
      // last may still want its B part)
      for (int m = max(0, issued - 2); m < issued; ++m) tc::mbar_wait_bounded(&done[m & 1], (m >> 1) & 1, tcdf::WAIT_LIMIT);
      bulk_stores_done();
      if (late_b) load_b(loads - 1, late);
      for (int m = max(0, loads - 2); m < loads; ++m) tc::mbar_wait_bounded(&full[m & 1], (m >> 1) & 1, tcdf::WAIT_LIMIT);
    }
    __syncwarp();
  } else {
    // ---- the folding warps
    const int qd = warp & 3, h = warp >> 2, row = (qd & 1) * 32 + lane;
    const bool upper = qd >= 2;
    dfloat* Xi = X + xoff[i] + col0;
    dfloat* S = reinterpret_cast<dfloat*>(sm + 2 * STAGE);
    float* facX = reinterpret_cast<float*>(sm + 2 * STAGE + S_BYTES);   // NC column factors per block of X
    // the row factor 2^(e_r - 8) of a factor tile
    auto row_fac = [&](int tile) {
      return tcdf::pow2f(__ldg(reinterpret_cast<const int*>(fdig + (size_t)tile * A_TILE + A_BYTES) + row) - 8);
    };
    dfloat* Srow = S + row * S_LD + h * 16;
    const int sj = tid & 31, sg = tid >> 5;   // the thread's part of a split: column sj, rows 8 sg .. 8 sg + 7
    const dfloat* Scol = S + sg * 8 * S_LD + sj;
    dfloat acc[16], xb[8];
    // S = the two lane halves' sums; ends with a barrier
    auto combine = [&]() {
      if (upper)
#pragma unroll
        for (int u = 0; u < 16; ++u) Srow[u] = acc[u];
      fold_sync();
      if (!upper)
#pragma unroll
        for (int u = 0; u < 16; ++u) Srow[u] = df_normalize(acc[u]) + df_normalize(Srow[u]);
      fold_sync();
    };
    auto clear = [&]() {
#pragma unroll
      for (int u = 0; u < 16; ++u) acc[u] = dfloat(0.f, 0.f);
    };
    auto fetch = [&](int b) {   // the block's X in the split's layout (zero outside the block and the columns)
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int r = b * M + sg * 8 + k;
        xb[k] = (r < n && sj < p) ? Xi[(int64_t)r * ldx + sj] : dfloat(0.f, 0.f);
      }
    };
    int b = b0, blk = 0;
    bool ok = true, diag1 = false, diag2 = false;   // products m - 1, m - 2 ended blocks
    clear();
    fetch(b);
    int2 cur = it[0];
    float fr = row_fac(cur.x);
    for (int m = 0; m < nitems; ++m) {
      const int2 nxt = m + 1 < nitems ? it[m + 1] : cur;
      const float nfr = row_fac(nxt.x);   // used by the next fold
      const bool diag = cur.y < 0;
      if (diag) {
        // the digits of X_b - panel; those that the stage's B part last held (of X, two products back) have
        // been stored
        combine();
#pragma unroll
        for (int k = 0; k < 8; ++k) xb[k] = xb[k] - Scol[k * S_LD];
        if (diag2 && !wait(&stored, (diag1 ? blk - 2 : blk - 1) & 1)) ok = false;
        split_columns(xb, sm + (m & 1) * STAGE + STAGE_A, facS, red);
        arrive(&sdig);
        fold_sync();   // the factors are read by every thread below
        clear();
      }
      if (!wait(&done[m & 1], (m >> 1) & 1)) ok = false;
      ok = __all_sync(0xffffffffu, ok) != 0;   // the loads from TMEM are the whole warp's
      tc::fence_after_sync();
      if (ok) fold(tmem, m & 1, upper, h, fr, diag ? facS : facX + cur.y * NC, acc);
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) arrive(&folded[m & 1]);
      if (diag) {
        // X_b: to X and, for the later blocks of the sweep, as digits
        combine();
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int r = b * M + sg * 8 + k;
          const bool in = r < n && sj < p;
          xb[k] = in ? Scol[k * S_LD] : dfloat(0.f, 0.f);
          if (in) Xi[(int64_t)r * ldx + sj] = xb[k];
        }
        split_columns(xb, sm + (m & 1) * STAGE + STAGE_A, facX + b * NC, red);
        arrive(&xdig_rdy);
        fold_sync();
        b += dir;
        ++blk;
        clear();
        if (m + 1 < nitems) fetch(b);
      }
      diag2 = diag1;
      diag1 = diag;
      cur = nxt;
      fr = nfr;
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (tid == 0 && abort_flag) raise_status(st, A2LS_ERR_TIMEOUT, i, forward);   // whichever wait ran out
  if (warp == 0) tc::tmem_dealloc(tmem, TMEM_COLS);
}

}  // namespace tcs

// ---------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------
void tc_solve_prepare(a2ls_handle* h, const dfloat* fac, TcSolve& ts) {
  using namespace tcs;
  cudaStream_t st = h->st;
  const int N = h->N;
  const int T = h->h_toff[N];
  std::vector<int> tf(T), tg(T);
  A2LS_CUDA(cudaMemcpyAsync(tf.data(), h->d_tf, sizeof(int) * T, cudaMemcpyDeviceToHost, st));
  A2LS_CUDA(cudaMemcpyAsync(tg.data(), h->d_tg, sizeof(int) * T, cudaMemcpyDeviceToHost, st));
  A2LS_CUDA(cudaStreamSynchronize(st));
  std::vector<int64_t> xdoff(N + 1, 0);
  for (int i = 0; i < N; ++i) xdoff[i + 1] = xdoff[i] + (int64_t)((h->h_n[i] + M - 1) / M) * B_TILE;
  std::vector<int4> jobs;           // the factor digit tiles: subdomain, block row, block column, kind
  std::vector<int2> items[2];       // the products of the backward and the forward sweep
  std::vector<int64_t> ioff[2];
  for (int i = 0; i < N; ++i) {
    const int nb = (h->h_n[i] + M - 1) / M;
    const int* tfi = tf.data() + h->h_toff[i];
    const int* tgi = tg.data() + h->h_toff[i];
    auto add = [&](int b, int c, int kind) {
      jobs.push_back(make_int4(i, b, c, kind));
      return (int)jobs.size() - 1;
    };
    for (int fwd = 0; fwd < 2; ++fwd) {
      ioff[fwd].push_back((int64_t)items[fwd].size());
      for (int k = 0; k < nb; ++k) {
        const int b = fwd ? k : nb - 1 - k;
        // the panel, from the block finished last outwards: L's row block b reaches column tile c, U's
        // column tile c reaches row block b
        if (fwd) {
          for (int c = b - 1; c >= 0; --c)
            if (tfi[b] <= c * M + M - 1) items[1].push_back(make_int2(add(b, c, KIND_OFF), c));
        } else {
          for (int c = b + 1; c < nb; ++c)
            if (tgi[c] <= b * M + M - 1) items[0].push_back(make_int2(add(b, c, KIND_OFF), c));
        }
        items[fwd].push_back(make_int2(add(b, b, fwd ? KIND_DIAG_LOWER : KIND_DIAG_UPPER), -1));
      }
    }
  }
  ts.ntiles = (int64_t)jobs.size();
  ts.d_xdoff = dalloc<int64_t>(h, N + 1);
  ts.d_fdig = dalloc<unsigned char>(h, (size_t)ts.ntiles * A_TILE);
  ts.d_xdig = dalloc<unsigned char>(h, (size_t)xdoff[N]);
  int4* d_jobs = dalloc<int4>(h, jobs.size());
  for (int f = 0; f < 2; ++f) {
    ioff[f].push_back((int64_t)items[f].size());
    ts.d_ioff[f] = dalloc<int64_t>(h, N + 1);
    ts.d_items[f] = dalloc<int2>(h, items[f].size());
    A2LS_CUDA(cudaMemcpyAsync(ts.d_ioff[f], ioff[f].data(), sizeof(int64_t) * (N + 1), cudaMemcpyHostToDevice, st));
    A2LS_CUDA(cudaMemcpyAsync(ts.d_items[f], items[f].data(), sizeof(int2) * items[f].size(), cudaMemcpyHostToDevice, st));
  }
  A2LS_CUDA(cudaMemcpyAsync(ts.d_xdoff, xdoff.data(), sizeof(int64_t) * (N + 1), cudaMemcpyHostToDevice, st));
  A2LS_CUDA(cudaMemcpyAsync(d_jobs, jobs.data(), sizeof(int4) * jobs.size(), cudaMemcpyHostToDevice, st));
  // the grid dimension limit (2^31 - 1) is far above any tile count the 8192-row subdomains allow
  k_factor_digits<<<(unsigned)jobs.size(), THREADS, 0, st>>>(d_jobs, h->d_ni, h->d_ld, h->d_foff, fac, ts.d_fdig);
  A2LS_LAUNCH();
  A2LS_CUDA(cudaFuncSetAttribute(k_block_solve_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem_bytes(MAXN_LOCAL / M)));
  A2LS_CUDA(cudaStreamSynchronize(st));   // the job list is freed below
  dfree(h, d_jobs);
  ts.ready = true;
}

void tc_solve_release(a2ls_handle* h, TcSolve& ts) {
  if (!ts.ready) return;
  for (int f = 0; f < 2; ++f) {
    dfree(h, ts.d_ioff[f]);
    dfree(h, ts.d_items[f]);
  }
  dfree(h, ts.d_xdoff);
  dfree(h, ts.d_fdig);
  dfree(h, ts.d_xdig);
  ts = TcSolve{};
}

void tc_block_solve(a2ls_handle* h, const TcSolve& ts, dfloat* X, const int64_t* xoff, int col0, int ldx,
                    const int* pvec, const int* active, int forward, unsigned char* xdig, long wait_limit) {
  using namespace tcs;
  tcs::k_block_solve_tc<<<h->N, ALL_THREADS, smem_bytes(ceil_div(h->max_n, M)), h->st>>>(h->d_ni, h->d_sched, active, pvec, X, xoff, col0, ldx,
                                                            ts.d_ioff[forward != 0], ts.d_items[forward != 0], ts.d_fdig,
                                                            xdig ? xdig : ts.d_xdig, ts.d_xdoff, forward,
                                                            wait_limit, h->d_status);
  A2LS_LAUNCH();
}

}  // namespace a2ls
