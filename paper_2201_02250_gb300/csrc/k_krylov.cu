// The apply of the preconditioners of Section 2 (Eqs. 2.1-2.4) and the
// right-preconditioned restarted (F)GMRES of Section 4, all vectors FP64.
//
// Deflated RAS (Eq. 2.4), the default:
//   g = R_0 r            (tall-skinny W_i^T r(Omega_i), warp-shuffle reductions)
//   c = A_00^{-1} g      (dense FP64 matrix-vector product with the inverse)
//   q = R_0^H c          (prolongation)
//   t = r - A q          (CSR SpMV)
//   z = q + sum_i R_i^T D_i A_ii^{-1} R_i t   (gather, two triangular solves, weighted scatter)
#include "a2ls_internal.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>

namespace a2ls {

// ---------------------------------------------------------------------------
// CSR SpMV: y = A x, or y = bm - A x when bm != nullptr.  Bound by memory: 12 bytes an entry.
// Stencils (SPMV_SHORT entries a row on average, or fewer): a thread per row with SPMV_UNROLL entries in flight;
// the neighbours' entries share its cache lines.  4 lanes per row kept one gather in flight: 41.4 -> 22.3 us on
// the 96^3 seven-point operator (91 MB); 150,000 rows of 5, 9, 15 entries 15.0, 15.0, 19.1 -> 10.9, 13.0, 15.0.
// A row of more than SPMV_LONG entries is the whole warp's (that operator with one row of 2000: 140 us with four
// lanes, 42 so).
// ---------------------------------------------------------------------------
constexpr int SPMV_UNROLL = 8, SPMV_SHORT = 16, SPMV_LONG = 64;
__global__ void __launch_bounds__(128) k_spmv(int n, const int* __restrict__ rowptr, const int* __restrict__ colind,
                                              const double* __restrict__ val, const double* __restrict__ x,
                                              double* __restrict__ y, const double* __restrict__ bm) {
  const int r = blockIdx.x * 128 + threadIdx.x, lane = threadIdx.x & 31;
  const int a = r < n ? rowptr[r] : 0, b = r < n ? rowptr[r + 1] : 0;
  const bool is_long = b - a > SPMV_LONG;
  double s = 0.0;
  for (int q = a; q < b && !is_long; q += SPMV_UNROLL) {
    int c[SPMV_UNROLL];
    double v[SPMV_UNROLL], xv[SPMV_UNROLL];
#pragma unroll
    for (int u = 0; u < SPMV_UNROLL; ++u) {
      c[u] = q + u < b ? __ldg(colind + q + u) : 0;
      v[u] = q + u < b ? __ldg(val + q + u) : 0.0;
    }
#pragma unroll
    for (int u = 0; u < SPMV_UNROLL; ++u) xv[u] = q + u < b ? __ldg(x + c[u]) : 0.0;
#pragma unroll
    for (int u = 0; u < SPMV_UNROLL; ++u) s += v[u] * xv[u];
  }
  for (unsigned todo = __ballot_sync(0xffffffffu, is_long); todo; todo &= todo - 1) {
    const int owner = __ffs(todo) - 1;
    const int a2 = __shfl_sync(0xffffffffu, a, owner), b2 = __shfl_sync(0xffffffffu, b, owner);
    double t = 0.0;
#pragma unroll 4
    for (int q = a2 + lane; q < b2; q += 32) t += __ldg(val + q) * __ldg(x + __ldg(colind + q));
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == owner) s = t;
  }
  if (r < n) y[r] = bm ? bm[r] - s : s;
}

// Other matrices: 4 lanes per row.  150,000 rows of 17, 33, 65, 301 entries: 19, 25, 38, 122 us, with a thread each 19,
// 29, 50, 193.
__global__ void k_spmv_wide(int n, const int* __restrict__ rowptr, const int* __restrict__ colind,
                            const double* __restrict__ val, const double* __restrict__ x, double* __restrict__ y,
                            const double* __restrict__ bm) {
  const int sub = threadIdx.x & 3;
  const unsigned row_lanes = 0xfu << (threadIdx.x & 28);
  for (int r = (blockIdx.x * blockDim.x + threadIdx.x) >> 2; r < n; r += (gridDim.x * blockDim.x) >> 2) {
    double s = 0.0;
    const int a = rowptr[r], b = rowptr[r + 1];
    for (int q = a + sub; q < b; q += 4) s += val[q] * __ldg(x + colind[q]);
    s += __shfl_xor_sync(row_lanes, s, 1);
    s += __shfl_xor_sync(row_lanes, s, 2);
    if (sub == 0) y[r] = bm ? bm[r] - s : s;
  }
}

void spmv(a2ls_handle* h, const double* x, double* y, const double* b_minus, cudaStream_t st) {
  if (h->nnz <= (int64_t)SPMV_SHORT * h->n) {
    k_spmv<<<ceil_div(h->n, 128), 128, 0, st>>>(h->n, h->rowptr, h->colind, h->val, x, y, b_minus);
  } else {
    const int threads = 256;
    const int blocks = std::min(152 * 8, ceil_div((int64_t)h->n * 4, threads));
    k_spmv_wide<<<blocks, threads, 0, st>>>(h->n, h->rowptr, h->colind, h->val, x, y, b_minus);
  }
  A2LS_LAUNCH();
}

// ---------------------------------------------------------------------------
// g[coff_i + a] = sum_l W_i[l][a] r[idx[off_i + l]] over rows with D != 0.
// Lanes are split into groups of G >= m_i columns; the 32/G row groups of a warp
// are combined by warp shuffles, the warps of the CTA through shared memory.
// ---------------------------------------------------------------------------
constexpr int RESTRICT_THREADS = 512;
__global__ void __launch_bounds__(RESTRICT_THREADS) k_restrict(const int* ni, const int* nI, const int* off, const int* idx,
                                                  const int* m, const int* coff, const int64_t* woff,
                                                  const double* __restrict__ W, const double* __restrict__ r,
                                                  double* g, int boolean_pou) {
  __shared__ double part[RESTRICT_THREADS / 32][MAXM];
  const int i = blockIdx.x;
  const int mi = m[i];
  if (mi == 0) return;
  const int rows = boolean_pou ? nI[i] : ni[i];
  const int o = off[i];
  const double* Wi = W + woff[i];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int G = 1;
  while (G < mi && G < 32) G <<= 1;
  constexpr int RW = RESTRICT_THREADS / 32;
  const int rg = 32 / G;          // row groups per warp
  const int sub = lane / G, a = lane % G;
  for (int c0 = 0; c0 < mi; c0 += 32) {
    double acc = 0.0;
    const int col = c0 + a;
    // RU rows' gathers and coefficients in flight (one at a time and 8 warps: 65 us on 512 subdomains of 1728
    // rows and 12 columns, 120 MB; four and 16 warps 54 us)
    constexpr int RU = 4;
    for (int l0 = wid * rg + sub; l0 < rows; l0 += RU * RW * rg) {
      double rv[RU], wv[RU];
#pragma unroll
      for (int u = 0; u < RU; ++u) {
        const int l = l0 + u * RW * rg;
        rv[u] = l < rows ? __ldg(r + idx[o + l]) : 0.0;
        wv[u] = (l < rows && col < mi) ? Wi[(int64_t)l * mi + col] : 0.0;
      }
#pragma unroll
      for (int u = 0; u < RU; ++u) acc += wv[u] * rv[u];
    }
    for (int s = G; s < 32; s <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
    if (sub == 0 && col < mi) part[wid][col] = acc;
    __syncthreads();
    if (threadIdx.x < 32 && c0 + threadIdx.x < mi) {
      double t = 0.0;
      for (int w = 0; w < RW; ++w) t += part[w][c0 + threadIdx.x];
      g[coff[i] + c0 + threadIdx.x] = t;
    }
    __syncthreads();
  }
}

// c = Einv g; one warp per row, 16-byte loads (8-byte ones of odd n0, whose rows lose the alignment); bound
// by the FP64 pipes (2 flops per 8 bytes)
__global__ void __launch_bounds__(256) k_gemv(int n0, const double* __restrict__ Einv,
                                              const double* __restrict__ g, double* __restrict__ c) {
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const bool even = (n0 & 1) == 0;
  for (int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; row < n0; row += warps) {
    const double* er = Einv + (int64_t)row * n0;
    double s = 0.0;
    if (even) {
      const double2* e2 = reinterpret_cast<const double2*>(er);
      const double2* g2 = reinterpret_cast<const double2*>(g);
      // the matrix streams past the caches (evicted first; kept like other loads 131 us for n0 = 6206, 308 MB,
      // so 92)
      double s1 = 0.0;
#pragma unroll 4
      for (int k = lane; k < n0 / 2; k += 32) {
        const double2 a = __ldcs(e2 + k), b = __ldg(g2 + k);
        s += a.x * b.x;
        s1 += a.y * b.y;
      }
      s += s1;
    } else {
#pragma unroll 8
      for (int k = lane; k < n0; k += 32) s += __ldcs(er + k) * __ldg(g + k);
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) c[row] = s;
  }
}

// q[g] = sum over memberships (j, pos) of node g with D != 0 of W_j[pos - off_j, :] . c_j
__global__ void k_prolong(int n, const int* mrow, const int* mpos, const int* msub, const int* off, const int* m,
                          const int* coff, const int64_t* woff, const double* D, const double* __restrict__ W,
                          const double* __restrict__ c, double* q) {
  for (int gI = blockIdx.x * blockDim.x + threadIdx.x; gI < n; gI += gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int t = mrow[gI]; t < mrow[gI + 1]; ++t) {
      const int p = mpos[t];
      if (D[p] == 0.0) continue;
      const int j = msub[t], mj = m[j];
      const double* w = W + woff[j] + (int64_t)(p - off[j]) * mj;
      const double* cj = c + coff[j];
      for (int a = 0; a < mj; ++a) s += w[a] * cj[a];
    }
    q[gI] = s;
  }
}

// The same for the Boolean partition of unity, where a node's only weight is that of the subdomain it lies
// in: one CTA walks the interior rows of a subdomain, a thread a row, with c_i in shared memory and no
// membership lists to chase.  512 subdomains of 1728 rows, 12 columns (120 MB): 64 -> 32 us.
__global__ void __launch_bounds__(256) k_prolong_interior(const int* nI, const int* off, const int* idx, const int* m,
                                                          const int* coff, const int64_t* woff,
                                                          const double* __restrict__ W, const double* __restrict__ c,
                                                          double* q) {
  __shared__ double cs[MAXM];
  const int i = blockIdx.x, mi = m[i], n = nI[i], o = off[i];
  const double* Wi = W + woff[i];
  if (threadIdx.x < mi) cs[threadIdx.x] = c[coff[i] + threadIdx.x];
  __syncthreads();
  for (int l = blockIdx.y * 256 + threadIdx.x; l < n; l += gridDim.y * 256) {
    const double* w = Wi + (int64_t)l * mi;
    double s = 0.0;
#pragma unroll 4
    for (int a = 0; a < mi; ++a) s += w[a] * cs[a];
    q[idx[o + l]] = s;
  }
}

// z[g] = (q ? q[g] : 0) + sum over memberships of yloc[pos]
__global__ void k_combine(int n, const int* mrow, const int* mpos, const double* __restrict__ yloc,
                          const double* __restrict__ q, double* z) {
  for (int gI = blockIdx.x * blockDim.x + threadIdx.x; gI < n; gI += gridDim.x * blockDim.x) {
    double s = q ? q[gI] : 0.0;
    for (int t = mrow[gI]; t < mrow[gI + 1]; ++t) s += yloc[mpos[t]];
    z[gI] = s;
  }
}

// q = R_0^H c
void prolong(a2ls_handle* h, const double* c, double* q) {
  if (h->opt.pou == A2LS_POU_BOOLEAN) {
    const int parts = std::max(1, std::min(ceil_div(h->max_n, 256), 2 * 152 / std::max(h->N, 1) + 1));
    k_prolong_interior<<<dim3(h->N, parts), 256, 0, h->st>>>(h->d_nI, h->d_off, h->d_idx, h->d_m, h->d_coff, h->d_woff,
                                                             h->d_W, c, q);
  } else {
    k_prolong<<<std::max(1, std::min(152 * 8, ceil_div(h->n, 256))), 256, 0, h->st>>>(
        h->n, h->d_mrow, h->d_mpos, h->d_msub, h->d_off, h->d_m, h->d_coff, h->d_woff, h->d_D, h->d_W, c, q);
  }
  A2LS_LAUNCH();
}

static int grid1d(int64_t n, int threads = 256) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(152 * 8, (n + threads - 1) / threads));
}

static void local_part(a2ls_handle* h, const double* t, const double* q, double* z, bool ras) {
  const bool boolean = h->opt.pou == A2LS_POU_BOOLEAN;
  const int mode = ras ? (boolean ? 0 : 1) : 2;
  double* out = (mode == 0) ? z : h->d_yloc;
  local_solves_any(h, t, q, out, mode);
  if (mode != 0) {
    k_combine<<<grid1d(h->n), 256, 0, h->st>>>(h->n, h->d_mrow, h->d_mpos, h->d_yloc, q, z);
    A2LS_LAUNCH();
  }
}

static void coarse_correction(a2ls_handle* h, const double* r, double* q) {
  cudaStream_t st = h->st;
  k_restrict<<<h->N, RESTRICT_THREADS, 0, st>>>(h->d_ni, h->d_nI, h->d_off, h->d_idx, h->d_m, h->d_coff, h->d_woff, h->d_W,
                                   r, h->d_g, h->opt.pou == A2LS_POU_BOOLEAN);
  A2LS_LAUNCH();
  k_gemv<<<std::min(152 * 8, ceil_div((int64_t)h->n0 * 32, 256)), 256, 0, st>>>(h->n0, h->d_Einv, h->d_g, h->d_c);
  A2LS_LAUNCH();
  prolong(h, h->d_c, q);
}

void apply_preconditioner(a2ls_handle* h, const double* r, double* z) {
  const int v = h->opt.variant;
  const bool ras = (v == A2LS_DEFLATED_RAS || v == A2LS_ADDITIVE_RAS || v == A2LS_ONE_LEVEL_RAS);
  const bool coarse = (v != A2LS_ONE_LEVEL_RAS && v != A2LS_ONE_LEVEL_ASM) && h->n0 > 0;
  const bool deflated = (v == A2LS_DEFLATED_RAS || v == A2LS_DEFLATED_ASM);
  if (!coarse) {
    local_part(h, r, nullptr, z, ras);
    return;
  }
  coarse_correction(h, r, h->d_q);
  if (deflated) {
    spmv(h, h->d_q, h->d_t, r, h->st);  // t = r - A q
    local_part(h, h->d_t, h->d_q, z, ras);
  } else {
    local_part(h, r, h->d_q, z, ras);
  }
}

// The apply as a CUDA graph, captured once per (r, z) pair on an internal stream and replayed on
// the handle's stream: GMRES applies the preconditioner to the same m basis vectors every cycle.
void apply_preconditioner_graph(a2ls_handle* h, const double* r, double* z) {
  if (!h->opt.graphs) {
    apply_preconditioner(h, r, z);
    return;
  }
  for (const auto& g : h->graphs)
    if (g.r == r && g.z == z) {
      A2LS_CUDA(cudaGraphLaunch(g.exec, h->st));
      h->launches += 1;
      return;
    }
  if (!h->cap_st) A2LS_CUDA(cudaStreamCreateWithFlags(&h->cap_st, cudaStreamNonBlocking));
  cudaStream_t user = h->st;
  const int timing = h->opt.timing;
  h->opt.timing = 0;
  h->st = h->cap_st;
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamBeginCapture(h->cap_st, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    try {
      apply_preconditioner(h, r, z);
    } catch (...) {
      cudaStreamEndCapture(h->cap_st, &graph);
      if (graph) cudaGraphDestroy(graph);
      h->st = user;
      h->opt.timing = timing;
      throw;
    }
    e = cudaStreamEndCapture(h->cap_st, &graph);
  }
  h->st = user;
  h->opt.timing = timing;
  A2LS_CUDA(e);
  cudaGraphExec_t exec = nullptr;
  const cudaError_t ei = cudaGraphInstantiate(&exec, graph, 0);
  cudaGraphDestroy(graph);
  A2LS_CUDA(ei);
  h->graphs.push_back({r, z, exec});
  A2LS_CUDA(cudaGraphLaunch(exec, h->st));
  h->launches += 1;
}

// ---------------------------------------------------------------------------
// reductions for GMRES: multi-dot with a last-block-done final reduction
// out[k] = sum_r V[k][r] * w[r] for k < nv, out[nv] = w . w (if with_self)
//
// Bound by the FP64 pipes as much as by memory (two multiply-adds a cycle and SM: nv n / 304 cycles), so
// nothing may be added up with most lanes idle: a CTA takes MD_COLS vectors (blockIdx.y), its threads'
// sums meet in shared memory, a warp per vector, and so do the CTAs' in the last one.  One vector's load
// at a time, sums shuffled in every warp and the CTAs' partial sums added by one thread took 70 us for 8.5
// vectors of 884736 on average, now 30.
// ---------------------------------------------------------------------------
constexpr int MD_MAX = 33;
constexpr int MD_COLS = 8;
constexpr int MD_BLOCKS = 608;
constexpr int MD_GROUPS = (MD_MAX + MD_COLS - 1) / MD_COLS;

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The CTA's sums of val over its threads, for ncol <= 8 columns, added to those of the other gridDim.x
// CTAs of the same blockIdx.y: the last of them writes out[0 .. ncol).  256 threads; partial: 8 x gridDim.x
// values and counter (zero, left zero) of this blockIdx.y.
__device__ __forceinline__ void grid_sum(const double (&val)[MD_COLS], int ncol, double* partial, unsigned* counter,
                                         double* out) {
  __shared__ double red[MD_COLS][256];
  __shared__ bool last;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
#pragma unroll
  for (int k = 0; k < MD_COLS; ++k)
    if (k < ncol) red[k][tid] = val[k];
  __syncthreads();
  if (wid < ncol) {  // warp wid: column wid
    double s = 0.0;
#pragma unroll
    for (int u = 0; u < 8; ++u) s += red[wid][lane + 32 * u];
    s = warp_sum(s);
    if (lane == 0) {
      partial[wid * gridDim.x + blockIdx.x] = s;
      __threadfence();
    }
  }
  __syncthreads();
  if (tid == 0) last = (atomicAdd(counter, 1u) == gridDim.x - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (wid < ncol) {
    double s = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) s += __ldcg(partial + wid * gridDim.x + b);
    s = warp_sum(s);
    if (lane == 0) out[wid] = s;
  }
  if (tid == 0) *counter = 0u;
}

__global__ void __launch_bounds__(256) k_multidot(int n, const double* __restrict__ V, int64_t ldv, int nv,
                                                  const double* __restrict__ w, int with_self,
                                                  double* partial, unsigned* counter, double* out) {
  const int k0 = blockIdx.y * MD_COLS, nd = nv + (with_self ? 1 : 0), ncol = min(MD_COLS, nd - k0);
  double acc[MD_COLS];
  const double* col[MD_COLS];
#pragma unroll
  for (int k = 0; k < MD_COLS; ++k) {
    acc[k] = 0.0;
    // w itself as the last vector; columns past the end repeat the last one (cached) and are not used
    const int kk = min(k0 + k, nd - 1);
    col[k] = kk < nv ? V + (int64_t)kk * ldv : w;
  }
  const int stride = gridDim.x * 256;
  for (int r = blockIdx.x * 256 + threadIdx.x; r < n; r += stride) {
    const double wr = w[r];
    if (ncol == MD_COLS) {
      double v[MD_COLS];
#pragma unroll
      for (int k = 0; k < MD_COLS; ++k) v[k] = col[k][r];
#pragma unroll
      for (int k = 0; k < MD_COLS; ++k) acc[k] += v[k] * wr;
    } else {
      double v[MD_COLS - 1];
#pragma unroll
      for (int k = 0; k < MD_COLS - 1; ++k) v[k] = k < ncol ? col[k][r] : 0.0;
#pragma unroll
      for (int k = 0; k < MD_COLS - 1; ++k)
        if (k < ncol) acc[k] += v[k] * wr;
    }
  }
  grid_sum(acc, ncol, partial + (int64_t)blockIdx.y * MD_COLS * MD_BLOCKS, counter + blockIdx.y, out + k0);
}

// w -= sum_k hk V_k, with norm2 (if given) = |w|^2 of the result
// (norm2: at most MD_BLOCKS MD_COLS CTAs)
__global__ void __launch_bounds__(256) k_cgs_update(int n, const double* __restrict__ V, int64_t ldv, int nv,
                                                    const double* hcoef, double* w, double* partial, unsigned* counter,
                                                    double* norm2) {
  __shared__ double hs[MD_MAX + 3];
  if (threadIdx.x < MD_MAX + 3) hs[threadIdx.x] = threadIdx.x < nv ? hcoef[threadIdx.x] : 0.0;
  __syncthreads();
  double sq[MD_COLS] = {};
  for (int r = blockIdx.x * 256 + threadIdx.x; r < n; r += gridDim.x * 256) {
    double s = w[r];
#pragma unroll 4
    for (int k = 0; k < nv; ++k) s -= hs[k] * V[(int64_t)k * ldv + r];
    w[r] = s;
    sq[0] += s * s;
  }
  if (norm2) grid_sum(sq, 1, partial, counter, norm2);
}

// y = x * (1 / *alpha) or y = x * alpha_host when alpha_dev == nullptr
__global__ void k_scale(int n, const double* x, double* y, const double* alpha_dev, int sqrt_of, double alpha_host) {
  double a = alpha_host;
  if (alpha_dev) a = 1.0 / (sqrt_of ? sqrt(*alpha_dev) : *alpha_dev);
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) y[r] = x[r] * a;
}

// y = sum_k c_k V_k (c on device); optionally x += y
__global__ void k_lincomb(int n, const double* __restrict__ V, int64_t ldv, int nv, const double* coef, double* y,
                          double* xacc) {
  __shared__ double cs[MD_MAX];
  if (threadIdx.x < nv) cs[threadIdx.x] = coef[threadIdx.x];
  __syncthreads();
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
    double s = 0.0;
#pragma unroll 4
    for (int k = 0; k < nv; ++k) s += cs[k] * V[(int64_t)k * ldv + r];
    if (xacc) xacc[r] += s;
    else y[r] = s;
  }
}

__global__ void k_axpy(int n, double a, const double* x, double* y) {
  for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) y[r] += a * x[r];
}

struct Reducer {
  double* partial = nullptr;
  unsigned* counter = nullptr;
  double* out = nullptr;
};

static Reducer& reducer(a2ls_handle* h) {
  constexpr size_t parts = (size_t)MD_BLOCKS * MD_COLS * MD_GROUPS;
  if (!h->d_red) {
    h->d_red = dalloc<double>(h, parts + 4 * MD_MAX + 16);
    A2LS_CUDA(cudaMemsetAsync(h->d_red, 0, sizeof(double) * (parts + 4 * MD_MAX + 16), h->st));
  }
  static thread_local Reducer r;
  r.partial = h->d_red;
  r.out = h->d_red + parts;                                  // 4 * MD_MAX doubles of outputs
  r.counter = reinterpret_cast<unsigned*>(r.out + 4 * MD_MAX);
  return r;
}

static void multidot(a2ls_handle* h, const double* V, int64_t ldv, int nv, const double* w, int with_self,
                     double* out) {
  Reducer& R = reducer(h);
  const int nd = nv + (with_self ? 1 : 0);
  const dim3 grid(std::min(MD_BLOCKS, std::max(1, ceil_div(h->n, 256))), ceil_div(nd, MD_COLS));
  k_multidot<<<grid, 256, 0, h->st>>>(h->n, V, ldv, nv, w, with_self, R.partial, R.counter, out);
  A2LS_LAUNCH();
}

// w -= sum_k h_k V_k; norm2 (device, may be null) receives |w|^2 of the result
static void cgs_update(a2ls_handle* h, const double* V, int64_t ldv, int nv, const double* hcoef, double* w,
                       double* norm2) {
  Reducer& R = reducer(h);
  k_cgs_update<<<grid1d(h->n), 256, 0, h->st>>>(h->n, V, ldv, nv, hcoef, w, R.partial, R.counter, norm2);
  A2LS_LAUNCH();
}

double dot(a2ls_handle* h, const double* x, const double* y) {
  Reducer& R = reducer(h);
  multidot(h, x, 0, 1, y, 0, R.out);
  double v;
  A2LS_CUDA(cudaMemcpyAsync(&v, R.out, sizeof(double), cudaMemcpyDeviceToHost, h->st));
  A2LS_CUDA(cudaStreamSynchronize(h->st));
  return v;
}

double nrm2(a2ls_handle* h, const double* x) {
  Reducer& R = reducer(h);
  multidot(h, x, 0, 0, x, 1, R.out);
  double v;
  A2LS_CUDA(cudaMemcpyAsync(&v, R.out, sizeof(double), cudaMemcpyDeviceToHost, h->st));
  A2LS_CUDA(cudaStreamSynchronize(h->st));
  return std::sqrt(v);
}

// ---------------------------------------------------------------------------
// GMRES(m), right preconditioned (Section 4); flexible variant stores z_j.
// Stopping rule: the estimated residual |g_{j+1}| <= rtol ||b|| ends a cycle;
// the iterate is formed and the true residual decides; restarts otherwise.
// ---------------------------------------------------------------------------
int gmres(a2ls_handle* h, const double* b, double* x, double rtol, int* iters_out, double* relres_out) {
  cudaStream_t st = h->st;
  const int n = h->n;
  const int m = std::max(1, std::min(h->opt.restart > 0 ? h->opt.restart : 30, MD_MAX - 2));
  const bool flexible = h->opt.flexible < 0 ? (h->opt.precision != A2LS_FP64) : (h->opt.flexible != 0);
  const int max_it = h->opt.max_it > 0 ? h->opt.max_it : 1000;
  if (h->gm_restart != m || !h->d_V) {
    if (h->d_V) dfree(h, h->d_V);
    if (h->d_Z) dfree(h, h->d_Z);
    if (h->d_w) dfree(h, h->d_w);
    h->d_V = dalloc<double>(h, (size_t)(m + 1) * n);
    h->d_Z = dalloc<double>(h, (size_t)m * n);
    h->d_w = dalloc<double>(h, (size_t)2 * n);
    h->d_h = dalloc<double>(h, 4 * MD_MAX);
    h->gm_restart = m;
  }
  if (!h->h_pinned) A2LS_CUDA(cudaMallocHost(&h->h_pinned, sizeof(double) * 4 * MD_MAX));
  double* V = h->d_V;
  double* Zs = h->d_Z;
  double* w = h->d_w;
  double* tmp = h->d_w + n;
  double* dh = h->d_h;              // [0, MD_MAX): h1 (+ w.w), [MD_MAX, 2MD_MAX): h2, [2MD_MAX]: |w|^2, [3MD_MAX..): coefs
  double* hp = h->h_pinned;
  Reducer& R = reducer(h);
  const int gb = grid1d(n);
  const double bnorm = nrm2(h, b);
  if (bnorm == 0.0) {
    A2LS_CUDA(cudaMemsetAsync(x, 0, sizeof(double) * n, st));
    if (iters_out) *iters_out = 0;
    if (relres_out) *relres_out = 0.0;
    return A2LS_OK;
  }
  int total = 0;
  std::vector<double> H((m + 1) * m), cs(m), sn(m), g(m + 1), y(m);
  while (true) {
    spmv(h, x, w, b, st);  // w = b - A x
    const double beta = nrm2(h, w);
    if (beta <= rtol * bnorm || total >= max_it) {
      if (iters_out) *iters_out = total;
      if (relres_out) *relres_out = beta / bnorm;
      return beta <= rtol * bnorm ? A2LS_OK : A2LS_ERR_NOT_CONVERGED;
    }
    k_scale<<<gb, 256, 0, st>>>(n, w, V, nullptr, 0, 1.0 / beta);
    A2LS_LAUNCH();
    std::fill(H.begin(), H.end(), 0.0);
    std::fill(g.begin(), g.end(), 0.0);
    g[0] = beta;
    int k = 0;
    for (int j = 0; j < m; ++j) {
      double* vj = V + (size_t)j * n;
      double* zj = flexible ? Zs + (size_t)j * n : tmp;
      apply_preconditioner_graph(h, vj, zj);
      spmv(h, zj, w, nullptr, st);  // w = A z_j
      // CGS2 against V_0..V_j
      multidot(h, V, n, j + 1, w, 1, dh);                 // h1, |w|^2
      cgs_update(h, V, n, j + 1, dh, w, nullptr);
      multidot(h, V, n, j + 1, w, 0, dh + MD_MAX);        // h2
      cgs_update(h, V, n, j + 1, dh + MD_MAX, w, dh + 2 * MD_MAX);  // and |w|^2 after orthogonalisation
      k_scale<<<gb, 256, 0, st>>>(n, w, V + (size_t)(j + 1) * n, dh + 2 * MD_MAX, 1, 0.0);
      A2LS_LAUNCH();
      A2LS_CUDA(cudaMemcpyAsync(hp, dh, sizeof(double) * 3 * MD_MAX, cudaMemcpyDeviceToHost, st));
      A2LS_CUDA(cudaStreamSynchronize(st));
      const double wnorm0 = std::sqrt(std::max(hp[j + 1], 0.0));
      double* col = &H[0];
      for (int i2 = 0; i2 <= j; ++i2) col[i2 * m + j] = hp[i2] + hp[MD_MAX + i2];
      const double hn = std::sqrt(std::max(hp[2 * MD_MAX], 0.0));
      col[(j + 1) * m + j] = hn;
      const bool breakdown = hn <= 1e-14 * wnorm0;
      for (int i2 = 0; i2 < j; ++i2) {
        const double t = cs[i2] * H[i2 * m + j] + sn[i2] * H[(i2 + 1) * m + j];
        H[(i2 + 1) * m + j] = -sn[i2] * H[i2 * m + j] + cs[i2] * H[(i2 + 1) * m + j];
        H[i2 * m + j] = t;
      }
      const double den = std::hypot(H[j * m + j], H[(j + 1) * m + j]);
      cs[j] = H[j * m + j] / den;
      sn[j] = H[(j + 1) * m + j] / den;
      H[j * m + j] = den;
      H[(j + 1) * m + j] = 0.0;
      g[j + 1] = -sn[j] * g[j];
      g[j] = cs[j] * g[j];
      ++total;
      k = j + 1;
      if (std::fabs(g[j + 1]) <= rtol * bnorm || breakdown || total >= max_it) break;
    }
    for (int i2 = k - 1; i2 >= 0; --i2) {
      double s = g[i2];
      for (int c = i2 + 1; c < k; ++c) s -= H[i2 * m + c] * y[c];
      y[i2] = s / H[i2 * m + i2];
    }
    for (int i2 = 0; i2 < k; ++i2) hp[3 * MD_MAX + i2] = y[i2];
    A2LS_CUDA(cudaMemcpyAsync(dh + 3 * MD_MAX, hp + 3 * MD_MAX, sizeof(double) * k, cudaMemcpyHostToDevice, st));
    if (flexible) {
      k_lincomb<<<gb, 256, 0, st>>>(n, Zs, n, k, dh + 3 * MD_MAX, nullptr, x);
      A2LS_LAUNCH();
    } else {
      k_lincomb<<<gb, 256, 0, st>>>(n, V, n, k, dh + 3 * MD_MAX, w, nullptr);
      A2LS_LAUNCH();
      apply_preconditioner_graph(h, w, tmp);
      k_axpy<<<gb, 256, 0, st>>>(n, 1.0, tmp, x);
      A2LS_LAUNCH();
    }
    A2LS_CUDA(cudaStreamSynchronize(st));  // the host buffer hp is reused next cycle
    (void)R;
  }
}

}  // namespace a2ls
