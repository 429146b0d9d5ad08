// Dense real non-symmetric eigensolver for the small Rayleigh-Ritz matrices of
// the local eigenproblems (order <= a few hundred).  Householder reduction to
// upper Hessenberg form, Francis implicit double-shift QR iteration to real
// Schur form (Golub & Van Loan, Matrix Computations, Sections 7.4-7.5),
// eigenvectors by back-substitution on the quasi-triangular factor.
//
// The routines run on a "team": on the GPU the threads of one CTA (lane = thread
// id, size = block size, sync = __syncthreads), on the host a single thread
// (lane 0, size 1, no sync).
// The matrix is row-major with leading dimension ld and lives in memory the
// whole team can address (shared memory on the GPU).
#pragma once

#include <math.h>
#include <string.h>

#ifdef __CUDACC__
#define SE_HD __host__ __device__
#else
#define SE_HD
#endif

namespace a2ls {
namespace se {

struct Team {
  int lane, size;
  int* red = nullptr;  // GPU: one int of shared scratch per warp, for max()
  SE_HD void sync() const {
#ifdef __CUDA_ARCH__
    __syncthreads();
#endif
  }
  // the largest v over the team (on the GPU full warps, and a barrier: shared memory written before the
  // call may be overwritten after it)
  SE_HD int max(int v) const {
#ifdef __CUDA_ARCH__
    v = __reduce_max_sync(0xffffffffu, v);
    __syncthreads();  // red may still be read by the previous call
    if ((lane & 31) == 0) red[lane >> 5] = v;
    __syncthreads();
    for (int w = 0; w < (size >> 5); ++w) v = red[w] > v ? red[w] : v;
#endif
    return v;
  }
};

// Scalar helpers of the arithmetic R the routines run in (double here; other arithmetics provide
// their own overloads of se_abs, se_sqrt and se_dbl next to their type and specialise SeEps).
SE_HD inline double se_abs(double x) { return fabs(x); }
SE_HD inline double se_sqrt(double x) { return sqrt(x); }
SE_HD inline double se_dbl(double x) { return x; }
// acc += a * b in the dot products, and the value of an accumulator (an arithmetic with a cheaper
// unnormalised multiply-add overloads both)
SE_HD inline void se_mac(double& acc, double a, double b) { acc += a * b; }
SE_HD inline double se_fin(double a) { return a; }
// Whether hessenberg() and schur() form their reflectors from se_rsqrt(a) = 1 / sqrt(a), se_recip12(b) = 1 / b for b in
// [1, 2], se_scale_to_one(a), a factor that brings a to about 1, se_pow2(a) and se_pow2_inv(p), a's power of two
// and its inverse, and the warp sums and maxima se_warp_sum and se_warp_maxabs (double-float brings them), or keep
// to the library's roots and quotients.  FP64 keeps to those and with them its results
// bit for bit: the block Krylov iteration amplifies a changed rounding until the eigenvectors, kept at a
// residual of 1e-10, differ at that size, and with them the ninth digit of the preconditioner, which FP64
// callers compare.
template <class R> struct SeFast { static constexpr bool v = false; };
SE_HD inline bool se_is_zero(double a) {
#ifdef __CUDA_ARCH__
  return (__double_as_longlong(a) << 1) == 0;
#else
  return a == 0.0;
#endif
}
SE_HD inline double se_warp_get(double v, int lane) {
#ifdef __CUDA_ARCH__
  return __shfl_sync(0xffffffffu, v, lane);
#else
  (void)lane;
  return v;
#endif
}
template <class R> struct SeEps {
  static constexpr double v = 2.220446049250313e-16;  // machine epsilon of R
  static constexpr double big = 1e100;                // rescaling threshold of the back substitution
};

template <class R>
SE_HD inline R sgn(R a, R b) { return b >= R(0.0) ? se_abs(a) : -se_abs(a); }
SE_HD inline double sgn(double a, double b) {
#ifdef __CUDA_ARCH__
  // the same rule (-0 counts as positive) in bits, b's before a's: a is the end of a chain of FP64 instructions
  const int hi = __double2hiint(b), sign = ((hi << 1) | __double2loint(b)) != 0 ? hi & (int)0x80000000 : 0;
  return __hiloint2double((__double2hiint(a) & 0x7fffffff) | sign, __double2loint(a));
#else
  return b >= 0.0 ? fabs(a) : -fabs(a);
#endif
}

// x_r -= d v_r for r = 0 .. n-1 (x with stride st), four elements loaded ahead of their stores: x and v may
// be the same kind of memory, so the compiler may not move a load over a store by itself
template <class R>
SE_HD inline void subtract_multiple(R* x, int st, const R* v, int n, R d) {
  int r = 0;
  for (; r + 4 <= n; r += 4) {
    R a[4], b[4];
    for (int u = 0; u < 4; ++u) {
      a[u] = x[(r + u) * st];
      b[u] = v[r + u];
    }
    for (int u = 0; u < 4; ++u) x[(r + u) * st] = a[u] - d * b[u];
  }
  for (; r < n; ++r) x[r * st] -= d * v[r];
}

// sum of x_r v_r for r = 0 .. n-1
template <class R>
SE_HD inline R strided_dot(const R* x, int st, const R* v, int n) {
  R d = 0.0;
#ifdef __CUDACC__
#pragma unroll 4
#endif
  for (int r = 0; r < n; ++r) se_mac(d, v[r], x[r * st]);
  return se_fin(d);
}

// Reduce H (m x m) to upper Hessenberg form, accumulating the orthogonal factor in Q (Q <- Q P).
// v: scratch of m values.  Each reflector takes two phases of the team: the left update (one column
// per thread) together with the first rows of Q, then the right update of H (one row per thread)
// together with the remaining rows of Q (with 128 threads and m <= 85 no thread holds more than one
// item per phase).
template <class R>
SE_HD inline void hessenberg(R* H, int ld, R* Q, int ldq, int m, R* v, const Team& t) {
  for (int k = 0; k + 2 < m; ++k) {
    [[maybe_unused]] R up = 1.0;
    R x0, alpha, beta;
    if constexpr (SeFast<R>::v) {
      // Householder vector for x = H[k+1.., k], scaled; every warp sums |x|^2 for itself, in the same order
#ifdef __CUDA_ARCH__
      const int l0 = t.lane & 31, ls = 32;
#else
      const int l0 = 0, ls = 1;
#endif
      R xm = 0.0;
      for (int r = k + 1 + l0; r < m; r += ls) {
        const R a = se_abs(H[r * ld + k]);
        if (a > xm) xm = a;
      }
      up = se_pow2(se_warp_maxabs(xm));
      const R dn = se_pow2_inv(up);
      R nrm2 = 0.0;
      for (int r = k + 1 + l0; r < m; r += ls) {
        const R a = H[r * ld + k] * dn;
        se_mac(nrm2, a, a);
      }
      nrm2 = se_warp_sum(se_fin(nrm2));
      if (se_is_zero(nrm2)) continue;
      const R rn = se_rsqrt(nrm2);
      x0 = H[(k + 1) * ld + k] * dn;
      alpha = -sgn(nrm2 * rn, x0);
      // v = x - alpha e1; P = I - beta v v^T with beta = 2 / v^T v, v^T v = 2 |x| (|x| + |x0|)
      beta = rn * rn * se_recip12(R(1.0) + se_abs(x0) * rn);
      t.sync();
      for (int r = k + 1 + t.lane; r < m; r += t.size) v[r] = (r == k + 1) ? (x0 - alpha) : H[r * ld + k] * dn;
    } else {
      // Householder vector for x = H[k+1.., k]
      R nrm2 = 0.0;
      for (int r = k + 1; r < m; ++r) se_mac(nrm2, H[r * ld + k], H[r * ld + k]);
      nrm2 = se_fin(nrm2);
      const R nrm = se_sqrt(nrm2);
      if (nrm == 0.0) continue;
      x0 = H[(k + 1) * ld + k];
      alpha = -sgn(nrm, x0);
      // v = x - alpha e1, scaled so that P = I - 2 v v^T / (v^T v); v^T v = 2 nrm |x0 - alpha|
      const R vtv = nrm2 - x0 * x0 + (x0 - alpha) * (x0 - alpha);
      if (vtv == 0.0) continue;
      t.sync();
      for (int r = k + 1 + t.lane; r < m; r += t.size) v[r] = (r == k + 1) ? (x0 - alpha) : H[r * ld + k];
      beta = 2.0 / vtv;
    }
    t.sync();
    const int len = m - k - 1;
    const int ncol = m - k;                                  // left update: columns k..m-1
    const int qa = (t.size > ncol) ? ((t.size - ncol < m) ? t.size - ncol : m) : 0;  // Q rows in phase 1
    for (int idx = t.lane; idx < ncol + qa; idx += t.size) {
      R* x = idx < ncol ? H + (k + 1) * ld + k + idx : Q + (idx - ncol) * ldq + k + 1;
      const int st = idx < ncol ? ld : 1;
      const R d = strided_dot(x, st, v + k + 1, len) * beta;
      subtract_multiple(x, st, v + k + 1, len, d);
    }
    t.sync();
    // right: all rows of H, columns k+1..; the remaining rows of Q
    for (int idx = t.lane; idx < m + (m - qa); idx += t.size) {
      R* x = idx < m ? H + idx * ld + k + 1 : Q + (qa + idx - m) * ldq + k + 1;
      const R d = strided_dot(x, 1, v + k + 1, len) * beta;
      subtract_multiple(x, 1, v + k + 1, len, d);
    }
    t.sync();
    for (int r = k + 1 + t.lane; r < m; r += t.size) H[r * ld + k] = r == k + 1 ? alpha * up : R(0.0);
    t.sync();
  }
}

// The largest lo <= hi whose subdiagonal entry is negligible (0 if there is none), one entry per thread: below
// leps times its two diagonal neighbours or below eps times hnorm.
template <class R>
SE_HD inline int first_negligible(const R* H, int ld, int hi, R leps, R eps, R hnorm, const Team& t) {
  int lo = 0;
  for (int j = hi - t.lane; j > 0; j -= t.size) {
    const R s = se_abs(H[(j - 1) * ld + j - 1]) + se_abs(H[j * ld + j]);
    const R sub = se_abs(H[j * ld + j - 1]);
    if (sub <= leps * s || sub <= eps * hnorm) {
      lo = j;
      break;
    }
  }
  return t.max(lo);
}

// ---- with the library's square root and division ----
// GB300's FP64 pipe takes about 64 cycles for every warp instruction of an SM quarter, however few lanes
// are active, so the chain of the reflectors' FP64 instructions is the time: the next reflector's three
// entries and its two quotients go to lanes of one warp (order 48: 7.5 -> 5.2 million cycles, the same
// bits).

// Apply a 2-element reflector I - beta u u^T with u = (1, u1) to rows k, k+1 of H from the left (columns c0..m-1) and to
// columns k, k+1 from the right (rows 0..r1) and to Q's columns.
template <class R>
SE_HD inline void apply_reflector2(R* H, int ld, R* Q, int ldq, int m, int k, R u1, R beta, int c0, int r1, const Team& t) {
  auto reflect = [&](R* a, int st) {
    R d = a[0] + u1 * a[st];
    d *= beta;
    a[0] -= d;
    a[st] -= d * u1;
  };
  for (int c = c0 + t.lane; c < m; c += t.size) reflect(H + k * ld + c, ld);
  t.sync();
  for (int r = t.lane; r <= r1; r += t.size) reflect(H + r * ld + k, 1);
  for (int r = t.lane; r < m; r += t.size) reflect(Q + r * ldq + k, 1);
  t.sync();
}

// Householder reflector mapping (x, y, z) to (alpha, 0, 0): returns alpha, beta and u = (1, u1, u2).
// With v = (v0, y, z), v0 = x - alpha, v^T v = 2 |alpha| |v0|, so beta = 2 v0^2 / v^T v = v0 / (-alpha).
template <class R>
SE_HD inline bool make_reflector_div(R x, R y, R z, R& u1, R& u2, R& beta, R& alpha) {
  R nrm = se_sqrt(x * x + y * y + z * z);
  if (nrm == 0.0) return false;
  alpha = -sgn(nrm, x);
  R v0 = x - alpha;
  if (v0 == 0.0) return false;
  R iv;
#ifdef __CUDA_ARCH__
  {
    // the two quotients in the even and the odd lanes, one division long
    const int lane = threadIdx.x & 31;
    const R q = ((lane & 1) ? v0 : R(1.0)) / ((lane & 1) ? -alpha : v0);
    iv = se_warp_get(q, lane & ~1);
    beta = se_warp_get(q, lane | 1);
  }
#else
  iv = R(1.0) / v0;
  beta = v0 / (-alpha);
#endif
  u1 = y * iv;
  u2 = z * iv;
  return true;
}

// Make a 2x2 diagonal block with real eigenvalues upper triangular by a rotation (rows/cols p, p+1).
template <class R>
SE_HD inline void split_2x2_div(R* H, int ld, R* Q, int ldq, int m, int p, const Team& t) {
  t.sync();
  R a = H[p * ld + p], b = H[p * ld + p + 1], c = H[(p + 1) * ld + p], d = H[(p + 1) * ld + p + 1];
  R hm = 0.5 * (a - d);
  R disc = hm * hm + b * c;
  if (disc < 0.0 || c == 0.0) return;
  // eigenvalue closest to d: lambda = d + (hm +- se_sqrt(disc)) ... pick the one of larger magnitude shift
  R sq = se_sqrt(disc);
  R lam = 0.5 * (a + d) + (hm >= 0 ? sq : -sq);
  // eigenvector (lam - d, c) of the block; rotation taking it to e1
  R x = lam - d, y = c;
  R r = se_sqrt(x * x + y * y);
  if (r == 0.0) return;
  R cs = x / r, sn = y / r;
  // rows p, p+1: G^T H
  for (int col = p + t.lane; col < m; col += t.size) {
    R h1 = H[p * ld + col], h2 = H[(p + 1) * ld + col];
    H[p * ld + col] = cs * h1 + sn * h2;
    H[(p + 1) * ld + col] = -sn * h1 + cs * h2;
  }
  t.sync();
  for (int row = t.lane; row <= p + 1; row += t.size) {
    R h1 = H[row * ld + p], h2 = H[row * ld + p + 1];
    H[row * ld + p] = cs * h1 + sn * h2;
    H[row * ld + p + 1] = -sn * h1 + cs * h2;
  }
  for (int row = t.lane; row < m; row += t.size) {
    R q1 = Q[row * ldq + p], q2 = Q[row * ldq + p + 1];
    Q[row * ldq + p] = cs * q1 + sn * q2;
    Q[row * ldq + p + 1] = -sn * q1 + cs * q2;
  }
  t.sync();
  if (t.lane == 0) H[(p + 1) * ld + p] = 0.0;
  t.sync();
}

// schur() with the library's square root and division (see there for the arguments)
template <class R>
SE_HD inline int schur_single(R* H, int ld, R* Q, int ldq, int m, double hnorm_, const Team& t, R* snap,
                              double local_tol) {
  const R eps = R(SeEps<R>::v), hnorm = R(hnorm_);
  const R leps = R(local_tol > SeEps<R>::v ? local_tol : SeEps<R>::v);
  int hi = m - 1, iter = 0, total = 0;
  while (hi >= 0) {
    int lo = first_negligible(H, ld, hi, leps, eps, hnorm, t);
    if (lo > 0) {
      t.sync();
      if (t.lane == 0) H[lo * ld + lo - 1] = 0.0;
      t.sync();
    }
    if (lo == hi) {
      --hi;
      iter = 0;
      continue;
    }
    if (lo == hi - 1) {
      split_2x2_div(H, ld, Q, ldq, m, lo, t);
      hi -= 2;
      iter = 0;
      continue;
    }
    ++iter;
    if (++total > 60 * m) return -1;
    // Shifts: the eigenvalues of the trailing 2x2 block (a real pair is replaced by its member
    // closer to the last diagonal entry, used twice), or an exceptional pair every 11th step.
    R s1r, s1i, s2r, s2i;
    {
      R a, b, c, d;
      if (iter % 11 == 10) {
        const R w = se_abs(H[hi * ld + hi - 1]) + se_abs(H[(hi - 1) * ld + hi - 2]);
        a = 0.75 * w + H[hi * ld + hi];
        b = -0.4375 * w;
        c = w;
        d = a;
      } else {
        a = H[(hi - 1) * ld + hi - 1];
        b = H[(hi - 1) * ld + hi];
        c = H[hi * ld + hi - 1];
        d = H[hi * ld + hi];
      }
      const R hm = 0.5 * (a - d);
      const R disc = hm * hm + b * c;
      const R mean = 0.5 * (a + d);
      if (disc >= 0.0) {
        const R sq = se_sqrt(disc);
        const R r1 = mean + sq, r2 = mean - sq;
        const R sh = (se_abs(r1 - d) <= se_abs(r2 - d)) ? r1 : r2;
        s1r = s2r = sh;
        s1i = s2i = 0.0;
      } else {
        s1r = s2r = mean;
        s1i = se_sqrt(-disc);
        s2i = -s1i;
      }
    }
    // first column of (H - s1)(H - s2), formed from differences to avoid cancellation
    R x, y, z;
    {
      const R h00 = H[lo * ld + lo], h01 = H[lo * ld + lo + 1], h10 = H[(lo + 1) * ld + lo];
      const R h11 = H[(lo + 1) * ld + lo + 1], h21 = H[(lo + 2) * ld + lo + 1];
      const R sc = se_abs(h00 - s2r) + se_abs(s2i) + se_abs(h10);
      const R g = (sc > 0.0) ? h10 / sc : 0.0;
      x = g * h01 + (h00 - s1r) * ((h00 - s2r) / (sc > 0.0 ? sc : 1.0)) - s1i * (s2i / (sc > 0.0 ? sc : 1.0));
      y = g * (h00 + h11 - s1r - s2r);
      z = g * h21;
    }
    // Bulge chase.  For k > lo the reflector is built from column k-1 (rows k..k+2), which it maps to
    // (alpha, 0, 0) exactly; that column is therefore not part of the left update but written
    // directly, after the barrier that separates every thread's read of (x, y, z) from the writes,
    // which keeps each step at two barriers.  The next step's reflector comes from column k after
    // this step's right update; one thread recomputes its three entries from a snapshot of rows
    // k+1..k+3 (columns k..k+2) taken in the left phase and forms the reflector while the others run
    // the right update, instead of every thread forming it after that update (the entries are the
    // values the right update writes).
    t.sync();  // the shift and deflation reads above precede the first update
    R u1, u2, beta, alpha;
    bool have = make_reflector_div(x, y, z, u1, u2, beta, alpha);
    for (int k = lo; k <= hi - 2; ++k) {
      const bool more = k + 1 <= hi - 2;  // a next step exists (then k + 3 <= hi)
      R nu1 = R(0.0), nu2 = R(0.0), nbeta = R(0.0), nalpha = R(0.0);
      bool nhave = false;
      if (have) {
        const int c0 = k > lo ? k : lo;
        const int r1 = (k + 3 <= hi) ? k + 3 : hi;
        // phase 1: rows k..k+2 from the left (columns c0..m-1) and the first qa rows of Q; phase 2:
        // columns k..k+2 from the right (rows 0..r1) and the remaining rows of Q (Q's update depends
        // on the reflector only, so it fills the threads that the H updates leave idle)
        const int ncol = m - c0;
        const int qa = (t.size > ncol) ? ((t.size - ncol < m) ? t.size - ncol : m) : 0;
        for (int idx = t.lane; idx < ncol + qa; idx += t.size) {
          R* a;
          int st;
          if (idx < ncol) {
            a = H + k * ld + c0 + idx;
            st = ld;
          } else {
            a = Q + (idx - ncol) * ldq + k;
            st = 1;
          }
          R d = a[0];
          se_mac(d, u1, a[st]);
          se_mac(d, u2, a[2 * st]);
          d = se_fin(d) * beta;
          a[0] -= d;
          a[st] -= d * u1;
          a[2 * st] -= d * u2;
          if (more && idx < 3) {  // column c0 + idx = k + idx
            snap[idx] = a[st];
            snap[3 + idx] = a[2 * st];
            snap[6 + idx] = H[(k + 3) * ld + k + idx];
          }
        }
        t.sync();
        if (k > lo && t.lane == 0) {
          H[k * ld + k - 1] = alpha;
          H[(k + 1) * ld + k - 1] = 0.0;
          H[(k + 2) * ld + k - 1] = 0.0;
        }
        // the last warp, usually idle in the right update, with one lane per entry
#ifdef __CUDA_ARCH__
        const bool forms = t.lane >= t.size - 32;
#else
        const bool forms = true;
#endif
        if (more && forms) {
          auto entry = [&](int rr) {
            const R a0 = snap[3 * rr], a1 = snap[3 * rr + 1], a2 = snap[3 * rr + 2];
            R d = a0;
            se_mac(d, u1, a1);
            se_mac(d, u2, a2);
            d = se_fin(d) * beta;
            return a0 - d;
          };
#ifdef __CUDA_ARCH__
          const R e = entry((t.lane & 31) < 3 ? t.lane & 31 : 2);
          const R v[3] = {se_warp_get(e, 0), se_warp_get(e, 1), se_warp_get(e, 2)};
#else
          const R v[3] = {entry(0), entry(1), entry(2)};
#endif
          const bool ok = make_reflector_div(v[0], v[1], v[2], nu1, nu2, nbeta, nalpha);
          if (t.lane == t.size - 1) {
            snap[9] = nu1;
            snap[10] = nu2;
            snap[11] = nbeta;
            snap[12] = nalpha;
            snap[13] = ok ? R(1.0) : R(0.0);
          }
        }
        for (int idx = t.lane; idx < (r1 + 1) + (m - qa); idx += t.size) {
          R* a = (idx <= r1) ? H + idx * ld + k : Q + (qa + idx - (r1 + 1)) * ldq + k;
          R d = a[0];
          se_mac(d, u1, a[1]);
          se_mac(d, u2, a[2]);
          d = se_fin(d) * beta;
          a[0] -= d;
          a[1] -= d * u1;
          a[2] -= d * u2;
        }
        t.sync();
        if (more) {
          nu1 = snap[9];
          nu2 = snap[10];
          nbeta = snap[11];
          nalpha = snap[12];
          nhave = !se_is_zero(snap[13]);
        }
      } else if (more) {
        nhave = make_reflector_div(H[(k + 1) * ld + k], H[(k + 2) * ld + k], H[(k + 3) * ld + k], nu1, nu2, nbeta,
                               nalpha);
      }
      u1 = nu1;
      u2 = nu2;
      beta = nbeta;
      alpha = nalpha;
      have = nhave;
    }
    x = H[(hi - 1) * ld + hi - 2];
    y = H[hi * ld + hi - 2];
    // final 2-element reflector on rows hi-1, hi
    {
      R u1, u2, beta, alpha;
      if (make_reflector_div<R>(x, y, R(0.0), u1, u2, beta, alpha)) {
        t.sync();
        apply_reflector2<R>(H, ld, Q, ldq, m, hi - 1, u1, beta, hi - 2, hi, t);
        if (t.lane == 0) H[hi * ld + hi - 2] = 0.0;
        t.sync();
      }
    }
  }
  return 0;
}

// ---- reflectors without square roots and quotients ----

// Householder reflector mapping (x, y, z) to (alpha, 0, 0): returns alpha, beta and u = (1, u1, u2).
// With v = (v0, y, z), v0 = x - alpha, v^T v = 2 |alpha| |v0|, so beta = 2 v0^2 / v^T v = v0 / (-alpha).
// (0, 0, 0) gives beta = 0 and alpha = x: no reflection.
// The chain of a sweep's reflectors is what bounds the Schur iteration, so it has no square root and no
// division: with r = 1 / |(x, y, z)|, beta = 1 + |x| r (between 1 and 2) and 1 / v0 = sign(x) r / beta.  The
// three are scaled first: entries of 1e-16 and less, as a converging block has them, would lose the low
// parts of their squares to FP32's exponent range, and the reflector its orthogonality.
template <class R>
SE_HD inline void make_reflector(R x, R y, R z, R& u1, R& u2, R& beta, R& alpha) {
  R xm = se_abs(x);
  if (se_abs(y) > xm) xm = se_abs(y);
  if (se_abs(z) > xm) xm = se_abs(z);
  const R up = se_pow2(xm), dn = se_pow2_inv(up);
  x *= dn;
  y *= dn;
  z *= dn;
  const R s = x * x + y * y + z * z;
  if (se_is_zero(s)) {
    u1 = u2 = beta = R(0.0);
    alpha = x;
    return;
  }
  const R r = se_rsqrt(s);
  beta = R(1.0) + se_abs(x) * r;
  alpha = -sgn(s * r, x) * up;
  const R iv = sgn(r * se_recip12(beta), x);
  u1 = y * iv;
  u2 = z * iv;
}

// Make a 2x2 diagonal block with real eigenvalues upper triangular by a rotation (rows/cols p, p+1).
template <class R>
SE_HD inline void split_2x2(R* H, int ld, R* Q, int ldq, int m, int p, const Team& t) {
  t.sync();
  R a = H[p * ld + p], b = H[p * ld + p + 1], c = H[(p + 1) * ld + p], d = H[(p + 1) * ld + p + 1];
  R hm = 0.5 * (a - d);
  R disc = hm * hm + b * c;
  if (disc < 0.0 || c == 0.0) return;
  // eigenvalue closest to d: lambda = d + (hm +- sqrt(disc)) ... pick the one of larger magnitude shift
  R sq = se_is_zero(disc) ? R(0.0) : disc * se_rsqrt(disc);
  R lam = 0.5 * (a + d) + (hm >= 0 ? sq : -sq);
  // eigenvector (lam - d, c) of the block (scaled); rotation taking it to e1
  R x = lam - d, y = c;
  const R dn = se_pow2_inv(se_pow2(se_abs(x) > se_abs(y) ? se_abs(x) : se_abs(y)));
  x *= dn;
  y *= dn;
  const R r2 = x * x + y * y;
  if (se_is_zero(r2)) return;
  const R ri = se_rsqrt(r2);
  const R cs = x * ri, sn = y * ri;
  // rows p, p+1: G^T H
  for (int col = p + t.lane; col < m; col += t.size) {
    R h1 = H[p * ld + col], h2 = H[(p + 1) * ld + col];
    H[p * ld + col] = cs * h1 + sn * h2;
    H[(p + 1) * ld + col] = -sn * h1 + cs * h2;
  }
  t.sync();
  for (int row = t.lane; row <= p + 1; row += t.size) {
    R h1 = H[row * ld + p], h2 = H[row * ld + p + 1];
    H[row * ld + p] = cs * h1 + sn * h2;
    H[row * ld + p + 1] = -sn * h1 + cs * h2;
  }
  for (int row = t.lane; row < m; row += t.size) {
    R q1 = Q[row * ldq + p], q2 = Q[row * ldq + p + 1];
    Q[row * ldq + p] = cs * q1 + sn * q2;
    Q[row * ldq + p + 1] = -sn * q1 + cs * q2;
  }
  t.sync();
  if (t.lane == 0) H[(p + 1) * ld + p] = 0.0;
  t.sync();
}

// The scratch schur() wants: the nine entries of the next reflector's snapshot and, from SE_REFL, two sets of u1, u2,
// beta, alpha.
constexpr int SE_REFL = 9;
constexpr int SE_SNAP = SE_REFL + 8;

// The shift pair (s1r, s2r, s1i, s2i) of the 2 x 2 block a, b; c, d: a real pair is replaced by its member
// closer to d, used twice.
template <class R>
SE_HD inline void shift_pair(R a, R b, R c, R d, R* s) {
  const R hm = 0.5 * (a - d);
  const R disc = hm * hm + b * c;
  const R mean = 0.5 * (a + d);
  if (disc >= 0.0) {
    const R sq = se_is_zero(disc) ? R(0.0) : disc * se_rsqrt(disc);
    const R r1 = mean + sq, r2 = mean - sq;
    s[0] = s[1] = (se_abs(r1 - d) <= se_abs(r2 - d)) ? r1 : r2;
    s[2] = s[3] = 0.0;
  } else {
    s[0] = s[1] = mean;
    s[2] = -disc * se_rsqrt(-disc);
    s[3] = -s[2];
  }
}

// One sweep over the active block lo .. hi (see schur); exceptional: with shifts of the size of the last
// subdiagonal entries.  Starts after the team has seen H, ends with a barrier.
template <class R>
SE_HD inline void se_sweep(R* H, int ld, R* Q, int ldq, int m, int lo, int hi, bool exceptional, const Team& t,
                           R* snap) {
  // On the GPU the last warp forms the reflectors (its lane 0 keeps them); the right updates and Q are left to
  // the other warps.
#ifdef __CUDA_ARCH__
  const int nwork = t.size - 32, rl = t.lane - nwork;
  const bool maker = rl >= 0, keeps = rl == 0;
#else
  const int nwork = t.size;
  const bool maker = true, keeps = true;
#endif
  if (maker) {
    R a, b, c, d;
    if (exceptional) {
      const R e = se_abs(H[hi * ld + hi - 1]) + se_abs(H[(hi - 1) * ld + hi - 2]);
      a = 0.75 * e + H[hi * ld + hi];
      b = -0.4375 * e;
      c = e;
      d = a;
    } else {
      a = H[(hi - 1) * ld + hi - 1];
      b = H[(hi - 1) * ld + hi];
      c = H[hi * ld + hi - 1];
      d = H[hi * ld + hi];
    }
    R s[4];
    shift_pair(a, b, c, d, s);
    // the first column of (H - s1)(H - s2), formed from differences to avoid cancellation, times a factor
    // that keeps it in range (only its direction matters)
    const R s1r = s[0], s2r = s[1], s1i = s[2], s2i = s[3];
    const R h00 = H[lo * ld + lo], h01 = H[lo * ld + lo + 1], h10 = H[(lo + 1) * ld + lo];
    const R h11 = H[(lo + 1) * ld + lo + 1], h21 = H[(lo + 2) * ld + lo + 1];
    const R sc = se_abs(h00 - s2r) + se_abs(s2i) + se_abs(h10);
    const R f = se_is_zero(sc) ? R(1.0) : se_scale_to_one(sc);
    const R g = h10 * f;
    R r[4];
    make_reflector<R>(g * h01 + (h00 - s1r) * ((h00 - s2r) * f) - s1i * (s2i * f), g * (h00 + h11 - s1r - s2r),
                      g * h21, r[0], r[1], r[2], r[3]);
    if (keeps)
      for (int u = 0; u < 4; ++u) snap[SE_REFL + u] = r[u];
  }
  t.sync();  // the reads of H above precede the first update
  // The bulge is at row k.  For k > lo its reflector was built from column k - 1 (rows k .. k + 2), which it
  // maps to (alpha, 0, 0) exactly; that column is therefore not part of the left update but written directly,
  // after the barrier that separates the reads of it from the writes.  At k = hi - 1 the reflector has two
  // rows.  The next reflector comes from column k after this step's right update; its three entries are
  // recomputed from a snapshot of rows k + 1 .. k + 3 (columns k .. k + 2) taken in the left phase, and the
  // reflector is formed while the others run the right update (the entries are the values the right update
  // writes).
  auto reflect = [&](R* a, int st, const R* r, bool three) {
    const R u1 = r[0], u2 = r[1], beta = r[2];
    const R a0 = a[0], a1 = a[st], a2 = three ? a[2 * st] : R(0.0);
    R d = a0;
    se_mac(d, u1, a1);
    se_mac(d, u2, a2);
    d = se_fin(d) * beta;
    a[0] = a0 - d;
    a[st] = a1 - d * u1;
    if (three) a[2 * st] = a2 - d * u2;
  };
  for (int k = lo; k < hi; ++k) {
    const R* r = snap + SE_REFL + 4 * ((k - lo) & 1);
    const bool three = k <= hi - 2;
    // phase 1: rows k .. k + 2 from the left (columns k .. m - 1), one column per item
    for (int c = k + t.lane; c < m; c += t.size) {
      R* a = H + k * ld + c;
      reflect(a, ld, r, three);
      if (c < k + 3 && three) {
        R* v = snap + (c - k);
        v[0] = a[ld];
        v[3] = a[2 * ld];
        v[6] = k + 3 <= hi ? a[3 * ld] : R(0.0);
      }
    }
    t.sync();
    // phase 2: columns k .. k + 2 from the right (rows 0 .. k + 3) and Q, one row per item; the next reflector
    if (maker) {
      const R u1 = r[0], u2 = r[1], beta = r[2];
      auto entry = [&](int rr) {
        const R a0 = snap[3 * rr], a1 = snap[3 * rr + 1], a2 = snap[3 * rr + 2];
        R d = a0;
        se_mac(d, u1, a1);
        se_mac(d, u2, a2);
        d = se_fin(d) * beta;
        return a0 - d;
      };
      if (three) {
        R v[3], n[4];
#ifdef __CUDA_ARCH__
        const R e = entry(rl < 3 ? rl : 2);   // one lane per entry
        for (int rr = 0; rr < 3; ++rr) v[rr] = se_warp_get(e, rr);
#else
        for (int rr = 0; rr < 3; ++rr) v[rr] = entry(rr);
#endif
        make_reflector<R>(v[0], v[1], v[2], n[0], n[1], n[2], n[3]);
        if (keeps)
          for (int u = 0; u < 4; ++u) snap[SE_REFL + 4 * ((k + 1 - lo) & 1) + u] = n[u];
      }
      if (keeps && k > lo) {
        H[k * ld + k - 1] = r[3];
        H[(k + 1) * ld + k - 1] = 0.0;
        if (three) H[(k + 2) * ld + k - 1] = 0.0;
      }
    }
    if (t.lane < nwork) {
      const int rows = (k + 3 <= hi ? k + 3 : hi) + 1;
      for (int e = t.lane; e < rows + m; e += nwork)
        reflect((e < rows ? H + e * ld : Q + (e - rows) * ldq) + k, 1, r, three);
    }
    t.sync();
  }
}

// schur() without square roots and quotients (see there for the arguments)
template <class R>
SE_HD inline int schur_fast(R* H, int ld, R* Q, int ldq, int m, double hnorm_, const Team& t, R* snap,
                            double local_tol) {
  const R eps = R(SeEps<R>::v), hnorm = R(hnorm_);
  const R leps = R(local_tol > SeEps<R>::v ? local_tol : SeEps<R>::v);
  int hi = m - 1, iter = 0, total = 0;
  while (hi >= 0) {
    const int lo = first_negligible(H, ld, hi, leps, eps, hnorm, t);
    if (lo > 0) {
      t.sync();
      if (t.lane == 0) H[lo * ld + lo - 1] = 0.0;
      t.sync();
    }
    if (lo == hi) {
      --hi;
      iter = 0;
      continue;
    }
    if (lo == hi - 1) {
      split_2x2(H, ld, Q, ldq, m, lo, t);
      hi -= 2;
      iter = 0;
      continue;
    }
    ++iter;
    if (++total > 60 * m) return -1;
    se_sweep(H, ld, Q, ldq, m, lo, hi, iter % 11 == 10, t, snap);
  }
  return 0;
}

// Francis implicit double-shift QR on an upper Hessenberg H, full Schur form, Q accumulated.
// A subdiagonal entry is neglected when it is below eps times its two diagonal
// neighbours or below eps times hnorm (the largest entry of the input), which keeps
// clusters of eigenvalues near zero from stalling the iteration; the result is
// backward stable relative to hnorm.  Returns 0 on success, -1 on no convergence.
// snap: SE_SNAP values of scratch shared by the team (may be null for a one-thread team).
// local_tol (>= the machine epsilon of R; 0 selects it): the neighbour-relative test may use a looser
// threshold when the caller needs the Schur form only to that relative accuracy; the test against
// hnorm always uses the machine epsilon.
//
// A sweep's time is the chain of its reflectors, each formed from what the one before it leaves, and not
// the updates.  Three bulges chased in step with one another (the small-bulge multishift iteration of Braman, Byers
// and Mathias, SIAM J. Matrix Anal. Appl. 23, 2002) shorten it by a further third, but neglect other entries: with
// a loose local_tol the Ritz vectors then differ by up to 6e-5 from one bulge's, as far as these are from the
// exact Schur form's.  Set-up and solve with 256 subdomains of order 72: 120.5 ms with roots and quotients, 116.2
// without; later, with the other kernels faster, 95.8 against 93.4 with three bulges.
template <class R>
SE_HD inline int schur(R* H, int ld, R* Q, int ldq, int m, double hnorm, const Team& t, R* snap = nullptr,
                       double local_tol = 0.0) {
  R snap_local[SE_SNAP];
  if (!snap) snap = snap_local;
  if constexpr (SeFast<R>::v) return schur_fast(H, ld, Q, ldq, m, hnorm, t, snap, local_tol);
  else return schur_single(H, ld, Q, ldq, m, hnorm, t, snap, local_tol);
}

// Eigenvalues of the quasi-triangular S: wr[j], wi[j] (a complex pair occupies j, j+1 with wi[j] > 0).
template <class R>
SE_HD inline void schur_eigenvalues(const R* S, int ld, int m, double* wr, double* wi) {
  int j = 0;
  while (j < m) {
    if (j + 1 < m && S[(j + 1) * ld + j] != 0.0) {
      R a = S[j * ld + j], b = S[j * ld + j + 1], c = S[(j + 1) * ld + j], d = S[(j + 1) * ld + j + 1];
      R hm = 0.5 * (a - d);
      R disc = hm * hm + b * c;
      R re = 0.5 * (a + d);
      R im = se_sqrt(se_abs(disc));
      if (disc >= 0.0) {  // not split (should not happen after split_2x2); report real values
        wr[j] = se_dbl(re + im);
        wr[j + 1] = se_dbl(re - im);
        wi[j] = wi[j + 1] = 0.0;
      } else {
        wr[j] = wr[j + 1] = se_dbl(re);
        wi[j] = se_dbl(im);
        wi[j + 1] = -se_dbl(im);
      }
      j += 2;
    } else {
      wr[j] = se_dbl(S[j * ld + j]);
      wi[j] = 0.0;
      j += 1;
    }
  }
}

// Eigenvector of the quasi-triangular S for the eigenvalue at position p (real: x; complex
// pair starting at p: x + i y).  x, y have m entries; entries above p are filled, below zero.
template <class R>
SE_HD inline void schur_vector(const R* S, int ld, int m, int p, double lr_, double li_, R* x, R* y,
                               double snorm) {
  const R small = R(1e-300 + SeEps<R>::v * snorm);
  const R lr = R(lr_), li = R(li_);
  for (int q = 0; q < m; ++q) {
    x[q] = 0.0;
    y[q] = 0.0;
  }
  int top;
  if (li == 0.0) {
    x[p] = 1.0;
    top = p - 1;
  } else {
    // block rows p, p+1: (a - lambda) x_p + b x_{p+1} = 0 -> x_p = b, x_{p+1} = lambda - a
    R a = S[p * ld + p], b = S[p * ld + p + 1];
    x[p] = b;
    y[p] = 0.0;
    x[p + 1] = lr - a;
    y[p + 1] = li;
    top = p - 1;
  }
  const int last = (li == 0.0) ? p : p + 1;
  R mx = 0.0;
  for (int c = top + 1; c <= last; ++c) {
    const R v = se_abs(x[c]) + se_abs(y[c]);
    if (v > mx) mx = v;
  }
  int q = top;
  while (q >= 0) {
    if (q > 0 && S[q * ld + q - 1] != 0.0) {
      // 2x2 block rows q-1, q: solve (S_blk - lambda I) [u; w] = -rhs
      R r1r = 0, r1i = 0, r2r = 0, r2i = 0;
      for (int c = q + 1; c <= last; ++c) {
        se_mac(r1r, S[(q - 1) * ld + c], x[c]);
        se_mac(r1i, S[(q - 1) * ld + c], y[c]);
        se_mac(r2r, S[q * ld + c], x[c]);
        se_mac(r2i, S[q * ld + c], y[c]);
      }
      r1r = se_fin(r1r);
      r1i = se_fin(r1i);
      r2r = se_fin(r2r);
      r2i = se_fin(r2i);
      R a11r = S[(q - 1) * ld + q - 1] - lr, a11i = -li;
      R a12 = S[(q - 1) * ld + q], a21 = S[q * ld + q - 1];
      R a22r = S[q * ld + q] - lr, a22i = -li;
      // det = a11*a22 - a12*a21 (complex)
      R dr = a11r * a22r - a11i * a22i - a12 * a21;
      R di = a11r * a22i + a11i * a22r;
      R dn = dr * dr + di * di;
      if (dn < small * small) {
        dr = small;
        di = 0.0;
        dn = small * small;
      }
      // [u; w] = -inv(A) r,  inv(A) = [a22 -a12; -a21 a11] / det
      R ur = -(a22r * r1r - a22i * r1i - a12 * r2r);
      R ui = -(a22r * r1i + a22i * r1r - a12 * r2i);
      R wr_ = -(-a21 * r1r + a11r * r2r - a11i * r2i);
      R wi_ = -(-a21 * r1i + a11r * r2i + a11i * r2r);
      x[q - 1] = (ur * dr + ui * di) / dn;
      y[q - 1] = (ui * dr - ur * di) / dn;
      x[q] = (wr_ * dr + wi_ * di) / dn;
      y[q] = (wi_ * dr - wr_ * di) / dn;
      q -= 2;
    } else {
      R rr = 0, ri = 0;
      for (int c = q + 1; c <= last; ++c) {
        se_mac(rr, S[q * ld + c], x[c]);
        se_mac(ri, S[q * ld + c], y[c]);
      }
      rr = se_fin(rr);
      ri = se_fin(ri);
      R dr = S[q * ld + q] - lr, di = -li;
      R dn = dr * dr + di * di;
      if (dn < small * small) {
        dr = small;
        di = 0.0;
        dn = small * small;
      }
      x[q] = -(rr * dr + ri * di) / dn;
      y[q] = -(ri * dr - rr * di) / dn;
      q -= 1;
    }
    // rescale to avoid overflow: mx is the largest |x_c| + |y_c| over the entries computed so far
    for (int c = q + 1; c <= q + 2 && c <= last; ++c) {
      const R v = se_abs(x[c]) + se_abs(y[c]);
      if (v > mx) mx = v;
    }
    if (mx > R(SeEps<R>::big)) {
      const R inv = R(1.0) / mx;
      for (int c = 0; c <= last; ++c) {
        x[c] *= inv;
        y[c] *= inv;
      }
      mx = R(1.0);
    }
  }
}

// the bits of x: those of non-negative values are ordered like the values
SE_HD inline long long se_bits(double x) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(x);
#else
  long long u;
  memcpy(&u, &x, sizeof(u));
  return u;
#endif
}
// whether the non-negative values with these bits may be within 1e-14 of each other (96 ulp are 1.06e-14 at least)
// or are not ordered by their bits (a NaN)
SE_HD inline bool may_be_close(long long a, long long b) {
  const long long inf = 0x7ff0000000000000ll;
  return (a - b <= 96 && b - a <= 96) || a > inf || b > inf;
}

// Order of eigenvalues by decreasing modulus; within a pair the +imag member first.  Moduli that differ by
// 1e-14 or less count as equal and are taken as the selection below meets them, so that which of them comes
// first, and which one the cut at nev keeps, does not hang on their last bits.  perm: m ints; mod: m doubles of
// scratch (the moduli).  Where no moduli but those of a pair are that close, every rule gives the same order and each
// thread finds the rank of its eigenvalue; otherwise one thread selects.  The comparisons are of integers:
// an FP64 one holds GB300's FP64 pipe as long as a multiply-add of a whole warp.  Ends with a barrier.
SE_HD inline void order_by_modulus(const double* wr, const double* wi, int m, int* perm, double* mod,
                                   const Team& t = Team{0, 1}) {
  for (int j = t.lane; j < m; j += t.size) mod[j] = hypot(wr[j], wi[j]);
  t.sync();
  int close = 0;
  for (int j = t.lane; j < m; j += t.size) {
    int rank = 0;
    const long long mj = se_bits(mod[j]), rj = se_bits(wr[j]), ij = se_bits(wi[j]);
    for (int k = 0; k < m; ++k) {
      const long long mk = se_bits(mod[k]);
      rank += mk > mj ? 1 : 0;
      if (k != j && may_be_close(mk, mj)) {
        const long long ik = se_bits(wi[k]);
        if (se_bits(wr[k]) == rj && (ik ^ ij) < 0 && (ik << 1) == (ij << 1) && (ij << 1) != 0)
          rank += ij < 0 ? 1 : 0;   // the partner of its pair
        else
          close = 1;
      }
    }
    perm[rank] = j;
  }
  if (t.max(close)) {
    if (t.lane == 0) {
      for (int j = 0; j < m; ++j) perm[j] = j;
      for (int a = 0; a < m; ++a) {
        int best = a;
        double bm = mod[perm[a]];
        for (int b = a + 1; b < m; ++b) {
          const double mb = mod[perm[b]];
          if (may_be_close(se_bits(mb), se_bits(bm))
                  ? mb > bm * (1 + 1e-14) || (fabs(mb - bm) <= 1e-14 * bm && wi[perm[b]] > wi[perm[best]])
                  : se_bits(mb) > se_bits(bm)) {
            best = b;
            bm = mb;
          }
        }
        const int tmp = perm[a];
        perm[a] = perm[best];
        perm[best] = tmp;
      }
    }
  }
  t.sync();
}

}  // namespace se
}  // namespace a2ls
