// The double-float form of the small dense eigensolver (small_eig.cuh on dfloat.cuh) as a one-thread team on the host:
// the device's explicitly rounded operations are the host's, and its approximations 1 / sqrt and the fast
// quotient are off by up to two units in the last place.  Compile with -ffp-contract=off.  Reads "m" and an m x m
// matrix, prints the return code, the largest entry of |Q^T Q - I|, of |Q S Q^T - H|, and S's diagonal blocks'
// eigenvalues.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#define __CUDACC__   // (cuda_runtime.h is an empty file: what is wanted of it follows)
#define __host__
#define __device__
#define __forceinline__ inline
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmul_rn(float a, float b) { return a * b; }
static float __fdiv_rn(float a, float b) { return a / b; }
static float __fsqrt_rn(float a) { return std::sqrt(a); }
static float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static unsigned __float_as_uint(float a) { unsigned u; std::memcpy(&u, &a, 4); return u; }
static float __uint_as_float(unsigned u) { float a; std::memcpy(&a, &u, 4); return a; }
static float off_by_ulps(float v) {
  int k = std::rand() % 5 - 2;
  for (; k > 0; --k) v = std::nextafter(v, INFINITY);
  for (; k < 0; ++k) v = std::nextafter(v, 0.f);
  return v;
}
static float rsqrtf(float a) { return off_by_ulps((float)(1.0 / std::sqrt((double)a))); }
static float __fdividef(float a, float b) { return off_by_ulps(a / b); }
// a warp of one lane: nothing to add or to compare with
template <class T> static T __shfl_xor_sync(unsigned, T, int) { return T(0); }
template <class T> static T __shfl_sync(unsigned, T v, int) { return v; }
using std::fmaxf;

#include "../../paper_2201_02250_gb300/csrc/dfloat.cuh"
#include "../../paper_2201_02250_gb300/csrc/small_eig.cuh"

namespace a2ls {
namespace se {   // as in k_eig.cu
template <> struct SeEps<dfloat> {
  static constexpr double v = 1.4210854715202004e-14;
  static constexpr double big = 1e30;
};
template <> struct SeFast<dfloat> { static constexpr bool v = true; };
}  // namespace se
}  // namespace a2ls
using a2ls::dfloat;
using namespace a2ls::se;

int main() {
  int m;
  if (std::scanf("%d", &m) != 1) return 1;
  std::srand(1);
  const int ld = m + 1;
  std::vector<dfloat> H(m * ld), Q(m * ld, dfloat(0.f)), v(m);
  std::vector<double> H0(m * m), wr(m), wi(m);
  double hn = 0.0;
  for (int r = 0; r < m; ++r)
    for (int c = 0; c < m; ++c) {
      double x;
      if (std::scanf("%lf", &x) != 1) return 1;
      H[r * ld + c] = dfloat(x);
      H0[r * m + c] = (double)H[r * ld + c];
      hn = std::max(hn, std::fabs(x));
    }
  for (int r = 0; r < m; ++r) Q[r * ld + r] = dfloat(1.f);
  const Team t{0, 1};
  hessenberg(H.data(), ld, Q.data(), ld, m, v.data(), t);
  for (int r = 0; r < m; ++r)   // (below the subdiagonal exactly zero)
    for (int c = 0; c + 1 < r; ++c)
      if ((double)H[r * ld + c] != 0.0) return 2;
  const int rc = schur(H.data(), ld, Q.data(), ld, m, hn, t);
  for (int j = 0; j + 2 < m; ++j)   // quasi-triangular: no two blocks touch
    if ((double)H[(j + 1) * ld + j] != 0.0 && (double)H[(j + 2) * ld + j + 1] != 0.0 && rc == 0) return 3;
  schur_eigenvalues(H.data(), ld, m, wr.data(), wi.data());
  std::vector<long double> QS(m * m);
  double orth = 0.0, back = 0.0;
  for (int r = 0; r < m; ++r)
    for (int c = 0; c < m; ++c) {
      long double s = 0, q = 0;
      for (int k = 0; k < m; ++k) {
        q += (long double)(double)Q[k * ld + r] * (double)Q[k * ld + c];
        if (k <= c + 1) s += (long double)(double)Q[r * ld + k] * (double)H[k * ld + c];
      }
      QS[r * m + c] = s;
      orth = std::max(orth, (double)std::fabs(q - (r == c)));
    }
  for (int r = 0; r < m; ++r)
    for (int c = 0; c < m; ++c) {
      long double s = 0;
      for (int k = 0; k < m; ++k) s += QS[r * m + k] * (double)Q[c * ld + k];
      back = std::max(back, (double)std::fabs(s - H0[r * m + c]));
    }
  std::printf("%d %.17g %.17g %.17g\n", rc, orth, back, hn);
  for (int j = 0; j < m; ++j) std::printf("%.17g %.17g\n", wr[j], wi[j]);
  return 0;
}
