// The device's double-float reciprocal square root, reciprocal and digit split against exact values.  Prints the
// largest errors: of rsqrt and recip relative to 2^-47, of the digits relative to 2^-56 of the scale, and how many
// digits are out of their range or not BF16 values.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "../../paper_2201_02250_gb300/csrc/a2ls_internal.cuh"
#include "../../paper_2201_02250_gb300/csrc/tc_dfloat.cuh"

using namespace a2ls;

__global__ void k_eval(int n, const dfloat* a, const dfloat* b, const dfloat* x, const int* e, dfloat* ra, dfloat* rb, float* d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  ra[i] = se_rsqrt(a[i]);
  rb[i] = se_recip12(b[i]);
  float t[tcdf::NDIG];
  tcdf::df_digits(x[i], e[i], t);
  for (int s = 0; s < tcdf::NDIG; ++s) d[i * tcdf::NDIG + s] = t[s];
}

template <class T> T* up(const std::vector<T>& v) {
  T* p = nullptr;
  cudaMalloc(&p, v.size() * sizeof(T));
  cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
  return p;
}
static double uniform() { return ((double)std::rand() + (double)std::rand() / RAND_MAX) / ((double)RAND_MAX + 1.0); }

int main() {
  const int n = 1 << 20;
  std::vector<dfloat> a, b, x;
  std::vector<int> e;
  for (int i = 0; i < n; ++i) {
    // rsqrt over the range of a scaled sum of three squares, 1 to 12, and far from it; reciprocal over [1, 2]
    a.push_back(dfloat(i & 1 ? 1.0 + 11.0 * uniform() : std::ldexp(1.0 + uniform(), std::rand() % 200 - 100)));
    b.push_back(dfloat(i < 2 ? 1.0 + i : 1.0 + uniform()));
    // digits: any size below the scale 2^e, the scale itself and zero among them
    const int ei = std::rand() % 200 - 100;
    double v = std::ldexp(2.0 * uniform() - 1.0, ei - std::rand() % 40);
    if (i % 1000 == 0) v = std::ldexp(i % 2000 ? 1.0 : -1.0, ei);
    if (i % 1000 == 1) v = 0.0;
    x.push_back(dfloat(v));
    e.push_back(ei);
  }
  dfloat *ra, *rb;
  float* d;
  cudaMalloc(&ra, n * sizeof(dfloat));
  cudaMalloc(&rb, n * sizeof(dfloat));
  cudaMalloc(&d, n * tcdf::NDIG * sizeof(float));
  k_eval<<<n / 256, 256>>>(n, up(a), up(b), up(x), up(e), ra, rb, d);
  std::vector<dfloat> hra(n), hrb(n);
  std::vector<float> hd(n * tcdf::NDIG);
  cudaMemcpy(hra.data(), ra, n * sizeof(dfloat), cudaMemcpyDeviceToHost);
  cudaMemcpy(hrb.data(), rb, n * sizeof(dfloat), cudaMemcpyDeviceToHost);
  if (cudaMemcpy(hd.data(), d, hd.size() * sizeof(float), cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  auto val = [](dfloat v) { return (long double)v.hi + (long double)v.lo; };
  double er = 0, eb = 0, ed = 0;
  int bad = 0;
  for (int i = 0; i < n; ++i) {
    // (1 + r)^2 - 1 = 2 r of a relative error r
    er = std::max(er, (double)std::fabs(val(hra[i]) * val(hra[i]) * val(a[i]) - 1) / 2 * std::ldexp(1.0, 47));
    eb = std::max(eb, (double)std::fabs(val(hrb[i]) * val(b[i]) - 1) * std::ldexp(1.0, 47));
    long double y = 0;
    for (int s = 0; s < tcdf::NDIG; ++s) {
      const float t = hd[i * tcdf::NDIG + s] * std::ldexp(1.f, 8 * s);   // the digit itself
      y += (long double)t * std::ldexp(1.0, -8 * (s + 1));
      unsigned bits;
      std::memcpy(&bits, &hd[i * tcdf::NDIG + s], 4);
      bad += t != std::rint(t) || std::fabs(t) > (s ? 128.f : 256.f) || (bits & 0xffffu) != 0;
    }
    ed = std::max(ed, (double)std::fabs(y - val(x[i]) * std::ldexp((long double)1, -e[i])) * std::ldexp(1.0, 56));
  }
  std::printf("%.6g %.6g %.6g %d\n", er, eb, ed, bad);
  return 0;
}
