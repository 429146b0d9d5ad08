// Double-float LU of one dense matrix by the library's batched kernel.  Arguments: n, tensor_cores, input file (n x n
// doubles, row-major), output file (the factors, likewise).
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../../paper_2201_02250_gb300/csrc/a2ls_internal.cuh"

using namespace a2ls;

template <class T> T* up(const std::vector<T>& v) {
  T* p = nullptr;
  cudaMalloc(&p, v.size() * sizeof(T));
  cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
  return p;
}

int main(int argc, char** argv) {
  if (argc < 5) return 1;
  const int n = std::atoi(argv[1]);
  std::vector<double> A((size_t)n * n);
  FILE* f = std::fopen(argv[3], "rb");
  if (!f || std::fread(A.data(), 8, A.size(), f) != A.size()) return 2;
  std::fclose(f);
  // a handle of one dense subdomain, for its layout
  std::vector<int> rp{0}, ci;
  std::vector<double> val;
  for (int r = 0; r < n; ++r) {
    for (int c = 0; c < n; ++c) ci.push_back(c), val.push_back(r == c ? n : 1.0);
    rp.push_back((int)ci.size());
  }
  a2ls_csr csr{n, n * n, up(rp), up(ci), up(val)};
  a2ls_options o;
  a2ls_default_options(&o);
  o.precision = A2LS_FP32;
  o.variant = A2LS_ONE_LEVEL_RAS;
  o.tensor_cores = std::atoi(argv[2]);
  a2ls_handle* h = nullptr;
  if (a2ls_setup(&csr, up(std::vector<int>(n, 0)), 0, 0, &o, &h) != A2LS_OK) {
    std::printf("%s\n", a2ls_last_error());
    return 3;
  }
  const int ld = h->h_ld[0];
  std::vector<dfloat> F(h->h_foff[1], dfloat(0.f, 0.f));
  for (int r = 0; r < n; ++r)
    for (int c = 0; c < n; ++c) F[(size_t)r * ld + c] = dfloat(A[(size_t)r * n + c]);
  dfloat* dF = up(F);
  double* scale = up(std::vector<double>(1, 1e-20));   // no pivot counts as tiny
  lu_batched<dfloat>(h, dF, 0, nullptr, scale);
  int st[ST_WORDS] = {-1};
  cudaMemcpy(st, h->d_status, sizeof(st), cudaMemcpyDeviceToHost);
  if (cudaMemcpy(F.data(), dF, F.size() * sizeof(dfloat), cudaMemcpyDeviceToHost) != cudaSuccess || st[ST_CODE] != 0) return 4;
  for (int r = 0; r < n; ++r)
    for (int c = 0; c < n; ++c) A[(size_t)r * n + c] = (double)F[(size_t)r * ld + c].hi + (double)F[(size_t)r * ld + c].lo;
  f = std::fopen(argv[4], "wb");
  std::fwrite(A.data(), 8, A.size(), f);
  std::fclose(f);
  return 0;
}
