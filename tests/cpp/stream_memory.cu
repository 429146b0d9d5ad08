// The copy of FP64 factors for the streaming solves: withheld where the vectors of GMRES would not fit beside it, made
// otherwise, given back by stream_release.  Prints "ok" or what failed.
#include <climits>
#include <cstdio>
#include <vector>

#include "../../paper_2201_02250_gb300/csrc/a2ls_internal.cuh"

using namespace a2ls;

#define REQUIRE(c) \
  if (!(c)) { std::printf("line %d: %s (%s)\n", __LINE__, #c, a2ls_last_error()); return 1; }

template <class T> T* up(const std::vector<T>& v) {
  T* p = nullptr;
  cudaMalloc(&p, v.size() * sizeof(T));
  cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
  return p;
}

int main() {
  const int n = 500;   // tridiagonal, two subdomains
  std::vector<int> rp{0}, ci, part;
  std::vector<double> val;
  for (int r = 0; r < n; ++r) {
    for (int c = r - 1; c <= r + 1; ++c)
      if (c >= 0 && c < n) ci.push_back(c), val.push_back(c == r ? 3.0 : -1.0);
    rp.push_back((int)ci.size());
    part.push_back(r >= n / 2);
  }
  a2ls_csr A{n, (int)ci.size(), up(rp), up(ci), up(val)};
  a2ls_options o;
  a2ls_default_options(&o);
  o.variant = A2LS_ONE_LEVEL_RAS;
  o.local_solve_kernel = 512;   // no copy by itself
  a2ls_handle* h = nullptr;
  REQUIRE(a2ls_setup(&A, up(part), 1, 0, &o, &h) == A2LS_OK);
  REQUIRE(!h->ss.d_stream && !h->ss.withheld);
  const size_t held = h->allocs.size();
  h->n = INT_MAX;   // 63 vectors of 2^31 doubles: a terabyte
  stream_prepare<double>(h, static_cast<const double*>(h->d_fac));
  h->n = n;
  REQUIRE(h->ss.withheld && !h->ss.d_stream && !h->ss.shape[0].ready && h->allocs.size() == held);
  h->ss = StreamSolve{};
  stream_prepare<double>(h, static_cast<const double*>(h->d_fac));
  REQUIRE(!h->ss.withheld && h->ss.d_stream && h->ss.shape[0].ready && h->allocs.size() > held);
  stream_release(h);
  REQUIRE(!h->ss.d_stream && !h->ss.shape[0].ready && h->allocs.size() == held);
  a2ls_destroy(h);
  std::printf("ok\n");
  return 0;
}
