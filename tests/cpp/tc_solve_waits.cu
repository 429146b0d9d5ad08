// Sweeps of the tensor-core triangular solves whose waits run out: every one ends, reports A2LS_ERR_TIMEOUT if
// any wait gave up, and leaves the device as it was.  Prints "ok" or what failed.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "../../paper_2201_02250_gb300/csrc/a2ls_internal.cuh"

using namespace a2ls;

#define REQUIRE(c) \
  if (!(c)) { std::printf("line %d: %s (%s) limit %ld\n", __LINE__, #c, cudaGetErrorString(cudaGetLastError()), limit); return 1; }

template <class T> T* up(const std::vector<T>& v) {
  T* p = nullptr;
  cudaMalloc(&p, v.size() * sizeof(T));
  cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
  return p;
}

int main() {
  long limit = -1;
  // a five-point operator on 56 x 56 nodes in 2 x 2 blocks: subdomains of about 800 rows, 13 block rows each
  const int m = 56, n = m * m;
  std::vector<int> rp{0}, ci, part;
  std::vector<double> val;
  for (int r = 0; r < n; ++r) {
    const int x = r / m, y = r % m, nb[5] = {r - m, r - 1, r, r + 1, r + m};
    const bool in[5] = {x > 0, y > 0, true, y < m - 1, x < m - 1};
    for (int k = 0; k < 5; ++k)
      if (in[k]) ci.push_back(nb[k]), val.push_back(k == 2 ? 4.0 : -1.0);
    rp.push_back((int)ci.size());
    part.push_back((x >= m / 2) * 2 + (y >= m / 2));
  }
  a2ls_csr A{n, (int)ci.size(), up(rp), up(ci), up(val)};
  a2ls_options o;
  a2ls_default_options(&o);
  o.precision = A2LS_FP32;
  a2ls_handle* h = nullptr;
  REQUIRE(a2ls_setup(&A, up(part), 1, 2, &o, &h) == A2LS_OK);
  // small random factors in its layout, and right-hand sides of p columns
  std::srand(7);
  std::vector<dfloat> fac(h->h_foff[h->N]), X0;
  for (auto& f : fac) f = dfloat(0.01f * (std::rand() % 2001 - 1000) / 1000.f, 0.f);
  const int p = 20, ldx = 32;
  std::vector<int64_t> xo{0};
  for (int i = 0; i < h->N; ++i) xo.push_back(xo[i] + (int64_t)h->h_n[i] * ldx);
  for (int64_t e = 0; e < xo[h->N]; ++e) X0.push_back(dfloat((std::rand() % 2001 - 1000) / 1000.f, 0.f));
  dfloat *df = up(fac), *X = up(X0);
  const int64_t* dxo = up(xo);
  const int* dp = up(std::vector<int>(h->N, p));
  TcSolve ts;
  tc_solve_prepare(h, df, ts);
  std::vector<dfloat> want[2], got(X0.size());
  int gave_up = 0;
  auto sweep = [&](int fwd, long lim) {   // the status code; X in got
    cudaMemcpy(X, X0.data(), X0.size() * sizeof(dfloat), cudaMemcpyHostToDevice);
    cudaMemset(h->d_status, 0, sizeof(int) * ST_WORDS);
    tc_block_solve(h, ts, X, dxo, 0, ldx, dp, nullptr, fwd, nullptr, lim);
    int st[ST_WORDS] = {-1};
    cudaMemcpy(got.data(), X, X0.size() * sizeof(dfloat), cudaMemcpyDeviceToHost);
    cudaMemcpy(st, h->d_status, sizeof(st), cudaMemcpyDeviceToHost);
    return st[ST_CODE];
  };
  auto same = [&](const std::vector<dfloat>& w) {
    for (size_t e = 0; e < w.size(); ++e)
      if (w[e].hi != got[e].hi || w[e].lo != got[e].lo) return false;
    return true;
  };
  for (int fwd = 0; fwd < 2; ++fwd) {
    REQUIRE(sweep(fwd, 1L << 26) == 0);
    want[fwd] = got;
  }
  for (limit = 0; limit < 300; limit += 1 + limit / 8)
    for (int fwd = 0; fwd < 2; ++fwd) {
      const int code = sweep(fwd, limit);
      REQUIRE(cudaGetLastError() == cudaSuccess);
      REQUIRE(code == A2LS_ERR_TIMEOUT || (code == A2LS_OK && limit > 0 && same(want[fwd])));
      gave_up += code == A2LS_ERR_TIMEOUT;
    }
  for (int fwd = 0; fwd < 2; ++fwd) REQUIRE(sweep(fwd, 1L << 26) == 0 && same(want[fwd]));
  std::printf("ok, %d gave up\n", gave_up);
  return 0;
}
