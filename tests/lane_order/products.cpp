// The sparse products' row accumulators (spgemm_acc.cuh) lane by lane: no data race
// under the programming model, and the sums of the sequential definition bit for bit.
#include <cstdio>
#include <map>
#include <random>

#include "warp.h"

alignas(16) unsigned char acc_sm[1 << 17];
#include "spgemm_acc.cuh"

struct Csr {
  std::vector<int32_t> rp{0}, ci;
  std::vector<double> v;
};

static Csr random_csr(int n, int m, int lo, int hi, unsigned seed) {
  std::mt19937 g(seed);
  Csr A;
  for (int i = 0; i < n; ++i) {
    std::vector<int> c(m);
    for (int j = 0; j < m; ++j) c[j] = j;
    std::shuffle(c.begin(), c.end(), g);
    c.resize(std::uniform_int_distribution<int>(lo, hi)(g));
    std::sort(c.begin(), c.end());
    for (int j : c) {
      A.ci.push_back(j);
      A.v.push_back(std::uniform_real_distribution<double>(-1, 1)(g));
    }
    A.rp.push_back((int32_t)A.ci.size());
  }
  return A;
}

// rows of 0 to `alen` entries times rows of 0 to `blen` among m columns
template <class K>
static int check(const char* name, K kernel, int rows_per_warp, int alen, int blen, int m) {
  const int n = 4 * rows_per_warp, nb = 40;  // the four warps of a block
  const Csr A = random_csr(n, nb, 0, alen, 7), B = random_csr(nb, m, 0, blen, 8);
  std::vector<long long> toff(n + 1, 0);
  std::vector<std::map<int, double>> ref(n);
  for (int i = 0; i < n; ++i) {
    long long p = 0;
    for (int t = A.rp[i]; t < A.rp[i + 1]; ++t)
      for (int u = B.rp[A.ci[t]]; u < B.rp[A.ci[t] + 1]; ++u, ++p) {
        const double prod = A.v[t] * B.v[u];
        ref[i][B.ci[u]] += prod;
      }
    toff[i + 1] = toff[i] + p;
  }
  std::vector<int32_t> cci(toff[n] + 1), cnt(n, -7), rows((kAccClasses + 1) * n);
  std::vector<double> cv(toff[n] + 1);
  int ncls[kAccClasses + 1] = {};
  AccArgs a{n,           A.rp.data(), A.ci.data(), A.v.data(), B.rp.data(),
            B.ci.data(), B.v.data(),  toff.data(), cci.data(), cv.data(),
            cnt.data(),  rows.data(), ncls,        0};
  gridDim.x = 1;
  for (int w = 0; w < kAccThreads / 32; ++w) run_warp(w, [=] { kernel(a, 0, 0); });
  int bad = 0;
  for (int i = 0; i < n; ++i) {
    bad += cnt[i] != (int)ref[i].size();
    long long o = toff[i];
    for (auto& e : ref[i]) {
      bad += cci[o] != e.first || bits_of(cv[o]) != bits_of(e.second);
      ++o;
    }
  }
  if (bad) std::printf("%s: %d differences\n", name, bad);
  return bad;
}

int main() {
  int bad = 0;
  // several steps of 32 products with columns that come back in later steps
  bad += check("flat", k_acc_flat<128>, 1, 20, 12, 60);
  // every step spans many rows of B: equal columns inside a step
  bad += check("flat, short rows", k_acc_flat<64>, 1, 36, 3, 20);
  bad += check("group", k_acc_group<4, 64>, 8, 12, 6, 30);
  return bad != 0;
}
