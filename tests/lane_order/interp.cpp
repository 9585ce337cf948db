// The lane-group extended+i kernels (interp_group.cuh) lane by lane: no data race, and
// the same rows of P from 16 and from 32 lanes per row.
#include <cstdio>
#include <random>

#include "warp.h"

enum { IF_S = 1, IF_SAME = 2, IF_C = 4, IF_DIAG = 8, IF_NEG = 16 };
alignas(16) unsigned char ix_sm[1 << 17];
#include "interp_group.cuh"

struct Rows {
  std::vector<int32_t> cnt, col;
  std::vector<double> val;
  int left;
};
static const int n = 60, pmax = 4;
static std::vector<int32_t> rp{0}, ci, cidx(n);
static std::vector<double> v;
static std::vector<uint8_t> ef;

template <class K>
static Rows run(K kernel, int rows_per_block) {
  Rows R;
  R.cnt.assign(n, -7);
  R.col.assign(n * pmax, -1);
  R.val.assign(n * pmax, 0.0);
  std::vector<int32_t> rows((kIxClasses + 1) * n);
  int ncls[kIxClasses + 1] = {};
  for (int i = 0; i < n; ++i)
    if (i % 3) rows[ncls[0]++] = i;
  IxArgs a{n, pmax, rp.data(), ci.data(), v.data(), ef.data(), cidx.data(), R.cnt.data(),
           R.col.data(), R.val.data(), rows.data(), ncls};
  gridDim.x = 1;
  for (int w = 0; w < 2; ++w) run_warp(w, [=] { kernel(a, 0, 0); });
  R.left = ncls[1];
  return R;
}

int main() {
  std::mt19937 g(5);
  for (int i = 0; i < n; ++i) cidx[i] = i / 3;  // every third point is a C point
  for (int i = 0; i < n; ++i) {
    for (int d = -6; d <= 6; ++d) {
      const int j = i + d * (d % 2 ? 1 : 3);
      if (j < 0 || j >= n || (d && g() % 4 == 0)) continue;
      ci.push_back(j);
    }
    std::sort(ci.begin() + rp[i], ci.end());
    ci.erase(std::unique(ci.begin() + rp[i], ci.end()), ci.end());
    for (size_t t = rp[i]; t < ci.size(); ++t) {
      const int j = ci[t];
      v.push_back(j == i ? 9.0 : std::uniform_real_distribution<double>(-1, 0.2)(g));
      ef.push_back((j != i && v.back() < -0.2 ? IF_S : 0) | (j % 2 == i % 2 || g() % 2 ? IF_SAME : 0) |
                   (j % 3 == 0 ? IF_C : 0) | (j == i ? IF_DIAG | IF_SAME : 0));
    }
    rp.push_back((int32_t)ci.size());
  }
  const Rows a = run(k_interp_group<16, 64, 40, 96, 16, 2>, 4);
  const Rows b = run(k_interp_group<32, 128, 64, 256, 40, 2>, 2);
  int bad = a.left + b.left, terms = 0;
  for (int i = 0; i < n; ++i) {
    bad += a.cnt[i] != b.cnt[i];
    terms += max(0, a.cnt[i]);
    for (int p = 0; p < a.cnt[i] && p < pmax; ++p)
      bad += a.col[i * pmax + p] != b.col[i * pmax + p] ||
             bits_of(a.val[i * pmax + p]) != bits_of(b.val[i * pmax + p]);
  }
  std::printf("%d terms, %d differences, %d and %d rows left\n", terms, bad, a.left, b.left);
  return bad != 0 || terms < n;
}
