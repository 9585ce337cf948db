// The ILU(0) factorisation of two rows per warp lane by lane: no data race, and the
// factors of the sequential definition (largest relative difference in the output;
// with "bits": the same bits).  ilu_pair.inc holds the kernel, cut from setup_ilu.cu.
#include <cmath>
#include <cstdio>
#include <random>

#include "warp.h"

#define CPTR_SPIN_LIMIT 1000u
enum { DEV_OK = 0, DEV_TIMEOUT = 1, DEV_BREAKDOWN = 2 };
struct Ctl {
  int status;
  unsigned fac_ctr;
};
inline void dev_fail(int* status, int code) { atomicCAS(status, DEV_OK, code); }
alignas(16) unsigned char fsm[1 << 16];
#include "ilu_pair.inc"

static void mul4(const double* a, const double* b, double* o) {
  for (int r = 0; r < 4; ++r)
    for (int c = 0; c < 4; ++c) {
      double s = 0.0;
      for (int q = 0; q < 4; ++q) s += a[4 * r + q] * b[4 * q + c];
      o[4 * r + c] = s;
    }
}
static bool inverse(const double* M, double* out) {
  double a[4][8];
  for (int r = 0; r < 4; ++r)
    for (int c = 0; c < 8; ++c) a[r][c] = c < 4 ? M[4 * r + c] : c - 4 == r;
  for (int k = 0; k < 4; ++k) {
    int p = k;
    for (int r = k + 1; r < 4; ++r)
      if (std::fabs(a[r][k]) > std::fabs(a[p][k])) p = r;
    if (!(std::fabs(a[p][k]) > 0.0)) return false;
    std::swap_ranges(a[k], a[k] + 8, a[p]);
    const double d = a[k][k];
    for (int c = 0; c < 8; ++c) a[k][c] /= d;
    for (int r = 0; r < 4; ++r) {
      const double f = a[r][k];
      for (int c = 0; c < 8 && r != k; ++c) a[r][c] -= f * a[k][c];
    }
  }
  for (int r = 0; r < 4; ++r)
    for (int c = 0; c < 4; ++c) out[4 * r + c] = a[r][4 + c];
  return true;
}

// Cells 0..n-1: `dense` groups in turn, group g with a dense pattern of size[g] cells
// (32 shared columns times the row's length do not fit a row's list from ten cells on),
// whose rows of equal rank share a level: long and short rows meet in one warp.
int main(int argc, char** argv) {
  const int size[] = {1, 2, 5, 12, 16, 3};
  std::vector<int> first;
  int n = 0, levels = 0, maxrow = 0;
  for (int s : size) {
    first.push_back(n);
    n += s;
    levels = max(levels, s);
    maxrow = max(maxrow, s);
  }
  std::mt19937 gen(3);
  std::vector<int32_t> rp{0}, ci, diag, ord;
  std::vector<double> A;
  for (size_t g = 0; g < first.size(); ++g)
    for (int i = 0; i < size[g]; ++i) {
      for (int j = 0; j < size[g]; ++j) {
        if (j == i) diag.push_back((int32_t)ci.size());
        ci.push_back(first[g] + j);
        for (int q = 0; q < 16; ++q)
          A.push_back(std::uniform_real_distribution<double>(-1, 1)(gen) +
                      (j == i && q % 5 == 0 ? 3.0 + size[g] : 0.0));
      }
      rp.push_back((int32_t)ci.size());
    }
  for (int l = 0; l < levels; ++l) {  // a level's rows, padded to eight positions
    for (size_t g = 0; g < first.size(); ++g)
      if (l < size[g]) ord.push_back(first[g] + l);
    while (ord.size() % 8) ord.push_back(-1);
  }
  std::vector<double> ref = A;
  double t[16];
  for (int i = 0; i < n; ++i) {
    for (int e = rp[i]; e < diag[i]; ++e) {
      const int k = ci[e];
      mul4(&ref[16 * e], &ref[16 * diag[k]], t);
      std::copy(t, t + 16, &ref[16 * e]);
      for (int f = e + 1; f < rp[i + 1]; ++f)
        for (int u = diag[k] + 1; u < rp[k + 1]; ++u)
          if (ci[u] == ci[f]) {
            mul4(&ref[16 * e], &ref[16 * u], t);
            for (int q = 0; q < 16; ++q) ref[16 * f + q] -= t[q];
          }
    }
    if (!inverse(&ref[16 * diag[i]], t)) return 3;
    std::copy(t, t + 16, &ref[16 * diag[i]]);
  }
  std::vector<int> done(n, 0);
  Ctl ctl{};
  Ctl* pc = &ctl;
  const FacRow lay = fac_row(maxrow);
  double* LU = A.data();
  int* pd = done.data();
  const int npos = (int)ord.size();
  const int32_t *po = ord.data(), *prp = rp.data(), *pci = ci.data(), *pdg = diag.data();
  run_warp(0, [=] { k_ilu_factor_pair(npos, lay, po, prp, pci, pdg, LU, pd, 1, pc); });
  double worst = 0.0;
  int bits = 0;
  for (size_t q = 0; q < A.size(); ++q) {
    worst = max(worst, std::fabs(A[q] - ref[q]) / (std::fabs(ref[q]) + 1e-3));
    bits += A[q] != ref[q];
  }
  std::printf("status %d, largest relative difference %.2e, %d of %d entries differ\n",
              ctl.status, worst, bits, (int)A.size());
  return ctl.status != DEV_OK || !(worst < 1e-10) || (argc > 1 && bits != 0);
}
