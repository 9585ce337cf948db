// Batched solves of many small systems at once.
//
// A small system (thousands of cells) leaves most of the GPU idle in the
// per-system path, whose Krylov loop launches a few dozen kernels per
// iteration and reads a host flag at every restart.  Here one thread block, or a
// cluster of up to eight, runs the whole flexible GMRES(m) loop of one system on
// the device, with the Eq. 3 preconditioner (Quasi-IMPES restriction, the
// system-AMG V-cycle, the correction, the ILU(0) solves, the combination), the
// outer block SpMV, CGS2 with Givens rotations, the back substitution, restarts
// and the true residual, with no host in between; a grid of them advances every
// system of the batch at once.  Each system reads its own
// context's hierarchy, factors and work vectors (built by cptr_setup), and
// every sum has a fixed order that does not depend on the batch: a system's
// result is the same alone and in any batch.
#include <algorithm>
#include <chrono>
#include <string>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "ctx.h"

namespace {

constexpr int kBT = 512;        // threads per block
constexpr int kBMaxLev = 25;    // AMG levels
constexpr int kBMaxM = 32;      // restart length

struct BLevel {
  int n;
  const int32_t *Arp, *Aci;
  const void* Av;    // apply precision
  const void* dinv;  // apply precision
  int nc;            // rows of the next level (R: nc x n, P: n x nc)
  const int32_t *Rrp, *Rci;
  const void* Rv;
  const int32_t *Prp, *Pci;
  const void* Pv;
  void *b, *x, *r, *x2, *t;
};

struct alignas(16) BSys {
  int N, m, maxit, nlev, ne, e0, e1, h0, h1, h2, nu_pre, nu_post, nlf, nlb, first;
  double tol;
  const int32_t *rp, *ci;
  const double* v;    // the FP64 operator
  const void* Wt;     // decoupling weights (apply precision)
  const void* AE;     // elliptic columns of A (apply precision)
  const double* Cinv; // dense inverse of the coarsest operator
  void *rhat, *zc, *r2, *u, *y2;
  const int32_t *offf, *ordf, *Lrp, *Lci;
  const void* Lv;
  const int32_t *offb, *ordb, *Urp, *Uci;
  const void *Uv, *Dinv;
  double *V, *w, *x, *b;
  void* Z;
  unsigned spin;  // reads a dependency wait makes before it gives up
  int* fail;      // set when one did
  BLevel lev[kBMaxLev];
};

struct BOut {
  int iters, status, fail;
  double rel_resid;
};

// A system runs on one block (Solo) or on a cluster of 2, 4 or 8 (Team; see
// cptr_solve_batch): every loop over rows is dealt over its threads, and a phase ends at
// its barrier, which also makes the blocks' writes to global memory visible.
// A row's sum never depends on the dealing, and the dots and norms are cut into
// kParts slices of the rows whatever the number of blocks, so the result is the
// same on any cluster size.
//
// One block is bound by its SM's FP64 rate (outer SpMV, CGS2) and by memory
// latency (V-cycle rows, ILU(0) levels); the cluster divides the first by its size.
// The kernel is compiled for one block apart, in line throughout and with constant
// strides: the clusters' code on one block took 30.5 instead of 21.7 ms for 152 grids of
// 8,000 cells (mixed; 39.0 and 28.2 FP64), 6.6 instead of 5.0 for 48 of 1,859, 4.9
// instead of 3.7 for one cloud of 507.  For a cluster every phase is a call: in line, the
// polling loop of the ILU(0) solves loses 2-8% to the code around it (24 grids of 30k
// cells on four blocks 29.2 instead of 27.5 ms).
struct Solo {
  static constexpr int rank = 0, size = 1, threads = kBT;
  int tid = (int)threadIdx.x;
  __device__ __forceinline__ void sync() const { __syncthreads(); }
};
struct Team {
  int rank, size;  // block of the cluster, blocks in it
  int tid, threads;
  __device__ __forceinline__ Team() {
    unsigned r, n;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
    rank = (int)r;
    size = (int)n;
    tid = rank * kBT + (int)threadIdx.x;
    threads = size * kBT;
  }
  __device__ __forceinline__ void sync() const {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
                 "barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
};
// Phase<f>::run(t, ...): f in line on one block, a call on a cluster.
template <auto F>
struct Phase;
template <class TM, class... A, void (*F)(const TM&, A...)>
struct Phase<F> {
  static __device__ __noinline__ void call(const TM& t, A... a) { F(t, a...); }
  static __device__ __forceinline__ void run(const TM& t, A... a) {
    if constexpr (std::is_same_v<TM, Solo>) F(t, a...);
    else call(t, a...);
  }
};
// A double of another block's shared memory.
__device__ __forceinline__ double team_read(const Solo&, const double* own, int) { return *own; }
__device__ __forceinline__ double team_read(const Team&, const double* own, int rank) {
  unsigned a = (unsigned)__cvta_generic_to_shared(own), r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(r) : "memory");
  return v;
}

constexpr int kParts = 32;
// Partial sums of a reduction, this block's slices; two of them alternate, so that
// a block may start the next reduction while another still reads this one.
struct Partials {
  double v[2][kParts * (kBMaxM + 1)];
  int flip;
};

// out[l] = V_l . w for l < nc (V_l = V + l n), the same in every block: a warp sums
// G columns over one slice, the slices are combined by a shuffle tree.  The slices are
// short (kParts of them whatever the blocks), so the columns share the tree of warp_sum:
// its first two steps halve the columns a lane holds, with the same pairs of lanes added
// for every column, in 6 additions for four columns instead of 20.
template <int G>
__device__ __forceinline__ void part_dot(const double* V, size_t n, const double* w, int lo,
                                         int hi, double* out) {
  const int lane = threadIdx.x & 31;
  double acc[G];
#pragma unroll
  for (int u = 0; u < G; ++u) acc[u] = 0.0;
#pragma unroll 4
  for (int i = lo + lane; i < hi; i += 32) {
    const double wi = w[i];
#pragma unroll
    for (int u = 0; u < G; ++u) acc[u] += V[(size_t)u * n + i] * wi;
  }
  // lanes with the bit of step o clear keep the even columns
  auto halve = [&](double a, double b, int o) {
    const bool high = lane & o;
    return (high ? b : a) + __shfl_xor_sync(0xffffffffu, high ? a : b, o);
  };
  double s;
  if (G == 1) s = acc[0] + __shfl_xor_sync(0xffffffffu, acc[0], 16);
  else s = halve(acc[0], acc[G > 1 ? 1 : 0], 16);
  if (G <= 2) s += __shfl_xor_sync(0xffffffffu, s, 8);
  else s = halve(s, halve(acc[G > 2 ? 2 : 0], G > 3 ? acc[G > 3 ? 3 : 0] : 0.0, 16), 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  const int u = (lane >> 4 & 1) + (G > 2 ? 2 * (lane >> 3 & 1) : 0);
  if ((lane & 7) == 0 && u < G && (G > 2 || (lane & 8) == 0)) out[u] = s;
}
template <class TM>
__device__ __forceinline__ void team_dots(const TM& t, Partials& P, const double* V,
                                          const double* w, int n, int nc, double* out) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = kBT / 32;
  const int mine = kParts / t.size;
  const int per = ((n + kParts - 1) / kParts + 31) & ~31;
  const int groups = (nc + 3) / 4;
  double* part = P.v[P.flip];
  for (int unit = warp; unit < mine * groups; unit += nw) {
    const int p = unit / groups, g = unit % groups;
    const int lo = min(n, (t.rank * mine + p) * per), hi = min(n, lo + per);
    double* o = part + p * (kBMaxM + 1) + 4 * g;
    const double* Vg = V + (size_t)(4 * g) * n;
    switch (min(4, nc - 4 * g)) {
      case 1: part_dot<1>(Vg, n, w, lo, hi, o); break;
      case 2: part_dot<2>(Vg, n, w, lo, hi, o); break;
      case 3: part_dot<3>(Vg, n, w, lo, hi, o); break;
      default: part_dot<4>(Vg, n, w, lo, hi, o); break;
    }
  }
  t.sync();
  for (int l = warp; l < nc; l += nw) {
    const double s = warp_sum(team_read(t, part + (lane % mine) * (kBMaxM + 1) + l, lane / mine));
    if (lane == 0) out[l] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) P.flip ^= 1;
  __syncthreads();
}

// w -= V h over the first nc columns, four elements per thread at a time (their
// loads overlap; each element takes its columns in order).
template <class TM>
__device__ __forceinline__ void team_update(const TM& t, const double* V, double* w, int n, int nc,
                                            const double* h) {
  for (int i0 = t.tid; i0 < n; i0 += 4 * t.threads) {
    double wi[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) wi[u] = i0 + u * t.threads < n ? w[i0 + u * t.threads] : 0.0;
    const double* v = V + i0;
#pragma unroll 2
    for (int l = 0; l < nc; ++l, v += n) {
      const double hl = h[l];
      double x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = i0 + u * t.threads < n ? v[u * t.threads] : 0.0;
#pragma unroll
      for (int u = 0; u < 4; ++u) wi[u] -= hl * x[u];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (i0 + u * t.threads < n) w[i0 + u * t.threads] = wi[u];
  }
}

// The row loops below load several entries before summing their products (in
// entry order, the same sums as an entry-by-entry loop).

__device__ __forceinline__ void ld4x(const double* p, double* o) {
  const double2 a = *reinterpret_cast<const double2*>(p);
  const double2 b = *(reinterpret_cast<const double2*>(p) + 1);
  o[0] = a.x; o[1] = a.y; o[2] = b.x; o[3] = b.y;
}
__device__ __forceinline__ void ld4x(const float* p, float* o) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  o[0] = a.x; o[1] = a.y; o[2] = a.z; o[3] = a.w;
}
__device__ __forceinline__ void ld4x(const float* p, double* o) {  // (off the FP64 pipe)
  float f[4];
  ld4x(p, f);
  widen<4>(f, o);
}

// y = A x (4x4 blocks, FP64 accumulation in block order), y = b - A x when b
template <class TM, class TX>
__device__ __forceinline__ void bspmv(const TM& t, const BSys& S, const TX* x, const double* b,
                                      double* y) {
  const int n4 = 4 * S.N;
  const int32_t* __restrict__ rp = S.rp;
  const int32_t* __restrict__ ci = S.ci;
  const double* __restrict__ v = S.v;
  for (int g = t.tid; g < n4; g += t.threads) {
    const int i = g >> 2, r = g & 3;
    double acc = 0.0;
    int k = rp[i];
    const int k1 = rp[i + 1];
    for (; k + 4 <= k1; k += 4) {
      int j[4];
      double a[4][4], xv[4][4];
#pragma unroll
      for (int u = 0; u < 4; ++u) j[u] = ci[k + u];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        ld4(v + 16 * (size_t)(k + u) + 4 * r, a[u]);
        ld4x(x + 4 * (size_t)j[u], xv[u]);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc = fma(a[u][q], xv[u][q], acc);
    }
    for (; k < k1; ++k) {
      double a[4], xv[4];
      ld4(v + 16 * (size_t)k + 4 * r, a);
      ld4x(x + 4 * (size_t)ci[k], xv);
#pragma unroll
      for (int q = 0; q < 4; ++q) acc = fma(a[q], xv[q], acc);
    }
    y[g] = b ? b[g] - acc : acc;
  }
}

// f(i, sum) for every row i < n of a CSR operator, sum = its val * x in entry order
// (a thread per row; four entries are loaded before their products are added.  Eight
// at a time, predicated, took 62 million clocks against 49 in the V-cycles of a
// 24.6k-cell cloud on one block; the last one to three are read together.)
template <class TM, class T, class F>
__device__ __forceinline__ void rows(const TM& t, int n, const int32_t* __restrict__ rp,
                                     const int32_t* __restrict__ ci, const T* __restrict__ val,
                                     const T* x, F f) {
  for (int i = t.tid; i < n; i += t.threads) {
    T s = 0;
    int k = rp[i];
    const int t1 = rp[i + 1];
    for (; k + 4 <= t1; k += 4) {
      int j[4];
      T a[4], xv[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        j[u] = ci[k + u];
        a[u] = val[k + u];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) xv[u] = x[j[u]];
#pragma unroll
      for (int u = 0; u < 4; ++u) s += a[u] * xv[u];
    }
    if (k < t1) {
      int j[3];
      T a[3], xv[3];
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        const int e = min(k + u, t1 - 1);
        j[u] = ci[e];
        a[u] = val[e];
      }
#pragma unroll
      for (int u = 0; u < 3; ++u) xv[u] = x[j[u]];
      s += a[0] * xv[0];
      if (k + 1 < t1) s += a[1] * xv[1];
      if (k + 2 < t1) s += a[2] * xv[2];
    }
    f(i, s);
  }
}

// r = b - A x on one AMG level (scalar CSR, apply precision)
template <class TM, class T>
__device__ __forceinline__ void lresid(const TM& t, const BLevel& L, const T* b, const T* x, T* r) {
  rows(t, L.n, L.Arp, L.Aci, (const T*)L.Av, x, [=](int i, T s) { r[i] = b[i] - s; });
}

// xout = xin + D_l1^-1 (b - A xin): one l1-Jacobi sweep
template <class TM, class T>
__device__ __forceinline__ void lsweep(const TM& t, const BLevel& L, const T* b, const T* xin, T* xout) {
  const T* dv = (const T*)L.dinv;
  rows(t, L.n, L.Arp, L.Aci, (const T*)L.Av, xin,
          [=](int i, T s) { xout[i] = xin[i] + dv[i] * (b[i] - s); });
}

// b_{l+1} = R r and x += P xc
template <class TM, class T>
__device__ __forceinline__ void lrestrict(const TM& t, const BLevel& L, const T* r, T* bn) {
  const int32_t *rp = L.Rrp, *ci = L.Rci;
  const T* rv = (const T*)L.Rv;
  rows(t, L.nc, rp, ci, rv, r, [=](int i, T s) { bn[i] = s; });
}
template <class TM, class T>
__device__ __forceinline__ void lprolong(const TM& t, const BLevel& L, const T* xc, T* x) {
  rows(t, L.n, L.Prp, L.Pci, (const T*)L.Pv, xc, [=](int i, T s) { x[i] += s; });
}

// One V(nu_pre, nu_post) cycle with l1-Jacobi from a zero guess on the
// system's hierarchy: b0 (level 0 right-hand side) -> zc.
template <class TM, class T>
__device__ __forceinline__ void bvcycle(const TM& t, const BSys& S, const T* b0) {
  const int last = S.nlev - 1;
  for (int l = 0; l < last; ++l) {
    const BLevel& L = S.lev[l];
    const T* b = l == 0 ? b0 : (const T*)L.b;
    T* x = (T*)L.x;
    T* tt = (T*)L.t;
    if (S.nu_pre == 0) {
      for (int i = t.tid; i < L.n; i += t.threads) x[i] = 0;
    } else {
      // first sweep from zero: x = D^-1 b; the others alternate so the last writes x
      T* dst = ((S.nu_pre - 1) % 2 == 0) ? x : tt;
      const T* dv = (const T*)L.dinv;
      for (int i = t.tid; i < L.n; i += t.threads) dst[i] = dv[i] * b[i];
      const T* src = dst;
      for (int k = 1; k < S.nu_pre; ++k) {
        t.sync();
        T* d2 = ((S.nu_pre - 1 - k) % 2 == 0) ? x : tt;
        Phase<lsweep<TM, T>>::run(t, L, b, src, d2);
        src = d2;
      }
    }
    t.sync();
    Phase<lresid<TM, T>>::run(t, L, b, x, (T*)L.r);
    t.sync();
    // b_{l+1} = R r
    T* bn = (T*)S.lev[l + 1].b;
    Phase<lrestrict<TM, T>>::run(t, L, (const T*)L.r, bn);
    t.sync();
  }
  {
    // coarsest level: x = Cinv b in FP64, one warp per row, lanes over the columns,
    // then a fixed shuffle tree
    const BLevel& Lc = S.lev[last];
    const T* b = last == 0 ? b0 : (const T*)Lc.b;
    T* xo = last == 0 ? (T*)S.zc : (T*)Lc.x;
    const int n = Lc.n;
    const double* __restrict__ Cinv = S.Cinv;
    const int lane = threadIdx.x & 31;
    for (int i = t.tid >> 5; i < n; i += t.threads >> 5) {
      double s = 0.0;
      for (int q = lane; q < n; q += 32) s += Cinv[(size_t)i * n + q] * (double)b[q];
      s = warp_sum(s);
      if (lane == 0) xo[i] = (T)s;
    }
    t.sync();
  }
  for (int l = last - 1; l >= 0; --l) {
    const BLevel& L = S.lev[l];
    const T* b = l == 0 ? b0 : (const T*)L.b;
    const T* xc = (l + 1 == last) ? (const T*)S.lev[l + 1].x : (const T*)S.lev[l + 1].x2;
    T* x = (T*)L.x;
    T* tt = (T*)L.t;
    T* out = l == 0 ? (T*)S.zc : (T*)L.x2;
    Phase<lprolong<TM, T>>::run(t, L, xc, x);
    t.sync();
    if (S.nu_post == 0) {
      for (int i = t.tid; i < L.n; i += t.threads) out[i] = x[i];
    } else {
      const T* src = x;
      for (int k = 0; k < S.nu_post; ++k) {
        T* dst = (k == S.nu_post - 1) ? out : (src == x ? tt : x);
        Phase<lsweep<TM, T>>::run(t, L, b, src, dst);
        if (k + 1 < S.nu_post) t.sync();
        src = dst;
      }
    }
    t.sync();
  }
}

// The ILU(0) solves, one quad per row (lane r: component r), with the library's
// rounding sequence.  A level is a few dozen rows, so a solve is the latency of its
// levels, one after the other.
//
// One block (tri_solve) separates the levels by its barrier.  (Reading the rows of the
// coming levels ahead of the barrier made the solves of clouds up to a third shorter,
// those of grids up to twice as long, and the other phases longer with its registers:
// with everything else alike 27.7 instead of 21.9 ms for 152 grids of 8,000 cells, 22.0
// instead of 23.0 for 152 clouds of 3,750.)  On a cluster a barrier that publishes global memory costs about
// 5 us, so there (tri_solve_poll) the rows are dealt over the cluster's quads in
// schedule order and wait for their dependencies' values instead (a sentinel until
// they are written, read a bounded number of times).  The quads take their rows in order
// and the blocks of a cluster run together, so each wait ends: a 32k-point cloud (405
// levels) on eight blocks, 7 iterations, 41.5 ms with a barrier per level, 25 ms so.
//
// Forward: y = L^-1 rhs.  Backward (UPPER): y = U^-1 rhs and z = P zc + y.
template <class T, bool UPPER>
__device__ __forceinline__ void tri_solve(const Solo&, const BSys& S, const T* rhs, T* y, T* z) {
  const int32_t* off = UPPER ? S.offb : S.offf;
  const int32_t* ord = UPPER ? S.ordb : S.ordf;
  const int32_t* rp = UPPER ? S.Urp : S.Lrp;
  const int32_t* ci = UPPER ? S.Uci : S.Lci;
  const T* F = (const T*)(UPPER ? S.Uv : S.Lv);
  const int nl = UPPER ? S.nlb : S.nlf;
  const int r = threadIdx.x & 3, quad = threadIdx.x >> 2, nquad = kBT >> 2;
  const unsigned qmask = 0xFu << ((threadIdx.x & 31) & ~3);
  const int q0 = (threadIdx.x & 31) & ~3;
  for (int lv = 0; lv < nl; ++lv) {
    const int pe = off[lv + 1];
    for (int p = off[lv] + quad; p < pe; p += nquad) {
      const int i = ord[p];
      if (i < 0) continue;
      T d[4] = {0, 0, 0, 0}, y1 = 0;
      if (UPPER) {
        // inv(U_ii) and the first-stage part before the row's sums
        const T* dp = (const T*)S.Dinv + 16 * (size_t)p + 4 * r;
#pragma unroll
        for (int q = 0; q < 4; ++q) d[q] = dp[q];
        if (S.first) {
          const T* zc = (const T*)S.zc;
          if (r == S.e0) y1 = zc[S.ne * (size_t)i];
          else if (S.ne == 2 && r == S.e1) y1 = zc[2 * (size_t)i + 1];
        }
      }
      T acc = rhs[4 * (size_t)i + r];
      for (int k = rp[p]; k < rp[p + 1]; ++k) {
        T f[4], yj[4];
        const T* fp = F + 16 * (size_t)k + 4 * r;
        const T* yp = y + 4 * (size_t)ci[k];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          f[q] = fp[q];
          yj[q] = yp[q];
        }
        acc = sub_rn(acc, dot4(f, yj));
      }
      if (UPPER) {
        T s4[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) s4[q] = __shfl_sync(qmask, acc, q0 + q);
        acc = dot4(d, s4);
        z[4 * (size_t)i + r] = y1 + acc;
      }
      y[4 * (size_t)i + r] = acc;
    }
    __syncthreads();
  }
}

// The same solves on a cluster; forward: y_next becomes the sentinel.
template <class T, bool UPPER>
__device__ __noinline__ void tri_solve_poll(const Team& t, const BSys& S, const T* rhs, T* y,
                                            T* y_next, T* z) {
  const int32_t* __restrict__ ord = UPPER ? S.ordb : S.ordf;
  const int32_t* __restrict__ rp = UPPER ? S.Urp : S.Lrp;
  const int32_t* __restrict__ ci = UPPER ? S.Uci : S.Lci;
  const T* __restrict__ F = (const T*)(UPPER ? S.Uv : S.Lv);
  constexpr int K = sizeof(T) == 4 ? 4 : 3;  // dependencies read together
  const int npos = UPPER ? S.offb[S.nlb] : S.offf[S.nlf];
  const int r = threadIdx.x & 3, quad = t.tid >> 2, nquad = t.threads >> 2;
  const unsigned qmask = 0xFu << ((threadIdx.x & 31) & ~3);
  const int q0 = (threadIdx.x & 31) & ~3;
  for (int p = quad; p < npos; p += nquad) {
    const int i = ord[p];
    if (i < 0) continue;
    const int kb = rp[p], ke = rp[p + 1];
    T acc = rhs[4 * (size_t)i + r], y1 = 0, d[4];
    if (UPPER) {
      // inv(U_ii) and the first-stage part
      ld4((const T*)S.Dinv + 16 * (size_t)p + 4 * r, d);
      if (S.first) {
        const T* zc = (const T*)S.zc;
        if (r == S.e0) y1 = zc[S.ne * (size_t)i];
        else if (S.ne == 2 && r == S.e1) y1 = zc[2 * (size_t)i + 1];
      }
    }
    for (int k = kb; k < ke; k += K) {
      const T* yp[K];
      T f[K][4], x[K][4];
      unsigned todo = 0;
#pragma unroll
      for (int u = 0; u < K; ++u)
        if (k + u < ke) {
          yp[u] = y + 4 * (size_t)ci[k + u];
          ld4(F + 16 * (size_t)(k + u) + 4 * r, f[u]);
          todo |= 1u << u;
        }
      for (unsigned s = 0; todo; ++s) {
#pragma unroll
        for (int u = 0; u < K; ++u)
          if (todo >> u & 1u) ld_volatile4(yp[u], x[u]);
#pragma unroll
        for (int u = 0; u < K; ++u)
          if ((todo >> u & 1u) && !is_sentinel(x[u][0]) && !is_sentinel(x[u][1]) &&
              !is_sentinel(x[u][2]) && !is_sentinel(x[u][3]))
            todo &= ~(1u << u);
        if (!todo) break;
        if (s + 1 >= S.spin) {
          atomicExch(S.fail, 1);
          break;
        }
        if ((s & 255u) == 255u && ld_volatile_i32(S.fail)) break;
      }
#pragma unroll
      for (int u = 0; u < K; ++u)
        if (k + u < ke) acc = sub_rn(acc, dot4(f[u], x[u]));
    }
    if (UPPER) {
      T s4[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) s4[q] = __shfl_sync(qmask, acc, q0 + q);
      acc = dot4(d, s4);
    }
    st_volatile(y + 4 * (size_t)i + r, desentinel(acc));
    if (UPPER) z[4 * (size_t)i + r] = y1 + acc;
    else y_next[4 * (size_t)i + r] = sentinel_of(T(0));
  }
  t.sync();
}

// z = M^-1 v (Eq. 3) for the FP64 vector v; z in the apply precision.
template <class TM, class T>
__device__ __forceinline__ void bprecond(const TM& t, const BSys& S, const double* v, T* z) {
  const int N = S.N;
  T* rhat = (T*)S.rhat;
  T* zc = (T*)S.zc;
  T* r2 = (T*)S.r2;
  T* u = (T*)S.u;
  T* y2 = (T*)S.y2;
  if (S.first) {
    // Quasi-IMPES restriction: rhat_i = v_i[e] - W_i v_i[h]
    const T* W = (const T*)S.Wt;
    for (int i = t.tid; i < N; i += t.threads) {
      const double* rv = v + 4 * (size_t)i;
      const T* w = W + 4 * (size_t)i;
      if (S.ne == 2) {
        T re0 = (T)rv[S.e0], re1 = (T)rv[S.e1], rh0 = (T)rv[S.h0], rh1 = (T)rv[S.h1];
        rhat[2 * (size_t)i] = re0 - w[0] * rh0 - w[1] * rh1;
        rhat[2 * (size_t)i + 1] = re1 - w[2] * rh0 - w[3] * rh1;
      } else {
        rhat[i] = (T)rv[S.e0] - w[0] * (T)rv[S.h0] - w[1] * (T)rv[S.h1] - w[2] * (T)rv[S.h2];
      }
    }
    t.sync();
    Phase<bvcycle<TM, T>>::run(t, S, rhat);
    // correction: r2 = v - A P zc (elliptic columns of A only)
    const T* __restrict__ ae = (const T*)S.AE;
    const int32_t* __restrict__ rp = S.rp;
    const int32_t* __restrict__ ci = S.ci;
    const int ne = S.ne;
    for (int g = t.tid; g < 4 * N; g += t.threads) {
      const int i = g >> 2, r = g & 3;
      T acc = 0;
      int k = rp[i];
      const int k1 = rp[i + 1];
      for (; k + 4 <= k1; k += 4) {
        int j[4];
        T a0[4], a1[4], z0[4], z1[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          j[q] = ci[k + q];
          a0[q] = ae[8 * (size_t)(k + q) + 2 * r];
          a1[q] = ae[8 * (size_t)(k + q) + 2 * r + 1];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          z0[q] = ne == 2 ? zc[2 * (size_t)j[q]] : zc[j[q]];
          z1[q] = ne == 2 ? zc[2 * (size_t)j[q] + 1] : T(0);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (ne == 2) acc += a0[q] * z0[q] + a1[q] * z1[q];
          else acc += a0[q] * z0[q];
        }
      }
      for (; k < k1; ++k) {
        const int jj = ci[k];
        const T* a = ae + 8 * (size_t)k + 2 * r;
        if (ne == 2) acc += a[0] * zc[2 * (size_t)jj] + a[1] * zc[2 * (size_t)jj + 1];
        else acc += a[0] * zc[jj];
      }
      r2[g] = (T)v[g] - acc;
    }
  } else {
    for (int g = t.tid; g < 4 * N; g += t.threads) r2[g] = (T)v[g];
  }
  if constexpr (std::is_same_v<TM, Solo>) {
    t.sync();
    tri_solve<T, false>(t, S, r2, u, nullptr);
    tri_solve<T, true>(t, S, u, y2, z);
  } else {
    for (int g = t.tid; g < 4 * N; g += t.threads) u[g] = sentinel_of(T(0));
    t.sync();
    tri_solve_poll<T, false>(t, S, r2, u, y2, nullptr);
    tri_solve_poll<T, true>(t, S, u, y2, nullptr, z);
  }
}

// Flexible GMRES(m) with CGS2 and Givens rotations for one system per cluster,
// the same algorithm (and stopping rules) as the per-system driver:
// convergence when ||b - A x|| <= tol ||b||, iterations = preconditioner
// applications, a cycle ends at m steps, on convergence of the estimate, at
// maxit or on an exact breakdown, and the true residual decides whether to
// start another.  Every block keeps the Hessenberg matrix and takes the same
// decisions from the same sums.
template <class T, class TM>
__global__ void __launch_bounds__(kBT, 1) k_batch_fgmres(const BSys* __restrict__ sys,
                                                      BOut* __restrict__ out) {
  const TM t;
  const int id = blockIdx.x / t.size;
  // the system's descriptor in shared memory: its pointers are then read
  // without a global load, and stores to global memory cannot alias them
  __shared__ BSys S;
  {
    const int4* src = reinterpret_cast<const int4*>(sys + id);
    int4* dst = reinterpret_cast<int4*>(&S);
    for (int k = threadIdx.x; k < (int)(sizeof(BSys) / 16); k += blockDim.x) dst[k] = src[k];
  }
  __shared__ Partials P;
  if (threadIdx.x == 0) P.flip = 0;
  t.sync();  // (every block of the cluster has started before any reads its memory)
  __shared__ double sH[(kBMaxM + 1) * kBMaxM];  // column j at j*(m+1), rotated
  __shared__ double scs[kBMaxM], ssn[kBMaxM], sg[kBMaxM + 1], sy[kBMaxM], sh1[kBMaxM + 1],
      sh2[kBMaxM + 1], snrm[1];
  __shared__ int s_stop;
  const int n4 = 4 * S.N, m = S.m;
  const int tid = threadIdx.x;
  T* Z = (T*)S.Z;
  // ||b||
  Phase<team_dots<TM>>::run(t, P, S.b, S.b, n4, 1, snrm);
  const double bnorm = sqrt(snrm[0]);
  const double tol_abs = S.tol * bnorm;
  int iters = 0, status = CPTR_OK;
  double beta = 0.0;
  if (bnorm == 0.0) {
    for (int i = t.tid; i < n4; i += t.threads) S.x[i] = 0.0;
  } else {
    for (;;) {
      // r = b - A x into V_0, beta = ||r||
      Phase<bspmv<TM, double>>::run(t, S, S.x, S.b, S.V);
      t.sync();
      Phase<team_dots<TM>>::run(t, P, S.V, S.V, n4, 1, snrm);
      beta = sqrt(snrm[0]);
      if (!isfinite(beta)) { status = CPTR_ERR_BREAKDOWN; break; }
      if (beta <= tol_abs) break;
      if (iters >= S.maxit) { status = CPTR_ERR_MAXIT; break; }
      for (int i = t.tid; i < n4; i += t.threads) S.V[i] = S.V[i] / beta;
      if (tid == 0) {
        sg[0] = beta;
        for (int l = 1; l <= m; ++l) sg[l] = 0.0;
      }
      t.sync();
      int k = 0;
      for (int j = 0; j < m; ++j) {
        const double* vj = S.V + (size_t)j * n4;
        T* zj = Z + (size_t)j * n4;
        Phase<bprecond<TM, T>>::run(t, S, vj, zj);
        if (t.size > 1 && ld_volatile_i32(S.fail)) {  // (set before the last barrier)
          status = CPTR_ERR_TIMEOUT;
          break;
        }
        Phase<bspmv<TM, T>>::run(t, S, zj, nullptr, S.w);
        t.sync();
        // CGS2: h1 = V^T w; w -= V h1; h2 = V^T w; w -= V h2
        for (int pass = 0; pass < 2; ++pass) {
          double* hh = pass == 0 ? sh1 : sh2;
          Phase<team_dots<TM>>::run(t, P, S.V, S.w, n4, j + 1, hh);
          Phase<team_update<TM>>::run(t, S.V, S.w, n4, j + 1, hh);
          t.sync();
        }
        Phase<team_dots<TM>>::run(t, P, S.w, S.w, n4, 1, snrm);
        const double hn = sqrt(snrm[0]);
        if (tid == 0) {
          double* col = sH + (size_t)j * (m + 1);
          for (int l = 0; l <= j; ++l) col[l] = sh1[l] + sh2[l];
          col[j + 1] = hn;
          for (int l = 0; l < j; ++l) {
            const double a = col[l], b = col[l + 1];
            col[l] = scs[l] * a + ssn[l] * b;
            col[l + 1] = -ssn[l] * a + scs[l] * b;
          }
          const double a = col[j], b = col[j + 1];
          const double dd = hypot(a, b);
          double cj = 1.0, sj = 0.0;
          if (dd != 0.0) { cj = a / dd; sj = b / dd; }
          scs[j] = cj;
          ssn[j] = sj;
          col[j] = cj * a + sj * b;
          col[j + 1] = 0.0;
          const double gj = sg[j];
          const double gn = -sj * gj;
          sg[j + 1] = gn;
          sg[j] = cj * gj;
          const bool conv = fabs(gn) <= tol_abs;
          s_stop = (!isfinite(gn) || !isfinite(hn) || conv || iters + 1 >= S.maxit ||
                    hn == 0.0 || j + 1 == m) ? 1 : 0;
        }
        __syncthreads();
        ++iters;
        k = j + 1;
        if (s_stop) break;
        const double rinv = 1.0 / hn;
        double* vn = S.V + (size_t)(j + 1) * n4;
        for (int i = t.tid; i < n4; i += t.threads) vn[i] = S.w[i] * rinv;
        t.sync();
      }
      if (status != CPTR_OK) break;
      // y = H^-1 g, x += Z y
      if (tid == 0) {
        for (int i = k - 1; i >= 0; --i) {
          double s = sg[i];
          for (int l = i + 1; l < k; ++l) s -= sH[(size_t)l * (m + 1) + i] * sy[l];
          sy[i] = s / sH[(size_t)i * (m + 1) + i];
        }
      }
      __syncthreads();
      for (int i = t.tid; i < n4; i += t.threads) {
        double xi = S.x[i];
        for (int l = 0; l < k; ++l) xi += sy[l] * (double)Z[(size_t)l * n4 + i];
        S.x[i] = xi;
      }
      t.sync();
    }
  }
  if (tid == 0 && t.rank == 0) {
    out[id].iters = iters;
    out[id].status = status;
    out[id].rel_resid = bnorm > 0.0 ? beta / bnorm : 0.0;
  }
  t.sync();  // no block leaves while another may read its shared memory
}

}  // namespace

namespace {

int hidx_of(int e0, int e1, int k) {
  int h[3] = {-1, -1, -1}, q = 0;
  for (int u = 0; u < 4; ++u)
    if (u != e0 && u != e1) h[q++] = u;
  return h[k];
}

// Descriptor of one set-up context; CPTR_ERR_INVALID for configurations the
// batched kernel does not run (see cptr.h).
cptr_status describe(cptr_ctx* c, double tol, int maxit, BSys* d, std::string& why) {
  if (!c->setup_done) { why = "context not set up"; return CPTR_ERR_INVALID; }
  const int pc = c->p.precond;
  if (pc != CPTR_PREC_CPTR && pc != CPTR_PREC_ILU) { why = "batched solves run CPTR, CPR or ILU(0) alone"; return CPTR_ERR_INVALID; }
  if (c->p.mgr) { why = "batched solves do not run the MGR reduction"; return CPTR_ERR_INVALID; }
  if (c->p.smoother != CPTR_SMOOTH_L1_JACOBI) { why = "batched solves smooth with l1-Jacobi"; return CPTR_ERR_INVALID; }
  if (c->p.restart > kBMaxM) { why = "batched solves need restart <= 32"; return CPTR_ERR_INVALID; }
  if ((int)c->lev.size() > kBMaxLev) { why = "too many AMG levels"; return CPTR_ERR_INVALID; }
  if (!c->Lrp || !c->Urp || !c->Dinv) {
    // the level-ordered factor arrays (built when another schedule was forced)
    cptr_status st = build_level_solve_arrays(c);
    if (st) return st;
    CTX_CUDA(c, cudaStreamSynchronize(c->stream));
  }
  *d = BSys();
  d->N = c->N;
  d->m = c->p.restart;
  d->maxit = maxit > 0 ? maxit : c->p.maxit;
  d->tol = tol > 0.0 ? tol : c->p.tol;
  d->first = pc == CPTR_PREC_CPTR ? 1 : 0;
  d->ne = c->se1 < 0 ? 1 : 2;
  d->e0 = c->se0;
  d->e1 = c->se1;
  d->h0 = hidx_of(c->se0, c->se1, 0);
  d->h1 = hidx_of(c->se0, c->se1, 1);
  d->h2 = hidx_of(c->se0, c->se1, 2);
  d->nu_pre = c->p.nu_pre;
  d->nu_post = c->p.nu_post;
  d->rp = c->rp; d->ci = c->ci; d->v = c->v;
  d->Wt = c->Wt; d->AE = c->AE; d->Cinv = c->Cinv;
  d->rhat = c->rhat; d->zc = c->zc; d->r2 = c->r2; d->u = c->u; d->y2 = c->y2;
  d->nlf = c->nlev_f; d->nlb = c->nlev_b;
  d->offf = c->loff_f; d->ordf = c->ord_f; d->Lrp = c->Lrp; d->Lci = c->Lci; d->Lv = c->Lv;
  d->offb = c->loff_b; d->ordb = c->ord_b; d->Urp = c->Urp; d->Uci = c->Uci; d->Uv = c->Uv;
  d->Dinv = c->Dinv;
  d->spin = c->spin_limit;
  d->fail = nullptr;
  d->V = c->V; d->w = c->w; d->x = c->xd; d->b = c->bd; d->Z = c->Z;
  d->nlev = (int)c->lev.size();
  for (int l = 0; l < d->nlev; ++l) {
    const Level& L = c->lev[l];
    BLevel& B = d->lev[l];
    B.n = L.A.n;
    B.Arp = L.A.rp; B.Aci = L.A.ci; B.Av = L.Av; B.dinv = L.dinv;
    const bool last = l == d->nlev - 1;
    B.nc = last ? 0 : L.nc;
    B.Rrp = L.R.rp; B.Rci = L.R.ci; B.Rv = L.Rv;
    B.Prp = L.P.rp; B.Pci = L.P.ci; B.Pv = L.Pv;
    B.b = L.b; B.x = L.x; B.r = L.r; B.x2 = L.x2; B.t = L.t;
  }
  return CPTR_OK;
}

}  // namespace

extern "C" cptr_status cptr_solve_batch(cptr_ctx* const* ctxs, int n, const double* const* rhs,
                                        double* const* x, double tol, int maxit,
                                        cptr_info* infos) {
  if (!ctxs || n <= 0 || !rhs || !x) return CPTR_ERR_INVALID;
  cptr_ctx* c0 = ctxs[0];
  if (!c0) return CPTR_ERR_INVALID;
  for (int k = 0; k < n; ++k) {
    if (!ctxs[k] || !rhs[k] || !x[k]) return CPTR_ERR_INVALID;
    if (ctxs[k]->dev != c0->dev || ctxs[k]->mixed != c0->mixed) {
      ctx_set_err(c0, "a batch needs one device and one precision");
      return CPTR_ERR_INVALID;
    }
    for (int q = 0; q < k; ++q)
      if (ctxs[q] == ctxs[k]) { ctx_set_err(c0, "a context appears twice in the batch"); return CPTR_ERR_INVALID; }
  }
  auto t0 = std::chrono::steady_clock::now();
  std::vector<BSys> h(n);
  for (int k = 0; k < n; ++k) {
    std::string why;
    cptr_status st = describe(ctxs[k], tol, maxit, &h[k], why);
    if (st) {
      if (!why.empty()) ctx_set_err(c0, why.c_str());
      return st;
    }
  }
  cudaStream_t s = c0->stream;
  // every context's own work (setup, earlier solves) precedes the batch
  for (int k = 0; k < n; ++k) CTX_CUDA(c0, cudaStreamSynchronize(ctxs[k]->stream));
  for (int k = 0; k < n; ++k) {
    size_t nb = sizeof(double) * 4 * (size_t)ctxs[k]->N;
    CTX_CUDA(c0, cudaMemcpyAsync(ctxs[k]->bd, rhs[k], nb, cudaMemcpyDefault, s));
    CTX_CUDA(c0, cudaMemcpyAsync(ctxs[k]->xd, x[k], nb, cudaMemcpyDefault, s));
  }
  // Blocks per system: the largest of 1, 2, 4 and 8 whose blocks hold at least a share of
  // cells each, so that the batch's largest system does not run alone on one SM when the
  // others are done; a block then holds fewer than two shares, but for systems of more
  // than sixteen.  A share is 0.6 of the cells per SM of the batch: with larger ones the
  // last systems leave SMs idle, with smaller ones the barriers cost more than they
  // divide (48 systems of 2k-30k cells take 27.9, 28.1, 27.7 and 36.5 ms with 0.5, 0.6, 0.7
  // and 1, 93.5 with one block each; 120 of 2k-20k 35.3, 35.7, 33.6, 33.7 and 57.9).  It
  // is at least kBlockCells, and at most kMostCells, whatever the batch: a block of many
  // cells loses more to its L1 than the barriers cost (160 systems of 2k-28k cells: 62.8 ms
  // without that limit, 62.8 with 5632, 52.4 with 4096, 55.1 with 3072; 200 of 2k-30k
  // 83.5, 69.4, 72.8, 71.7; 304 of 2k-28k 91.4, 90.9, 94.0, 96.1).  Systems are laid out by
  // their blocks and each group is one launch, side by side on its first system's second
  // stream.
  constexpr long long kBlockCells = 1024, kMostCells = 4096;
  long long cells = 0;
  for (int k = 0; k < n; ++k) cells += ctxs[k]->N;
  const long long share = std::clamp(3 * cells / (5 * std::max(1, c0->nsm)), kBlockCells,
                                     kMostCells);
  const char* env = getenv("CPTR_BATCH_BLOCKS");  // test hook
  const int forced = env ? atoi(env) : 0;
  std::vector<int> order(n), blocks(n);
  for (int k = 0; k < n; ++k) {
    order[k] = k;
    blocks[k] = 1;
    while (blocks[k] < 8 && 2 * blocks[k] * share <= ctxs[k]->N) blocks[k] *= 2;
    if (forced == 1 || forced == 2 || forced == 4 || forced == 8) blocks[k] = forced;
  }
  std::stable_sort(order.begin(), order.end(),
                   [&](int a, int b) { return blocks[a] > blocks[b]; });
  std::vector<BSys> hs(n);
  BSys* dsys = nullptr;
  BOut* dout = nullptr;
  CTX_CUDA(c0, cudaMallocAsync((void**)&dsys, sizeof(BSys) * (size_t)n, s));
  cudaError_t e = cudaMallocAsync((void**)&dout, sizeof(BOut) * (size_t)n, s);
  if (e != cudaSuccess) { cudaFreeAsync(dsys, s); return ctx_cuda_fail(c0, e, "batch outputs"); }
  std::vector<BOut> ho(n);
  for (int k = 0; k < n; ++k) {
    hs[k] = h[order[k]];
    hs[k].fail = &dout[k].fail;  // (an address on the device)
  }
  e = cudaMemsetAsync(dout, 0, sizeof(BOut) * (size_t)n, s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(dsys, hs.data(), sizeof(BSys) * (size_t)n, cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaEventRecord(c0->ev_fork, s);
  for (int k0 = 0; k0 < n && e == cudaSuccess;) {
    const int size = blocks[order[k0]];
    int k1 = k0;
    while (k1 < n && blocks[order[k1]] == size) ++k1;
    cptr_ctx* lead = ctxs[order[k0]];
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((k1 - k0) * size);
    cfg.blockDim = dim3(kBT);
    cfg.stream = lead->stream2;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = size;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = size > 1 ? 1 : 0;
    const BSys* sy = dsys + k0;
    auto kern = c0->mixed ? (size > 1 ? k_batch_fgmres<float, Team> : k_batch_fgmres<float, Solo>)
                          : (size > 1 ? k_batch_fgmres<double, Team> : k_batch_fgmres<double, Solo>);
    e = cudaStreamWaitEvent(lead->stream2, c0->ev_fork, 0);
    if (e == cudaSuccess) e = cudaLaunchKernelEx(&cfg, kern, sy, dout + k0);
    ++c0->nlaunch;
    // (also after a failed launch: what runs on the other streams is waited for)
    if (cudaEventRecord(lead->ev_join, lead->stream2) != cudaSuccess ||
        cudaStreamWaitEvent(s, lead->ev_join, 0) != cudaSuccess) {
      if (e == cudaSuccess) e = cudaErrorUnknown;
      cudaStreamSynchronize(lead->stream2);
    }
    k0 = k1;
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(ho.data(), dout, sizeof(BOut) * (size_t)n, cudaMemcpyDeviceToHost, s);
  for (int k = 0; k < n && e == cudaSuccess; ++k)
    e = cudaMemcpyAsync(x[k], ctxs[k]->xd, sizeof(double) * 4 * (size_t)ctxs[k]->N,
                        cudaMemcpyDefault, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFreeAsync(dsys, s);
  cudaFreeAsync(dout, s);
  if (e != cudaSuccess) return ctx_cuda_fail(c0, e, "batched solve");
  const double secs = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
  cptr_status worst = CPTR_OK;
  std::vector<BOut> hk(n);  // in the caller's order
  for (int k = 0; k < n; ++k) hk[order[k]] = ho[k];
  ho = hk;
  for (int k = 0; k < n; ++k) {
    cptr_ctx* c = ctxs[k];
    c->info.iters = ho[k].iters;
    c->info.rel_resid = ho[k].rel_resid;
    c->info.status = ho[k].status;
    c->info.solve_s = secs;
    c->info.launches = c->nlaunch;
    if (infos) infos[k] = c->info;
    if (ho[k].status == CPTR_ERR_TIMEOUT)
      ctx_set_err(c0, "a bounded device-side wait gave up");
    if (worst == CPTR_OK || (worst == CPTR_ERR_MAXIT && ho[k].status != CPTR_OK))
      worst = (cptr_status)ho[k].status;
  }
  return worst;
}
