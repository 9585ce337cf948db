// Block ILU(0) of the 4x4 BSR matrix on the device (paper Section 3.1: the
// second stage is ILU with zero fill-in on the global matrix), natural order,
// no pivoting: for each row i and each k < i in row i (ascending),
//   L_ik = A_ik inv(U_kk);  A_ij -= L_ik U_kj  for j > k present in rows i and k;
// then inv(U_ii) is stored in place of the diagonal block.
//
// Rows are factorised by a sync-free kernel that follows the level schedule of
// the lower triangle (level(i) = 1 + max level(k), k < i in row i): a warp
// claims the next two rows of the schedule (one, of matrices with a row of more than
// 32 blocks), waits (bounded) for the rows they need, and publishes their completion
// with release flags.  The same schedule, and the
// one of the upper triangle, order the triangular solves.
#include <vector>

#include "common.cuh"
#include "ctx.h"

namespace {

constexpr int kT = 256;
inline int nblk(long long n, int per = kT) { return n > 0 ? ceil_div(n, per) : 1; }

// level(i) = 1 + max over dependencies (0 if none) in one pass.  Warps claim
// groups of 32 rows in dependency order (increasing index for the lower
// triangle, decreasing for the upper), so every dependency of a row belongs to
// a group claimed earlier by a running warp; a row waits until its
// dependencies' levels are written (-1 before), polling a bounded number of times.
__global__ void __launch_bounds__(256) k_level_syncfree(int N, const int32_t* __restrict__ rp,
                                                        const int32_t* __restrict__ ci,
                                                        const int32_t* __restrict__ diag,
                                                        int32_t* lvl, bool upper, unsigned* ctr,
                                                        int* status) {
  const int lane = threadIdx.x & 31;
  for (;;) {
    unsigned g0 = 0;
    if (lane == 0) g0 = atomicAdd(ctr, 32u);
    g0 = __shfl_sync(0xffffffffu, g0, 0);
    if (g0 >= (unsigned)N) return;
    const int k = (int)g0 + lane;
    // A lane that gives up leaves its row unwritten and the whole warp stops
    // at the vote below: every lane must reach the next __shfl_sync, so no
    // lane may leave the kernel on its own.
    bool quit = false;
    if (k < N) {
      const int i = upper ? N - 1 - k : k;
      const int t0 = upper ? diag[i] + 1 : rp[i];
      const int t1 = upper ? rp[i + 1] : diag[i];
      int m = 0;
      for (int t = t0; t < t1 && !quit; ++t) {
        const int32_t* pj = lvl + ci[t];
        int q = ld_volatile_i32(pj);
        for (unsigned sp = 0; q < 0; ++sp) {
          if ((sp & 255u) == 255u) {
            if (ld_volatile_i32(status) != DEV_OK) { quit = true; break; }
            if (sp > CPTR_SPIN_LIMIT) {
              dev_fail(status, DEV_TIMEOUT);
              quit = true;
              break;
            }
          }
          q = ld_volatile_i32(pj);
        }
        m = q + 1 > m ? q + 1 : m;
      }
      if (!quit) st_release_i32(lvl + i, m);
    }
    if (__any_sync(0xffffffffu, quit)) return;
  }
}

__global__ void k_level_count(int N, const int32_t* __restrict__ lvl, int32_t* __restrict__ cnt,
                              int* maxlvl) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  atomicAdd(&cnt[lvl[i]], 1);
  atomicMax(maxlvl, lvl[i]);
}

__global__ void k_pad8(int n, const int32_t* __restrict__ cnt, int32_t* __restrict__ pc) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) pc[i] = (cnt[i] + 7) & ~7;
}

__global__ void k_level_fill(int N, const int32_t* __restrict__ lvl, const int32_t* __restrict__ off,
                             int32_t* __restrict__ cur, int32_t* __restrict__ ord) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  int L = lvl[i];
  ord[off[L] + atomicAdd(&cur[L], 1)] = i;
}

// 4x4 inverse by Gauss-Jordan elimination with partial pivoting.
__device__ bool inv4(const double* M, double* out) {
  double a[4][8];
  for (int r = 0; r < 4; ++r)
    for (int c = 0; c < 8; ++c) a[r][c] = (c < 4) ? M[r * 4 + c] : (c - 4 == r ? 1.0 : 0.0);
  for (int c = 0; c < 4; ++c) {
    int p = c;
    double best = fabs(a[c][c]);
    for (int r = c + 1; r < 4; ++r)
      if (fabs(a[r][c]) > best) { best = fabs(a[r][c]); p = r; }
    if (!(best > 0.0) || !isfinite(best)) return false;
    if (p != c)
      for (int k = 0; k < 8; ++k) { double t = a[c][k]; a[c][k] = a[p][k]; a[p][k] = t; }
    double d = a[c][c];
    for (int k = 0; k < 8; ++k) a[c][k] /= d;
    for (int r = 0; r < 4; ++r) {
      if (r == c) continue;
      double f = a[r][c];
      for (int k = 0; k < 8; ++k) a[r][k] -= f * a[c][k];
    }
  }
  for (int r = 0; r < 4; ++r)
    for (int c = 0; c < 4; ++c) out[r * 4 + c] = a[r][c + 4];
  return true;
}

// The same inversion of two blocks by one warp, in place: lane 4 r + c of each
// half holds entry (r, c) and returns that of the inverse.  Pivots as in inv4;
// the columns, exchanged instead of an augmented half, are put back at the end.
// ok is false for the half whose block has no finite nonzero pivot.
__device__ __forceinline__ double inv4_pair(double a, bool* ok) {
  constexpr unsigned FULL = 0xffffffffu;
  const int hl = threadIdx.x & 15, r = hl >> 2, c = hl & 3;
  int piv[4];
  *ok = true;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    // candidate pivots a[rr][k], rr >= k (first maximum wins; |x| and the
    // comparisons run on bit patterns with IEEE results: a NaN never wins, a NaN
    // first candidate is kept)
    int p = k;
    unsigned long long best = dmag(__shfl_sync(FULL, a, 4 * k + k, 16));
#pragma unroll
    for (int rr = k + 1; rr < 4; ++rr) {
      const unsigned long long v = dmag(__shfl_sync(FULL, a, 4 * rr + k, 16));
      if (v > best && v <= 0x7ff0000000000000ull && best <= 0x7ff0000000000000ull) {
        best = v;
        p = rr;
      }
    }
    if (best == 0 || best >= 0x7ff0000000000000ull) *ok = false;
    piv[k] = p;
    a = __shfl_sync(FULL, a, 4 * (r == k ? p : r == p ? k : r) + c, 16);  // rows k and p
    const double d = __shfl_sync(FULL, a, 4 * k + k, 16);
    const double t = (c == k ? 1.0 : a) / d;
    const double row = __shfl_sync(FULL, t, 4 * k + c, 16);
    const double f = __shfl_sync(FULL, a, 4 * r + k, 16);
    a = r == k ? t : (c == k ? 0.0 : a) - f * row;
  }
#pragma unroll
  for (int k = 3; k >= 0; --k)
    a = __shfl_sync(FULL, a, 4 * r + (c == k ? piv[k] : c == piv[k] ? k : c), 16);
  return a;
}

__device__ __forceinline__ bool wait_flag(const int* flag, int epoch, int* status) {
  for (unsigned s = 0;; ++s) {
    if (ld_acquire_i32(flag) == epoch) return true;
    if (s >= 32) __nanosleep(128);  // back off: fewer polls competing with working warps
    if ((s & 255u) == 255u) {
      if (ld_volatile_i32(status) != DEV_OK) return false;
      if (s > CPTR_SPIN_LIMIT) {
        dev_fail(status, DEV_TIMEOUT);
        return false;
      }
    }
  }
}

// One warp per row; lanes 0..15 hold one entry (r, c) of a 4x4 block product.
__global__ void __launch_bounds__(256) k_ilu_factor(int npos, const int32_t* __restrict__ ord,
                                                    const int32_t* __restrict__ rp,
                                                    const int32_t* __restrict__ ci,
                                                    const int32_t* __restrict__ diag, double* LU,
                                                    int* done, int epoch, Ctl* ctl) {
  int lane = threadIdx.x & 31;
  int r = lane >> 2, c = lane & 3;
  bool act = lane < 16;
  for (;;) {
    unsigned item = 0;
    if (lane == 0) item = atomicAdd(&ctl->fac_ctr, 1u);
    item = __shfl_sync(0xffffffffu, item, 0);
    if (item >= (unsigned)npos) return;
    int i = ord[item];
    if (i < 0) continue;
    int t0 = rp[i], td = diag[i], t1 = rp[i + 1];
    for (int t = t0; t < td; ++t) {
      int k = ci[t];
      if (lane == 0) wait_flag(done + k, epoch, &ctl->status);
      __syncwarp();
      const double* Ukk = LU + 16 * (size_t)diag[k];  // holds inv(U_kk)
      double* Aik = LU + 16 * (size_t)t;
      double s = 0.0;
      if (act)
        for (int q = 0; q < 4; ++q) s += __ldcg(Aik + r * 4 + q) * __ldcg(Ukk + q * 4 + c);
      __syncwarp();
      if (act) Aik[r * 4 + c] = s;
      __syncwarp();
      // A_ij -= L_ik U_kj for j > k present in both rows
      int k1 = rp[k + 1];
      int t2 = diag[k] + 1;
      for (int t3 = t + 1; t3 < t1; ++t3) {
        int j = ci[t3];
        while (t2 < k1 && ci[t2] < j) ++t2;
        if (t2 < k1 && ci[t2] == j) {
          const double* Ukj = LU + 16 * (size_t)t2;
          double p = 0.0;
          if (act)
            for (int q = 0; q < 4; ++q) p += __ldcg(Aik + r * 4 + q) * __ldcg(Ukj + q * 4 + c);
          __syncwarp();
          if (act) LU[16 * (size_t)t3 + r * 4 + c] = __ldcg(LU + 16 * (size_t)t3 + r * 4 + c) - p;
          __syncwarp();
        }
      }
    }
    if (lane == 0) {
      double blk[16], inv[16];
      double* Dii = LU + 16 * (size_t)td;
      for (int q = 0; q < 16; ++q) blk[q] = __ldcg(Dii + q);
      if (!inv4(blk, inv)) {
        dev_fail(&ctl->status, DEV_BREAKDOWN);
        for (int q = 0; q < 16; ++q) inv[q] = 0.0;
      }
      for (int q = 0; q < 16; ++q) Dii[q] = inv[q];
      __threadfence();
      st_release_i32(done + i, epoch);
    }
    __syncwarp();
  }
}

// The same factorisation, two rows per warp: sixteen lanes per row, lane 4 r + c
// holding entry (r, c) of a 4x4 block, both rows (neighbours in the schedule, so
// of one level) in lockstep.  Every product and sum rounds by itself, as in
// k_ilu_factor and in the definition: with fused products a pivot block that cancels
// exactly keeps a residue, and a singular matrix is no longer refused (of 93 two-cell
// systems with repeated block rows that the definition refuses, 72 went through).  The
// kernel is bound by FP64 issue on wide levels, where an instruction costs the same for
// 16 lanes as for 32, and by the
// chain flag - inv(U_kk) - L_ik - update - ... - inversion - flag on narrow ones,
// where a row's first dependency may be its last to come: the rows share every
// FP64 instruction; the row's blocks and the columns that row i and its
// dependencies share (pattern only) are ready before the first wait; the flags
// are read together, and a published dependency's blocks are loaded while the one
// before it is worked on; one release publishes the row.  Rows longer than maxrow
// blocks do not come here.  200x200x100 grid 34.8 -> 12.9 ms (9.8 with fused products),
// 64x64x32 grid 2.2 -> 1.4 ms; narrow levels of long rows gain nothing: 1M-point cloud
// 21.7 -> 22.1 ms (17.5 fused).  (Before: one row per warp, a dependency's loads after
// its own flag.)
constexpr int kRowMax = 32;
constexpr int kFacWarps = 4;
constexpr int kAhead = 2;  // shared blocks of a dependency loaded ahead
struct FacRow {  // shared memory of one row: byte offsets, cap shared columns listed
  int cj, ms, mp, mt, cap, bytes;
};
inline FacRow fac_row(int maxrow) {
  FacRow L;
  L.cap = 4 * maxrow;
  L.cj = 128 * maxrow;
  L.ms = L.cj + 4 * maxrow;
  L.mp = L.ms + 4 * (maxrow + 1);
  L.mt = L.mp + 4 * L.cap;
  L.bytes = (L.mt + L.cap + 15) & ~15;
  return L;
}

__global__ void __launch_bounds__(32 * kFacWarps) k_ilu_factor_pair(
    int npos, FacRow Ly, const int32_t* __restrict__ ord, const int32_t* __restrict__ rp,
    const int32_t* __restrict__ ci, const int32_t* __restrict__ diag, double* LU, int* done,
    int epoch, Ctl* ctl) {
  extern __shared__ __align__(16) unsigned char fsm[];
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, half = lane >> 4, hl = lane & 15, r = hl >> 2, c = hl & 3;
  unsigned char* base = fsm + (size_t)(threadIdx.x >> 4) * Ly.bytes;
  double* bi = reinterpret_cast<double*>(base);
  int* cj = reinterpret_cast<int*>(base + Ly.cj);
  int* ms = reinterpret_cast<int*>(base + Ly.ms);  // first shared column of each dependency
  int* mp = reinterpret_cast<int*>(base + Ly.mp);  // its block of row k
  unsigned char* mt = base + Ly.mt;                // its block of row i
  const unsigned ngroups = (unsigned)((npos + 1) >> 1);
  int* const status = &ctl->status;
  for (;;) {
    unsigned g = 0;
    if (lane == 0) g = atomicAdd(&ctl->fac_ctr, 1u);
    g = __shfl_sync(FULL, g, 0);
    if (g >= ngroups) return;
    const int pos = (int)(2 * g) + half;
    const int i = pos < npos ? ord[pos] : -1;
    const int t0 = i >= 0 ? rp[i] : 0, ni = i >= 0 ? rp[i + 1] - t0 : 0;
    const int di = i >= 0 ? diag[i] - t0 : 0;
    for (int e = hl; e < ni; e += 16) cj[e] = ci[t0 + e];
#pragma unroll 4
    for (int e = 0; e < ni; ++e) bi[16 * e + hl] = LU[16 * (size_t)(t0 + e) + hl];
    __syncwarp();
    const int maxd = __reduce_max_sync(FULL, di);
    // the later columns of row i in the upper part of row k = cj[e], listed from
    // slot n on; returns their number
    auto shared_columns = [&](int e, bool act, int n) {
      const int k = act ? cj[e] : 0, kd = act ? diag[k] : 0, ke = act ? rp[k + 1] : 0;
      const int maxl = __reduce_max_sync(FULL, act ? ni - e - 1 : 0);
      int nm = 0;
      for (int b = 0; b < maxl; b += 16) {
        const int t3 = e + 1 + b + hl;
        int at = -1;
        if (act && t3 < ni) {
          const int j = cj[t3];
          int lo = kd + 1, hi = ke - 1;
          while (lo <= hi) {
            const int mid = (lo + hi) >> 1, x = ci[mid];
            if (x == j) { at = mid; break; }
            if (x < j) lo = mid + 1; else hi = mid - 1;
          }
        }
        const unsigned m = (__ballot_sync(FULL, at >= 0) >> (16 * half)) & 0xffffu;
        const int slot = n + nm + __popc(m & ((1u << hl) - 1u));
        if (at >= 0 && slot < Ly.cap) {
          mt[slot] = (unsigned char)t3;
          mp[slot] = at;
        }
        nm += __popc(m);
      }
      return nm;
    };
    int listed = 0, late = 0;  // dependencies from `late` on did not fit the list
    {
      bool fits = true;
      for (int e = 0; e < maxd; ++e) {
        const int nm = shared_columns(e, fits && e < di, listed);
        if (fits && e < di) {
          fits = listed + nm <= Ly.cap;
          if (fits) {
            if (hl == 0) ms[e] = listed;
            listed += nm;
            late = e + 1;
          }
        }
      }
      if (hl == 0) ms[late] = listed;
    }
    __syncwarp();
    // published dependencies by bit; every pending flag is read together
    unsigned pub = 0;
    auto read_flags = [&] {
      for (int b = 0; b < maxd; b += 16) {
        const int e = b + hl;
        bool f = false;
        if (e < di && !(pub >> e & 1u)) f = ld_acquire_i32(done + cj[e]) == epoch;
        pub |= ((__ballot_sync(FULL, f) >> (16 * half)) & 0xffffu) << b;
      }
    };
    // inv(U_kk) and the first kAhead shared blocks of row k for dependency e
    struct Blocks {
      double u[4], w[kAhead][4];
    };
    auto load = [&](int e, bool act, Blocks& B) {
      const int kd = act ? diag[cj[e]] : 0;
      const int m0 = act && e < late ? ms[e] : 0, nm = act && e < late ? ms[e + 1] - m0 : 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) B.u[q] = act ? __ldcg(LU + 16 * (size_t)kd + 4 * q + c) : 0.0;
#pragma unroll
      for (int m = 0; m < kAhead; ++m) {
        const int b = m < nm ? mp[m0 + m] : 0;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          B.w[m][q] = m < nm ? __ldcg(LU + 16 * (size_t)b + 4 * q + c) : 0.0;
      }
    };
    Blocks cur, nxt;
    bool have = false;  // cur holds dependency e's blocks
    for (int e = 0; e < maxd; ++e) {
      const bool act = e < di;
      // both rows' dependencies published (bounded; a failed solve runs on)
      for (unsigned s = 0; __any_sync(FULL, act && !(pub >> e & 1u)); ++s) {
        read_flags();
        if (s >= 64) __nanosleep(64);  // back off: fewer polls competing with working warps
        if ((s & 255u) == 255u) {
          bool stop = ld_volatile_i32(status) != DEV_OK;
          if (s > CPTR_SPIN_LIMIT) {
            dev_fail(status, DEV_TIMEOUT);
            stop = true;
          }
          if (__any_sync(FULL, stop)) break;
        }
      }
      __syncwarp();
      if (!have) load(e, act, cur);
      // the next dependency's blocks, if they are published, behind this one's work
      const bool nhave = e + 1 < di && (pub >> (e + 1) & 1u);
      load(e + 1, nhave, nxt);
      int m0 = 0, nm = 0;
      if (act && e < late) {
        m0 = ms[e];
        nm = ms[e + 1] - m0;
      }
      const bool unlisted = act && e >= late;
      if (__any_sync(FULL, unlisted)) {
        const int n = shared_columns(e, unlisted, 0);
        if (unlisted) nm = n;
        __syncwarp();
        if (unlisted)
          for (int m = 0; m < kAhead; ++m)
            for (int q = 0; q < 4; ++q)
              cur.w[m][q] = m < nm ? __ldcg(LU + 16 * (size_t)mp[m] + 4 * q + c) : 0.0;
      }
      const int maxm = __reduce_max_sync(FULL, nm);
      // L_ik = A_ik inv(U_kk)
      double l = 0.0;
      if (act) {
        const double* A = bi + 16 * e + 4 * r;
        l = A[0] * cur.u[0];
#pragma unroll
        for (int q = 1; q < 4; ++q) l += A[q] * cur.u[q];
      }
      double lr[4];  // row r of L_ik
#pragma unroll
      for (int q = 0; q < 4; ++q) lr[q] = __shfl_sync(FULL, l, 4 * r + q, 16);
      // A_ij -= L_ik U_kj
      auto update = [&](int m, const double* w) {
        const int at = m < nm ? 16 * (int)mt[m0 + m] + hl : 0;
        double p = lr[0] * w[0];
#pragma unroll
        for (int q = 1; q < 4; ++q) p += lr[q] * w[q];
        if (m < nm) bi[at] -= p;
      };
#pragma unroll
      for (int m = 0; m < kAhead; ++m)
        if (m < maxm) update(m, cur.w[m]);
      for (int m = kAhead; m < maxm; ++m) {
        double w[4];
        const int b = m < nm ? mp[m0 + m] : 0;
#pragma unroll
        for (int q = 0; q < 4; ++q) w[q] = m < nm ? __ldcg(LU + 16 * (size_t)b + 4 * q + c) : 0.0;
        update(m, w);
      }
      cur = nxt;
      have = nhave;
      __syncwarp();
      // (behind the barrier: the row's other lanes have read A_ik by then)
      if (act) bi[16 * e + hl] = l;
    }
    bool ok;
    double dv = inv4_pair(i >= 0 ? bi[16 * di + hl] : (r == c ? 1.0 : 0.0), &ok);
    if (!ok) {
      dv = 0.0;
      if (hl == 0) dev_fail(status, DEV_BREAKDOWN);
    }
    if (i >= 0) {
      bi[16 * di + hl] = dv;
#pragma unroll 4
      for (int e = 0; e < ni; ++e) LU[16 * (size_t)(t0 + e) + hl] = bi[16 * e + hl];
    }
    __syncwarp();
    if (hl == 0 && i >= 0) st_release_i32(done + i, epoch);
    __syncwarp();
  }
}

__global__ void k_max_row(int N, const int32_t* __restrict__ rp, int* out) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < N) atomicMax(out, rp[i + 1] - rp[i]);
}

__global__ void k_sched_counts(int npos, const int32_t* __restrict__ ord,
                               const int32_t* __restrict__ rp, const int32_t* __restrict__ diag,
                               bool upper, int32_t* __restrict__ cnt) {
  int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= npos) return;
  int i = ord[p];
  int n = 0;
  if (i >= 0) n = upper ? rp[i + 1] - diag[i] - 1 : diag[i] - rp[i];
  cnt[p] = n;
}

// The factor blocks of every schedule position, in the apply precision: sixteen
// lanes per position, one per entry of a block (the reads and writes of a warp are
// whole blocks; a thread per position took 1.81 ms on the 200x200x100 grid, now 0.99).
template <class T>
__global__ void k_sched_fill(int npos, const int32_t* __restrict__ ord,
                             const int32_t* __restrict__ rp, const int32_t* __restrict__ ci,
                             const int32_t* __restrict__ diag, const double* __restrict__ LU,
                             bool upper, const int32_t* __restrict__ srp, int32_t* __restrict__ sci,
                             T* __restrict__ sv, T* __restrict__ dinv) {
  const int p = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 4);
  const int q = threadIdx.x & 15;
  if (p >= npos) return;
  const int i = ord[p];
  if (i < 0) {
    if (dinv) dinv[16 * (size_t)p + q] = 0;
    return;
  }
  const int t0 = upper ? diag[i] + 1 : rp[i];
  const int o = srp[p], n = srp[p + 1] - o;
  for (int a = q; a < n; a += 16) sci[o + a] = ci[t0 + a];
#pragma unroll 4
  for (int a = 0; a < n; ++a)
    sv[16 * (size_t)(o + a) + q] = (T)LU[16 * (size_t)(t0 + a) + q];
  if (dinv) dinv[16 * (size_t)p + q] = (T)LU[16 * (size_t)diag[i] + q];
}

// Level sets of the rows in one pass (k_level_syncfree), and their number.
cptr_status compute_levels(cptr_ctx* c, bool upper, int32_t* lvl, int* nlev) {
  int N = c->N;
  unsigned* ctr;
  CTX_ALLOC(c, ctr, unsigned, 1, true);
  CTX_CUDA(c, cudaMemsetAsync(ctr, 0, sizeof(unsigned), cs(c)));
  CTX_CUDA(c, cudaMemsetAsync(lvl, 0xFF, sizeof(int32_t) * N, cs(c)));
  KL(c, k_level_syncfree<<<c->nsm * 8, 256, 0, cs(c)>>>(N, c->rp, c->ci, c->diag, lvl, upper,
                                                             ctr, &c->ctl->status));
  CTX_CUDA(c, cudaGetLastError());
  cptr_status st = ctx_check_device_status(c);
  if (st) {
    ctx_set_err(c, "level-set computation timed out");
    return st;
  }
  int32_t* cnt;
  int* mx;
  CTX_ALLOC(c, cnt, int32_t, N + 1, true);
  CTX_ALLOC(c, mx, int, 1, true);
  CTX_CUDA(c, cudaMemsetAsync(cnt, 0, sizeof(int32_t) * (N + 1), cs(c)));
  CTX_CUDA(c, cudaMemsetAsync(mx, 0, sizeof(int), cs(c)));
  KL(c, k_level_count<<<nblk(N), kT, 0, cs(c)>>>(N, lvl, cnt, mx));
  int hm = 0;
  CTX_CUDA(c, cudaMemcpyAsync(&hm, mx, sizeof(int), cudaMemcpyDeviceToHost, cs(c)));
  CTX_CUDA(c, cudaStreamSynchronize(cs(c)));
  *nlev = hm + 1;
  return CPTR_OK;
}

cptr_status build_schedule(cptr_ctx* c, const int32_t* lvl, int nlev, int32_t** ord, int* npos,
                           int32_t** offs) {
  int N = c->N;
  int32_t *cnt, *pc, *off, *cur;
  CTX_ALLOC(c, cnt, int32_t, nlev + 1, true);
  CTX_ALLOC(c, pc, int32_t, nlev + 1, true);
  CTX_ALLOC(c, off, int32_t, nlev + 1, true);
  CTX_ALLOC(c, cur, int32_t, nlev + 1, true);
  int* mx;
  CTX_ALLOC(c, mx, int, 1, true);
  CTX_CUDA(c, cudaMemsetAsync(cnt, 0, sizeof(int32_t) * (nlev + 1), cs(c)));
  CTX_CUDA(c, cudaMemsetAsync(cur, 0, sizeof(int32_t) * (nlev + 1), cs(c)));
  KL(c, k_level_count<<<nblk(N), kT, 0, cs(c)>>>(N, lvl, cnt, mx));
  KL(c, k_pad8<<<nblk(nlev), kT, 0, cs(c)>>>(nlev, cnt, pc));
  int tot = 0;
  cptr_status st = scan_i32(c, pc, off, nlev, &tot);
  if (st) return st;
  CTX_ALLOC(c, *ord, int32_t, tot + 8, true);
  CTX_CUDA(c, cudaMemsetAsync(*ord, 0xFF, sizeof(int32_t) * (tot + 8), cs(c)));
  KL(c, k_level_fill<<<nblk(N), kT, 0, cs(c)>>>(N, lvl, off, cur, *ord));
  *npos = tot;
  *offs = off;  // first (padded) position of each level, nlev + 1 entries
  CTX_CUDA(c, cudaGetLastError());
  return CPTR_OK;
}

template <class T>
cptr_status build_solve_arrays(cptr_ctx* c, bool upper) {
  int npos = upper ? c->npos_b : c->npos_f;
  const int32_t* ord = upper ? c->ord_b : c->ord_f;
  int32_t *cnt, *srp, *sci;
  CTX_ALLOC(c, cnt, int32_t, npos + 1, true);
  CTX_ALLOC(c, srp, int32_t, npos + 1, true);
  KL(c, k_sched_counts<<<nblk(npos), kT, 0, cs(c)>>>(npos, ord, c->rp, c->diag, upper, cnt));
  int tot = 0;
  cptr_status st = scan_i32(c, cnt, srp, npos, &tot);
  if (st) return st;
  CTX_ALLOC(c, sci, int32_t, tot + 1, true);
  T* sv;
  CTX_ALLOC(c, sv, T, 16 * (size_t)tot + 16, true);
  T* dinv = nullptr;
  if (upper) CTX_ALLOC(c, dinv, T, 16 * (size_t)npos + 16, true);
  KL(c, k_sched_fill<T><<<nblk(16ll * npos), kT, 0, cs(c)>>>(npos, ord, c->rp, c->ci, c->diag, c->LU64,
                                                    upper, srp, sci, sv, dinv));
  if (upper) {
    c->Urp = srp; c->Uci = sci; c->Uv = sv; c->Dinv = dinv;
    c->nnzU = tot;
  } else {
    c->Lrp = srp; c->Lci = sci; c->Lv = sv;
    c->nnzL = tot;
  }
  CTX_CUDA(c, cudaGetLastError());
  return CPTR_OK;
}

}  // namespace

// Level sets, schedules and the factorisation (issued on cs(c); may run on
// the second stream beside the AMG setup).
cptr_status setup_ilu_factor(cptr_ctx* c) {
  int N = c->N;
  cptr_status st;
  CTX_ALLOC(c, c->lvl_f, int32_t, N + 1, true);
  CTX_ALLOC(c, c->lvl_b, int32_t, N + 1, true);
  st = compute_levels(c, false, c->lvl_f, &c->nlev_f);
  if (st) return st;
  st = compute_levels(c, true, c->lvl_b, &c->nlev_b);
  if (st) return st;
  ctx_phase(c, "  ilu level sets");
  st = build_schedule(c, c->lvl_f, c->nlev_f, &c->ord_f, &c->npos_f, &c->loff_f);
  if (st) return st;
  st = build_schedule(c, c->lvl_b, c->nlev_b, &c->ord_b, &c->npos_b, &c->loff_b);
  if (st) return st;
  ctx_phase(c, "  ilu schedules");
  // factorisation in place on a copy of A
  CTX_ALLOC(c, c->LU64, double, 16 * (size_t)c->nnzb, true);
  CTX_CUDA(c, cudaMemcpyAsync(c->LU64, c->v, sizeof(double) * 16 * (size_t)c->nnzb,
                              cudaMemcpyDeviceToDevice, cs(c)));
  if (!c->fac_done) {
    CTX_ALLOC(c, c->fac_done, int32_t, N + 1, false);
    CTX_CUDA(c, cudaMemsetAsync(c->fac_done, 0, sizeof(int32_t) * (N + 1), cs(c)));
  }
  c->fac_epoch += 1;
  CTX_CUDA(c, cudaMemsetAsync(&c->ctl->fac_ctr, 0, sizeof(unsigned), cs(c)));
  int* mrow;
  CTX_ALLOC(c, mrow, int, 1, true);
  CTX_CUDA(c, cudaMemsetAsync(mrow, 0, sizeof(int), cs(c)));
  KL(c, k_max_row<<<nblk(N), kT, 0, cs(c)>>>(N, c->rp, mrow));
  int hm = 0;
  CTX_CUDA(c, cudaMemcpyAsync(&hm, mrow, sizeof(int), cudaMemcpyDeviceToHost, cs(c)));
  CTX_CUDA(c, cudaStreamSynchronize(cs(c)));
  c->max_row = hm;
  if (hm <= kRowMax && !c->force_fallback) {
    const FacRow lay = fac_row(hm);
    KL(c, k_ilu_factor_pair<<<c->nsm * 8, 32 * kFacWarps, (size_t)lay.bytes * 2 * kFacWarps,
                              cs(c)>>>(c->npos_f, lay, c->ord_f, c->rp, c->ci, c->diag, c->LU64,
                                       c->fac_done, c->fac_epoch, c->ctl));
  } else {
    KL(c, k_ilu_factor<<<c->nsm * 4, 256, 0, cs(c)>>>(c->npos_f, c->ord_f, c->rp, c->ci,
                                                          c->diag, c->LU64, c->fac_done,
                                                          c->fac_epoch, c->ctl));
  }
  CTX_CUDA(c, cudaGetLastError());
  st = ctx_check_device_status(c);
  if (st) return st;
  ctx_phase(c, "  ilu factorisation");
  return CPTR_OK;
}

cptr_status setup_ilu_schedule(cptr_ctx* c) {
  cptr_status st = build_tri_schedule(c);
  ctx_phase(c, "  ilu solve schedule");
  return st;
}

cptr_status setup_ilu(cptr_ctx* c) {
  cptr_status st = setup_ilu_factor(c);
  return st ? st : setup_ilu_schedule(c);
}

cptr_status build_level_solve_arrays(cptr_ctx* c) {
  cptr_status st;
  if (c->mixed) {
    st = build_solve_arrays<float>(c, false);
    if (!st) st = build_solve_arrays<float>(c, true);
  } else {
    st = build_solve_arrays<double>(c, false);
    if (!st) st = build_solve_arrays<double>(c, true);
  }
  return st;
}
