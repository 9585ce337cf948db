// Extended+i rows of P by lane groups (included by setup_amg.cu, compiled with
// -fmad=false): the arithmetic and order of k_interp, bit for bit.
//
// An F point's row is a few dozen terms in ordered sums (the denominators of its
// strong F neighbours, the distribution, the diagonal, the truncation), so what
// binds it is the FP64 issue rate of GB300, where an instruction costs the same
// for one lane as for 32, and the latency of its dependent gathers.  G lanes take
// a row and 32 / G rows advance in lockstep in one warp, so that each FP64
// instruction serves all of them; every set and list is private to a row in
// shared memory, and there is no block barrier.  Ordered sums are split by what
// they sum, never inside: one lane per denominator, terms of equal target added in
// their order, a lane for the diagonal.
//
// A row that does not fit its class (or has a NaN weight, whose selection follows
// the definition's comparisons one by one) goes to the next class and in the end
// to k_interp_row.
//
// On the 200x200x100 grid all levels take 33 ms (129 ms with a block of 128 threads
// per row and barriers between the phases), level 0 (5.1M F points, rows of 14)
// 9.9 ms and level 1 (2.2M, rows of 60) 12.9 ms.  Lanes per row, in ms: level 0
// with 8 / 16 / 32: 10.5 / 9.9 / 15; level 1: 30.8 / 18.2 / 12.9 (rows of uneven
// length in lockstep cost more than shared FP64 instructions save).

// Shared memory of one row.  H: hash slots of Chat, Q: its columns at most, TC:
// terms, KC: strong F neighbours.
template <int H, int Q, int TC, int KC>
struct IxRow {
  double num[Q + 1];   // sums per column of Chat
  double tval[TC];     // diagonal terms of row i, then the neighbours' terms
  double ka[KC];       // a_ik, then the neighbour's term of the diagonal
  double kf[KC];       // a_ik / denominator
  int key[H];
  int list[Q];         // Chat, sorted
  int kst[KC], klen[KC];
  uint16_t pos[H];     // slot -> position in list
  uint16_t tpos[TC], tk[TC];  // target and neighbour of each term
  uint16_t tst[KC + 1];       // first term of each neighbour
};

struct IxArgs {
  int n, pmax;
  const int32_t *rp, *ci;
  const double* v;
  const uint8_t* ef;
  const int32_t* cidx;
  int32_t *pcnt, *pcol;
  double* pval;
  int32_t* rows;  // list k: rows[k * n ...]
  int* ncls;
};
constexpr int kIxClasses = 3;
// class of an F point with ub Chat candidates (repeats counted), nk strong F
// neighbours and a row of len entries; the distinct columns are less than half of
// the candidates on the hierarchies measured
__host__ __device__ inline int ix_class(int ub, int nk, int len) {
  return (nk <= 16 && ub <= 64 && len <= 40) ? 0
         : (nk <= 40 && ub <= 250 && len <= 250) ? 1 : nk <= 128 ? 2 : kIxClasses;
}

__device__ __forceinline__ void ix_defer(const IxArgs& a, int cls, int row) {
  if (cls + 1 == kIxClasses) a.pcnt[row] = -1;
  a.rows[(size_t)(cls + 1) * a.n + atomicAdd(&a.ncls[cls + 1], 1)] = row;
}

// C points get their unit rows; F points are listed by class.  kcnt[i]: strong F
// neighbours.  force >= 0: every F point starts in that class.
__global__ void k_ix_bin(IxArgs a, const int32_t* __restrict__ cf,
                         const int32_t* __restrict__ ub, const int32_t* __restrict__ kcnt,
                         int force) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
  int k = -1;
  if (i < a.n) {
    if (cf[i] == 1) {
      a.pcnt[i] = 1;
      a.pcol[(size_t)i * a.pmax] = a.cidx[i];
      a.pval[(size_t)i * a.pmax] = 1.0;
    } else {
      k = force >= 0 ? force : ix_class(ub[i], kcnt[i], a.rp[i + 1] - a.rp[i]);
      if (k == kIxClasses) a.pcnt[i] = -1;
    }
  }
  const unsigned same = __match_any_sync(0xffffffffu, k);
  int base = 0;
  if (k >= 0 && lane == __ffs(same) - 1) base = atomicAdd(&a.ncls[k], __popc(same));
  base = __shfl_sync(0xffffffffu, base, __ffs(same) - 1);
  if (k >= 0) a.rows[(size_t)k * a.n + base + __popc(same & ((1u << lane) - 1u))] = i;
}

template <int H>
__device__ __forceinline__ bool ix_insert(int* key, int col) {
  unsigned h = ((unsigned)col * 2654435761u) & (H - 1);
  for (int p = 0; p < (H < 64 ? H : 64); ++p) {
    const int k = atomicCAS(&key[h], -1, col);
    if (k == -1 || k == col) return true;
    h = (h + 1u) & (H - 1);
  }
  return false;
}
// position of col in Chat, or -1
template <int H>
__device__ __forceinline__ int ix_find(const int* key, const uint16_t* pos, int col) {
  unsigned h = ((unsigned)col * 2654435761u) & (H - 1);
  for (int p = 0; p < H; ++p) {
    const int k = key[h];
    if (k == col) return pos[h];
    if (k == -1) return -1;
    h = (h + 1u) & (H - 1);
  }
  return -1;
}

template <int G, int H, int Q, int TC, int KC, int WARPS>
__global__ void __launch_bounds__(32 * WARPS) k_interp_group(IxArgs a, int cls, int from) {
  extern __shared__ __align__(16) unsigned char ix_sm[];
  using Row = IxRow<H, Q, TC, KC>;
  static_assert(Q * 6 <= TC * 8, "the unsorted Chat lies in tval");
  constexpr int RW = 32 / G, R = RW * WARPS;
  constexpr unsigned FULL = 0xffffffffu, GM = G == 32 ? FULL : (1u << G) - 1u;
  const int lane = threadIdx.x & 31, gl = lane & (G - 1), sh = lane & ~(G - 1);
  const unsigned below = (1u << gl) - 1u;
  Row& S = reinterpret_cast<Row*>(ix_sm)[threadIdx.x / G];
  int* const tmpk = reinterpret_cast<int*>(S.tval);           // Chat in slot order
  uint16_t* const tmps = reinterpret_cast<uint16_t*>(tmpk + Q);
  // the group's bits of a warp vote
  auto vote = [&](bool p) { return (__ballot_sync(FULL, p) >> sh) & GM; };
  const int total = a.ncls[cls];
  const int32_t* rows = a.rows + (size_t)cls * a.n;
  for (int q0 = from + blockIdx.x * R + (int)(threadIdx.x >> 5) * RW; q0 < total;
       q0 += gridDim.x * R) {
    const int q = q0 + lane / G;
    const int i = q < total ? rows[q] : -1;
    const int t0 = i >= 0 ? a.rp[i] : 0, ni = i >= 0 ? a.rp[i + 1] - t0 : 0;
    const int maxni = __reduce_max_sync(FULL, ni);
    bool bad = false;
    for (int h = gl; h < H; h += G) S.key[h] = -1;
    __syncwarp();
    // ---- row i: strong C neighbours into Chat, strong F neighbours listed
    int K = 0;
    for (int b = 0; b < maxni; b += G) {
      const int e = t0 + b + gl;
      int f = 0, j = 0;
      if (b + gl < ni) {
        f = a.ef[e];
        if (f & IF_S) j = a.ci[e];
      }
      const bool sf = (f & IF_S) && !(f & IF_C);
      const unsigned m = vote(sf);
      if (sf) {
        const int k = K + __popc(m & below);
        if (k < KC) {
          const int s = a.rp[j];
          S.kst[k] = s;
          S.klen[k] = a.rp[j + 1] - s;
          S.ka[k] = a.v[e];
        }
      }
      K += __popc(m);
      if ((f & IF_S) && (f & IF_C) && !ix_insert<H>(S.key, j)) bad = true;
    }
    if (K > KC) { bad = true; K = KC; }
    __syncwarp();
    const int maxK = __reduce_max_sync(FULL, K);
    // ---- the strong C points of the strong F neighbours, four chunks at a time
    for (int k = 0; k < maxK; ++k) {
      const int s = k < K ? S.kst[k] : 0, l = k < K ? S.klen[k] : 0;
      const int maxl = __reduce_max_sync(FULL, l);
      for (int o = 0; o < maxl; o += 4 * G) {
        int f[4], col[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int p = o + u * G + gl;
          f[u] = p < l ? a.ef[s + p] : 0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if ((f[u] & (IF_S | IF_C)) == (IF_S | IF_C)) col[u] = a.ci[s + o + u * G + gl];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if ((f[u] & (IF_S | IF_C)) == (IF_S | IF_C) && !ix_insert<H>(S.key, col[u])) bad = true;
      }
    }
    __syncwarp();
    // ---- Chat sorted
    int nq = 0;
    for (int h = gl; h < H; h += G) {
      const int k = S.key[h];
      const unsigned m = vote(k != -1);
      const int p = nq + __popc(m & below);
      if (k != -1 && p < Q) {
        tmpk[p] = k;
        tmps[p] = (uint16_t)h;
      }
      nq += __popc(m);
    }
    if (vote(bad || nq > Q)) {  // does not fit: the rest of the row is empty work
      bad = true;
      K = nq = 0;
    }
    __syncwarp();
    for (int p = gl; p < nq; p += G) {
      const int k = tmpk[p];
      int r = 0;
      for (int o = 0; o < nq; ++o) r += tmpk[o] < k;
      S.list[r] = k;
      S.pos[tmps[p]] = (uint16_t)r;
      S.num[p] = 0.0;
    }
    __syncwarp();
    // ---- row i again: direct terms into num, diagonal terms to the front of tval
    int D = 0;
    for (int b = 0; b < maxni; b += G) {
      const int e = t0 + b + gl;
      int f = 0;
      bool dg = false;
      if (b + gl < ni) {
        f = a.ef[e];
        if (f & IF_DIAG) {
          dg = true;
        } else if (f & IF_SAME) {
          const int p = nq > 0 ? ix_find<H>(S.key, S.pos, a.ci[e]) : -1;
          if (p >= 0) S.num[p] = 0.0 + a.v[e];
          else dg = !(f & IF_S);
        }
      }
      const unsigned m = vote(dg);
      const int t = D + __popc(m & below);
      if (dg && t < TC) S.tval[t] = a.v[e];
      D += __popc(m);
    }
    if (D > TC) { bad = true; D = TC; }
    // ---- the neighbours' terms: abar_kl for l in Chat u {i}, in row order
    int T = D;
    for (int k = 0; k < maxK; ++k) {
      const int s = k < K ? S.kst[k] : 0, l = k < K ? S.klen[k] : 0;
      if (k < K && gl == 0) S.tst[k] = (uint16_t)T;
      const int maxl = __reduce_max_sync(FULL, l);
      for (int o = 0; o < maxl; o += 2 * G) {
        int f[2], p[2];
        double x[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int w = o + u * G + gl;
          f[u] = w < l ? a.ef[s + w] : 0;
          p[u] = -1;
        }
#pragma unroll
        for (int u = 0; u < 2; ++u)
          if ((f[u] & IF_SAME) && !(f[u] & IF_DIAG)) p[u] = a.ci[s + o + u * G + gl];
#pragma unroll
        for (int u = 0; u < 2; ++u)
          if (p[u] >= 0) p[u] = p[u] == i ? nq : ix_find<H>(S.key, S.pos, p[u]);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          x[u] = 0.0;
          if (p[u] >= 0) x[u] = a.v[s + o + u * G + gl];
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const bool pres = p[u] >= 0 && ((f[u] & IF_NEG) ? d_gt0(x[u]) : d_lt0(x[u]));
          const unsigned m = vote(pres);
          const int t = T + __popc(m & below);
          if (pres && t < TC) {
            S.tval[t] = x[u];
            S.tpos[t] = (uint16_t)p[u];
            S.tk[t] = (uint16_t)k;
          }
          T += __popc(m);
        }
      }
    }
    if (T > TC) { bad = true; T = TC; }
    if (gl == 0) S.tst[K] = (uint16_t)T;
    __syncwarp();
    // ---- one lane per ordered sum: the denominators, and (k = K) the diagonal terms
    double dg0 = 0.0;
    for (int k0 = 0; k0 <= maxK; k0 += G) {
      const int k = k0 + gl;
      int t = 0, te = 0;
      if (k < K) {
        t = min((int)S.tst[k], T);
        te = min((int)S.tst[k + 1], T);
      } else if (k == K) {
        te = D;
      }
      const int len = __reduce_max_sync(FULL, te - t);
      double sum = 0.0;
      for (int o = 0; o < len; ++o)
        if (t + o < te) sum += S.tval[t + o];
      if (k < K) {
        const bool z = d_eq0(sum);
        S.kf[k] = S.ka[k] / sum;
        S.klen[k] = z;  // the connection itself goes to the diagonal
        S.kst[k] = z;   // ka holds a term of the diagonal
      }
      const unsigned m = vote(k == K);
      const double d = __shfl_sync(FULL, sum, sh + (m ? __ffs(m) - 1 : 0));
      if (m) dg0 = d;
    }
    __syncwarp();
    // ---- f_k abar_kl; the term with l = i belongs to the diagonal
    for (int t = D + gl; t < T; t += G) {
      const int k = S.tk[t];
      if (S.klen[k]) {
        S.tpos[t] = 0xffff;
      } else {
        const double x = S.kf[k] * S.tval[t];
        S.tval[t] = x;
        if (S.tpos[t] == nq) {
          S.ka[k] = x;
          S.kst[k] = 1;  // (klen is read by the neighbour's other lanes)
          S.tpos[t] = 0xffff;
        }
      }
    }
    __syncwarp();
    // ---- distribution: terms of equal column are added in their order
    const int maxT = __reduce_max_sync(FULL, T - D);
    for (int b = 0; b < maxT; b += G) {
      const int t = D + b + gl;
      const int p = t < T ? (int)S.tpos[t] : 0xffff;
      const bool act = p != 0xffff;
      const unsigned same = __match_any_sync(FULL, act ? (sh << 16) + p : -1 - lane);
      const int rank = __popc(same & ((1u << lane) - 1u));
      const double x = act ? S.tval[t] : 0.0;
      const int ranks = __reduce_max_sync(FULL, act ? rank : 0);
      for (int r = 0; r <= ranks; ++r) {
        if (act && rank == r) S.num[p] += x;
        __syncwarp();
      }
    }
    // ---- diagonal, then the weights
    double dg = dg0;
    for (int k = 0; k < maxK; ++k)
      if (k < K && S.kst[k]) dg += S.ka[k];
    const bool ok = !(d_eq0(dg) || dmag(dg) >= 0x7ff0000000000000ull) && nq > 0;
    const int cols = ok ? nq : 0;
    const int maxq = __reduce_max_sync(FULL, cols);
    int m = 0;  // nonzero weights, moved to the front
    for (int b = 0; b < maxq; b += G) {
      const int p = b + gl;
      double w = 0.0;
      int col = 0;
      if (p < cols) {
        w = -S.num[p] / dg;
        col = S.list[p];
        if (d_isnan(w)) bad = true;
      }
      const unsigned mm = vote(p < cols && !d_eq0(w));
      __syncwarp();
      if (p < cols && !d_eq0(w)) {
        const int d = m + __popc(mm & below);
        S.list[d] = col;
        S.num[d] = w;
      }
      m += __popc(mm);
      __syncwarp();
    }
    const bool failed = vote(bad) != 0;
    if (failed) m = 0;
    // ---- truncation to the pmax largest |w| (ties: the smaller column)
    const bool cut = m > a.pmax;
    const int maxm = __reduce_max_sync(FULL, cut ? m : 0);
    int kept = 0;
    for (int b = 0; b < maxm; b += G) {
      const int p = b + gl;
      bool keep = false;
      if (cut && p < m) {
        const unsigned long long w = dmag(S.num[p]);
        int r = 0;
        for (int o = 0; o < m; ++o) {
          const unsigned long long x = dmag(S.num[o]);
          r += x > w || (x == w && o < p);
        }
        keep = r < a.pmax;
      }
      const unsigned mm = vote(keep);
      if (keep) S.tpos[kept + __popc(mm & below)] = (uint16_t)p;
      kept += __popc(mm);
    }
    __syncwarp();
    // both sums in index order, on two lanes
    double sum = 0.0;
    for (int o = 0; o < maxm; ++o) {
      const bool all = gl == 0 && cut && o < m, some = gl == 1 && cut && o < kept;
      if (all || some) sum += S.num[all ? o : (int)S.tpos[o]];
    }
    const double sum_all = __shfl_sync(FULL, sum, sh), sum_kept = __shfl_sync(FULL, sum, sh + 1);
    const double scale = d_eq0(sum_kept) ? 1.0 : sum_all / sum_kept;
    if (i >= 0 && !failed) {
      const int cnt = cut ? kept : m;
      for (int p = gl; p < cnt; p += G) {
        const int o = cut ? (int)S.tpos[p] : p;
        a.pcol[(size_t)i * a.pmax + p] = a.cidx[S.list[o]];
        a.pval[(size_t)i * a.pmax + p] = cut ? S.num[o] * scale : S.num[o];
      }
      if (gl == 0) a.pcnt[i] = cnt;
    }
    if (i >= 0 && failed && gl == 0) ix_defer(a, cls, i);
    __syncwarp();
  }
}
