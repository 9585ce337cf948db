// Row accumulators of the setup's sparse products C = A B (included by
// setup_amg.cu, compiled with -fmad=false).
//
// Every row of C is accumulated in a small open-addressing hash table in shared
// memory, keyed by column: the products a_ik b_kj are taken in the order of the
// entries of A (then of B's row k), and a column's sum starts at 0.0 and adds
// its products in that order, so the results equal the sequential definition
// bit for bit.  The row's columns are then sorted and written to the row's slot.
//
// What binds these kernels is the latency of the gathers of B and the number of
// instructions per product, with the FP64 add and multiply at GB300's narrow
// rate (an FP64 instruction costs the same for one lane as for 32); so a table
// belongs to one warp or to part of one, no block barrier is involved, and the
// lanes are filled:
//  - acc_group: four lanes per row, eight rows per warp in lockstep, for rows of
//    few columns and a B of short rows (P: at most pmax entries): one A entry
//    per step;
//  - acc_flat: one warp per row; 32 consecutive products of the row per step,
//    whatever the lengths of B's rows; equal columns inside a step are added in
//    lane order;
//  - acc_big: one block per row of thousands of columns; every warp walks all
//    products and accumulates the columns it owns.
// Rows are binned by their product count (acc_class) into classes with tables of
// 64 to 2,048 slots a warp and 256 for each of a block's 32 warps; a row whose columns do
// not fit goes to the next class, and in the end to k_spgemm_row.
//
// On the 200x200x100 grid the products of one setup take 56 ms (128 ms with a block
// per row and barriers between its phases), on the 1M-point cloud 17 ms (45 ms).
// One warp for a whole row beat lane groups from 128 columns on (level 1's A P,
// 2.2M rows of 184 products: 13.5 ms with four lanes per row, 5 ms with 32).

constexpr int kAccClasses = 7;  // tables of 64 << class slots, the last one acc_big's
constexpr int kAccBig = kAccClasses - 1;
constexpr int kBigWarps = 32, kBigH = 256;  // acc_big: slots per warp

// Largest product count a class starts with.  The distinct columns grow more
// slowly than the products (measured on the hierarchies of 7-point grids and
// neighbour clouds: 1.4 T^0.7 on average); a class takes the rows whose
// estimate fills at most three quarters of its table.
__host__ __device__ inline int acc_class(long long t) {
  return t <= 96 ? 0 : t <= 300 ? 1 : t <= 800 ? 2 : t <= 2200 ? 3 : t <= 6000 ? 4
         : t <= 16000 ? 5 : 6;
}

// Row lists of the classes: list k holds its rows at rows[k * n ...], ncls[k] of
// them; list kAccClasses takes the rows that fit no class.  all = k: class k
// works on all n rows instead of its list (-1: none does).
struct AccArgs {
  int n;
  const int32_t *arp, *aci;
  const double* av;
  const int32_t *brp, *bci;
  const double* bv;
  const long long* toff;  // first entry of each row's slot
  int32_t* cci;
  double* cv;
  int32_t* cnt;   // columns of each row
  int32_t* rows;
  int* ncls;
  int all;
};
__device__ __forceinline__ int acc_rows(const AccArgs& a, int cls) {
  return a.all == cls ? a.n : a.ncls[cls];
}
__device__ __forceinline__ int acc_row(const AccArgs& a, int cls, int q) {
  return a.all == cls ? q : a.rows[(size_t)cls * a.n + q];
}

__device__ __forceinline__ void acc_defer(const AccArgs& a, int cls, int row) {
  if (cls + 1 == kAccClasses) a.cnt[row] = -1;  // for the global-scratch kernel
  a.rows[(size_t)(cls + 1) * a.n + atomicAdd(&a.ncls[cls + 1], 1)] = row;
}

// Bins the rows by class: prods[i] = products of row i (force >= 0: all rows into
// that class).
__global__ void k_acc_bin(AccArgs a, const int32_t* __restrict__ prods, int force) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
  const int k = i >= a.n ? -1 : force >= 0 ? force : acc_class(prods[i]);
  const unsigned same = __match_any_sync(0xffffffffu, k);
  int base = 0;
  if (k >= 0 && lane == __ffs(same) - 1) base = atomicAdd(&a.ncls[k], __popc(same));
  base = __shfl_sync(0xffffffffu, base, __ffs(same) - 1);
  if (k >= 0) a.rows[(size_t)k * a.n + base + __popc(same & ((1u << lane) - 1u))] = i;
}

// Slot of `col` in the table (inserted when absent), or -1 when the table is
// full, which a longer probe sequence than any useful load factor gives counts
// as; *fresh: this call inserted it.  The columns that lanes insert at the same
// time are distinct.
template <int H>
__device__ __forceinline__ int acc_slot(int* key, int col, bool* fresh) {
  unsigned h = ((unsigned)col * 2654435761u) & (H - 1);
  *fresh = false;
  for (int p = 0; p < (H < 64 ? H : 64); ++p) {
    // (compare-and-swap at once: a read first and a swap only when empty makes
    // two paths, which a warp walks one after the other)
    const int k = atomicCAS(&key[h], -1, col);
    *fresh = k == -1;
    if (k == -1 || k == col) return (int)h;
    h = (h + 1u) & (H - 1);
  }
  return -1;
}
// Slot of a column the table holds.
template <int H>
__device__ __forceinline__ int acc_find(const int* key, int col) {
  unsigned h = ((unsigned)col * 2654435761u) & (H - 1);
  while (key[h] != col) h = (h + 1u) & (H - 1);
  return (int)h;
}

// Sorts 32 * NPL integers held NPL per lane (a bitonic network; lane l ends
// with the elements l * NPL ... of the sorted sequence).
template <int NPL>
__device__ __forceinline__ void warp_sort(int* x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 2; k <= 32 * NPL; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= NPL) {  // partner in another lane
        const int lj = j / NPL;
        const bool low = (lane & lj) == 0;
#pragma unroll
        for (int q = 0; q < NPL; ++q) {
          const int o = __shfl_xor_sync(0xffffffffu, x[q], lj);
          const bool up = ((lane * NPL + q) & k) == 0;
          x[q] = (low == up) ? min(x[q], o) : max(x[q], o);
        }
      } else {
#pragma unroll
        for (int q = 0; q < NPL; ++q)
          if ((q & j) == 0) {
            const bool up = ((lane * NPL + q) & k) == 0;
            const int a = x[q], b = x[q | j];
            x[q] = up ? min(a, b) : max(a, b);
            x[q | j] = up ? max(a, b) : min(a, b);
          }
      }
    }
  }
}

// Sorts lst[0..u) in place with the whole warp, u <= 32 * NPL.
template <int NPL>
__device__ __forceinline__ void sort_list_as(int* lst, int u) {
  const int lane = threadIdx.x & 31;
  int x[NPL];
#pragma unroll
  for (int q = 0; q < NPL; ++q) {
    const int p = q * 32 + lane;
    x[q] = p < u ? lst[p] : 0x7fffffff;
  }
  __syncwarp();
  warp_sort<NPL>(x);
#pragma unroll
  for (int q = 0; q < NPL; ++q) {
    const int p = lane * NPL + q;
    if (p < u) lst[p] = x[q];
  }
  __syncwarp();
}
template <int MAXN>
__device__ __forceinline__ void sort_list(int* lst, int u) {
  if (MAXN <= 32 || u <= 32) { sort_list_as<1>(lst, u); return; }
  if constexpr (MAXN > 32) { if (MAXN <= 64 || u <= 64) { sort_list_as<2>(lst, u); return; } }
  if constexpr (MAXN > 64) { if (MAXN <= 128 || u <= 128) { sort_list_as<4>(lst, u); return; } }
  if constexpr (MAXN > 128) { if (MAXN <= 256 || u <= 256) { sort_list_as<8>(lst, u); return; } }
  if constexpr (MAXN > 256) { if (MAXN <= 512 || u <= 512) { sort_list_as<16>(lst, u); return; } }
  if constexpr (MAXN > 512) { if (MAXN <= 1024 || u <= 1024) { sort_list_as<32>(lst, u); return; } }
  if constexpr (MAXN > 1024) sort_list_as<64>(lst, u);
}

// The occupied keys of a table, compacted by the whole warp; returns their number.
template <int H>
__device__ __forceinline__ int compact_keys(const int* key, int* lst) {
  const int lane = threadIdx.x & 31;
  int u = 0;
#pragma unroll 4
  for (int h = lane; h < H; h += 32) {
    const int k = key[h];
    const unsigned m = __ballot_sync(0xffffffffu, k != -1);
    if (k != -1) lst[u + __popc(m & ((1u << lane) - 1u))] = k;
    u += __popc(m);
  }
  __syncwarp();
  return u;
}

// Sorted row: columns and sums of the table to the row's slot.
template <int H>
__device__ __forceinline__ void write_row(const AccArgs& a, int row, int u, const int* key,
                                          const double* val, const int* lst) {
  const int lane = threadIdx.x & 31;
  const long long o = a.toff[row];
  for (int p = lane; p < u; p += 32) {
    const int k = lst[p];
    a.cci[o + p] = k;
    a.cv[o + p] = val[acc_find<H>(key, k)];
  }
  if (lane == 0) a.cnt[row] = u;
}

// Shared memory of one table: H sums, H keys, H list entries.
template <int H>
constexpr size_t acc_table_bytes() { return (size_t)H * 16; }

constexpr int kAccThreads = 128;

// G lanes per row, one A entry per step; the warp's rows advance in lockstep so
// that its instructions serve all of them.
template <int G, int H>
__global__ void __launch_bounds__(kAccThreads, 3) k_acc_group(AccArgs a, int cls, int from) {
  extern __shared__ __align__(16) unsigned char acc_sm[];
  constexpr int R = kAccThreads / G, RW = 32 / G;  // rows per block and per warp
  const int lane = threadIdx.x & 31, gl = lane & (G - 1), grp = threadIdx.x / G;
  double* const val0 = reinterpret_cast<double*>(acc_sm);
  int* const key0 = reinterpret_cast<int*>(val0 + (size_t)R * H);
  int* const lst0 = key0 + (size_t)R * H;
  double* val = val0 + (size_t)grp * H;
  int* key = key0 + (size_t)grp * H;
  const int total = acc_rows(a, cls);
  for (int q0 = from + blockIdx.x * R + (int)(threadIdx.x >> 5) * RW; q0 < total;
       q0 += gridDim.x * R) {
    const int q = q0 + lane / G;
    const int row = q < total ? acc_row(a, cls, q) : -1;
    const int t0 = row >= 0 ? a.arp[row] : 0, na = row >= 0 ? a.arp[row + 1] - t0 : 0;
    for (int h = gl; h < H; h += G) key[h] = -1;
    __syncwarp();
    bool bad = false;
    const int most = __reduce_max_sync(0xffffffffu, na);
    for (int base = 0; base < most; base += G) {
      int bs = 0, bl = 0;
      double av = 0.0;
      if (base + gl < na) {
        const int k = a.aci[t0 + base + gl];
        av = a.av[t0 + base + gl];
        bs = a.brp[k];
        bl = a.brp[k + 1] - bs;
      }
      // the first chunk of each of the G steps' B rows, loaded together
      int s[G], l[G], col[G];
      double b[G];
#pragma unroll
      for (int u = 0; u < G; ++u) {
        s[u] = __shfl_sync(0xffffffffu, bs, u, G) + gl;
        l[u] = __shfl_sync(0xffffffffu, bl, u, G) - gl;  // > 0: this lane has an entry
        if (l[u] > 0) { col[u] = a.bci[s[u]]; b[u] = a.bv[s[u]]; }
      }
#pragma unroll
      for (int u = 0; u < G; ++u) {
        const double x = __shfl_sync(0xffffffffu, av, u, G);
        while (__any_sync(0xffffffffu, l[u] > 0)) {
          if (l[u] > 0) {
            bool fresh;
            const int h = acc_slot<H>(key, col[u], &fresh);
            if (h < 0) {
              bad = true;
            } else {
              const double prod = x * b[u];
              val[h] = (fresh ? 0.0 : val[h]) + prod;
            }
          }
          __syncwarp();
          l[u] -= G;
          s[u] += G;
          if (l[u] > 0) { col[u] = a.bci[s[u]]; b[u] = a.bv[s[u]]; }
        }
      }
    }
    // the rows of the warp, one after the other, with all lanes
    const unsigned badm = __ballot_sync(0xffffffffu, bad);
#pragma unroll 1
    for (int w = 0; w < RW; ++w) {
      const int rw = __shfl_sync(0xffffffffu, row, w * G);
      if (rw < 0) continue;
      if (badm >> (w * G) & ((1ull << G) - 1)) {
        if (lane == 0) acc_defer(a, cls, rw);
        continue;
      }
      const size_t at = (size_t)((threadIdx.x >> 5) * RW + w) * H;
      const int u = compact_keys<H>(key0 + at, lst0 + at);
      sort_list<H>(lst0 + at, u);
      write_row<H>(a, rw, u, key0 + at, val0 + at, lst0 + at);
    }
    __syncwarp();
  }
}

// One step of a warp-wide walk over a row's products, 32 at a time in product
// order: fetch(col, prod) for lanes with a product.  OWN: only the columns for
// which own(col) holds are accumulated.  Returns false when the table is full.
template <int H, class Own>
__device__ __forceinline__ bool acc_walk(const AccArgs& a, int t0, int na, int* key, double* val,
                                         Own own) {
  const int lane = threadIdx.x & 31;
  bool bad = false;
  for (int base = 0; base < na; base += 32) {
    int bs = 0, bl = 0;
    double av = 0.0;
    if (base + lane < na) {
      const int k = a.aci[t0 + base + lane];
      av = a.av[t0 + base + lane];
      bs = a.brp[k];
      bl = a.brp[k + 1] - bs;
    }
    int end = bl;  // products up to and including this lane's A entry
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, end, o);
      if (lane >= o) end += y;
    }
    const int total = __shfl_sync(0xffffffffu, end, 31);
    bs -= end - bl;  // product p of A entry e is B's entry bs_e + p
    // A entry of product p: the number of entries that end at or before p
    auto load = [&](int p, int& col, double& b, int& e) {
      e = 0;
#pragma unroll
      for (int step = 16; step > 0; step >>= 1) {
        const int en = __shfl_sync(0xffffffffu, end, e + step - 1);
        if (en <= p) e += step;
      }
      e = min(e, 31);
      const int src = __shfl_sync(0xffffffffu, bs, e) + p;
      col = -1;
      b = 0.0;
      if (p < total) { col = a.bci[src]; b = a.bv[src]; }
    };
    int col, e, coln = -1, en = 0;
    double b, bn = 0.0;
    load(lane, col, b, e);
    for (int p0 = 0; p0 < total; p0 += 32) {
      if (p0 + 32 < total) load(p0 + 32 + lane, coln, bn, en);
      const double prod = __shfl_sync(0xffffffffu, av, e) * b;
      const bool act = col >= 0 && own(col);
      // equal columns can only meet inside a step that spans several A entries
      const int e0 = __shfl_sync(0xffffffffu, e, 0);
      int rank = 0, first = lane;
      if (__any_sync(0xffffffffu, col >= 0 && e != e0)) {
        const unsigned same = __match_any_sync(0xffffffffu, col);
        rank = __popc(same & ((1u << lane) - 1u));
        first = __ffs(same) - 1;
      }
      // the lane of a column's first product finds its slot, the others take it
      int h = -2;
      bool fresh = false;
      if (act && rank == 0) {
        h = acc_slot<H>(key, col, &fresh);
        if (h < 0) bad = true;
        else val[h] = (fresh ? 0.0 : val[h]) + prod;
      }
      h = __shfl_sync(0xffffffffu, h, first);
      for (int r = 1; __any_sync(0xffffffffu, act && rank >= r); ++r) {
        __syncwarp();
        if (act && rank == r && h >= 0) val[h] += prod;
      }
      if (__any_sync(0xffffffffu, bad)) return false;
      // the keys and sums of this step before the next one's, or before the caller
      // reads the table: shuffles and votes do not order shared memory
      __syncwarp();
      col = coln; b = bn; e = en;
    }
  }
  return true;
}

template <int H>  // (as many blocks resident as their tables allow)
__global__ void __launch_bounds__(kAccThreads, H <= 512 ? 6 : H <= 1024 ? 3 : 1) k_acc_flat(AccArgs a, int cls, int from) {
  extern __shared__ __align__(16) unsigned char acc_sm[];
  constexpr int R = kAccThreads / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double* val = reinterpret_cast<double*>(acc_sm) + (size_t)warp * H;
  int* key = reinterpret_cast<int*>(acc_sm + (size_t)R * H * 8) + (size_t)warp * H;
  int* lst = reinterpret_cast<int*>(acc_sm + (size_t)R * H * 12) + (size_t)warp * H;
  const int total = acc_rows(a, cls);
  for (int q = from + blockIdx.x * R + warp; q < total; q += gridDim.x * R) {
    const int row = acc_row(a, cls, q), t0 = a.arp[row], na = a.arp[row + 1] - t0;
    for (int h = lane; h < H; h += 32) key[h] = -1;
    __syncwarp();
    if (!acc_walk<H>(a, t0, na, key, val, [](int) { return true; })) {
      if (lane == 0) acc_defer(a, cls, row);
      __syncwarp();
      continue;
    }
    const int u = compact_keys<H>(key, lst);
    sort_list<H>(lst, u);
    write_row<H>(a, row, u, key, val, lst);
    __syncwarp();
  }
}

// One block per row of up to kBigWarps * kBigH columns: warp w owns the columns
// whose hash names it and accumulates them in a table of its own.
constexpr int kBigCols = kBigWarps * kBigH;
__device__ __forceinline__ int big_owner(int col) {
  return (int)(((unsigned)col * 0x9E3779B1u) >> 27);
}
static_assert(kBigWarps == 32, "big_owner names 32 warps");
__global__ void __launch_bounds__(32 * kBigWarps) k_acc_big(AccArgs a, int from) {
  extern __shared__ __align__(16) unsigned char acc_sm[];
  __shared__ int s_n, s_bad;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double* val = reinterpret_cast<double*>(acc_sm) + (size_t)warp * kBigH;
  int* key = reinterpret_cast<int*>(acc_sm + (size_t)kBigCols * 8) + (size_t)warp * kBigH;
  int* lst = reinterpret_cast<int*>(acc_sm + (size_t)kBigCols * 12);  // the block's columns
  const int total = acc_rows(a, kAccBig);
  for (int q = from + blockIdx.x; q < total; q += gridDim.x) {
    const int row = acc_row(a, kAccBig, q), t0 = a.arp[row], na = a.arp[row + 1] - t0;
    if (threadIdx.x == 0) s_n = s_bad = 0;
    for (int h = lane; h < kBigH; h += 32) key[h] = -1;
    __syncthreads();
    if (!acc_walk<kBigH>(a, t0, na, key, val, [warp](int c) { return big_owner(c) == warp; }) &&
        lane == 0)
      s_bad = 1;
    __syncthreads();
    if (s_bad) {
      if (threadIdx.x == 0) acc_defer(a, kAccBig, row);
      __syncthreads();
      continue;
    }
    // all columns to one list, sorted by the block
    for (int h = lane; h < kBigH; h += 32) {
      const int k = key[h];
      const unsigned m = __ballot_sync(0xffffffffu, k != -1);
      int at = 0;
      if (lane == 0 && m) at = atomicAdd(&s_n, __popc(m));
      at = __shfl_sync(0xffffffffu, at, 0);
      if (k != -1) lst[at + __popc(m & ((1u << lane) - 1u))] = k;
    }
    __syncthreads();
    const int u = s_n;
    int P = 1;
    while (P < u) P <<= 1;
    for (int p = u + (int)threadIdx.x; p < P; p += blockDim.x) lst[p] = 0x7fffffff;
    __syncthreads();
    for (int k = 2; k <= P; k <<= 1)
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int x = threadIdx.x; x < P / 2; x += blockDim.x) {
          const int i = 2 * x - (x & (j - 1)), o = i + j;  // the x-th pair at distance j
          const int v = lst[i], w = lst[o];
          if ((v > w) == ((i & k) == 0)) { lst[i] = w; lst[o] = v; }
        }
        __syncthreads();
      }
    const long long o = a.toff[row];
    const double* val0 = reinterpret_cast<const double*>(acc_sm);
    const int* key0 = reinterpret_cast<const int*>(acc_sm + (size_t)kBigCols * 8);
    for (int p = threadIdx.x; p < u; p += blockDim.x) {
      const int k = lst[p], w = big_owner(k);
      a.cci[o + p] = k;
      a.cv[o + p] = val0[(size_t)w * kBigH + acc_find<kBigH>(key0 + (size_t)w * kBigH, k)];
    }
    if (threadIdx.x == 0) a.cnt[row] = u;
    __syncthreads();
  }
}
