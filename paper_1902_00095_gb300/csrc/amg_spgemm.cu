// Sparse matrix products C = A B of the AMG setup (the Galerkin R (A P)) and
// their numeric-only recomputation on a known pattern.
//
// Row i of C: products a_ik * b_kj in ascending k (row i of A) then ascending
// j (row k of B); each column's sum starts at 0.0 and adds them in that order
// with correctly rounded operations (no FMA): one canonical result whatever
// kernel takes the row.
#include <algorithm>
#include "amg_dev.cuh"
#include "per_device.cuh"

namespace tp {

namespace {

constexpr int kSpFirst = 192;  // products up to which a row starts at the first group class
constexpr int kSpCap = 1024;   // products from which a long row takes the block kernel

// Products whose result has few columns (m <= kDenseCap: the Galerkin
// products of coarse levels): one warp per row accumulates into a dense
// shared-memory row. The entries of row i of A are visited in order and the
// lanes split row k of B (whose columns are distinct), so every column's sum
// still starts at 0.0 and adds its products in ascending k: the canonical
// order. Touched columns are flagged and compacted in column order.
constexpr int kDenseCap = 2048;
constexpr int kDenseWarps = 4;
constexpr size_t kDenseSmem = (size_t)kDenseWarps * kDenseCap * (sizeof(double) + 1);

__global__ void __launch_bounds__(32 * kDenseWarps) k_spgemm_dense(
    int n, int m, const int* __restrict__ Arp, const int* __restrict__ Acol,
    const double* __restrict__ Aval, const int* __restrict__ Brp, const int* __restrict__ Bcol,
    const double* __restrict__ Bval, const int* __restrict__ off, int* __restrict__ ccol,
    double* __restrict__ cval, int* __restrict__ cnt) {
  extern __shared__ double s_dense[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  double* acc = s_dense + (size_t)w * m;
  unsigned char* flg = reinterpret_cast<unsigned char*>(s_dense + (size_t)kDenseWarps * m) +
                       (size_t)w * m;
  for (int i = blockIdx.x * kDenseWarps + w; i < n; i += gridDim.x * kDenseWarps) {
    for (int j = lane; j < m; j += 32) {
      acc[j] = 0.0;
      flg[j] = 0;
    }
    __syncwarp();
    for (int e = Arp[i]; e < Arp[i + 1]; ++e) {
      const int k = Acol[e];
      const double a = Aval[e];
      for (int f = Brp[k] + lane; f < Brp[k + 1]; f += 32) {
        const int j = Bcol[f];
        acc[j] = __dadd_rn(acc[j], __dmul_rn(a, Bval[f]));
        flg[j] = 1;
      }
      __syncwarp();
    }
    int* cc = ccol + off[i];
    double* cv = cval + off[i];
    int base = 0;
    for (int j0 = 0; j0 < m; j0 += 32) {
      const int j = j0 + lane;
      const bool has = j < m && flg[j];
      const unsigned hm = __ballot_sync(0xffffffffu, has);
      if (has) {
        cc[base + __popc(hm & below)] = j;
        cv[base + __popc(hm & below)] = acc[j];
      }
      base += __popc(hm);
    }
    if (lane == 0) cnt[i] = base;
    __syncwarp();
  }
}


// Group-per-row form: G lanes take a row of C, 32 / G rows a warp. The group
// walks row i of A in ascending k and its lanes take the entries of row k of B
// (distinct columns), so no two lanes update one column at once and every
// column's additions stay in ascending k, each sum starting at 0.0: the
// canonical order. A column finds its accumulator through an open-addressing
// hash table of CAP slots in shared memory; G is matched to the rows of B (4
// lanes for P truncated to 4 weights, 8 to 32 for A P), since an FP64
// instruction occupies the FP64 pipe for the whole warp however few lanes take
// part. The table is sized for the row's distinct columns, not its products
// (on the layered A_pp's levels rows of R (A P) have 100-1100 products but
// 30-90 columns): a row of more than MAXU columns is dropped and listed for
// the next class. The groups of a warp stay together (trip counts are the
// warp's largest).
//
// Measured on GB300 (kernel time summed over a setup of the layered 256x256x64
// system, both hierarchies): the four kernels this replaces (a register merge
// and an insertion form by thread, two warp hash tables sized for the products)
// 37 ms, this 21 ms; the step 192.5 -> 186 ms. It is bound by the FP64 pipe
// (59-78 % busy, two instructions per lane step) and by shared-memory latency.
// Twice the lanes for A P (8 for rows of 4) 11.2 instead of 7.7 ms; starting
// rows of 128-192 products at the second class made no difference.
//
// KNOWN: numeric-only on C's pattern (off = C's row pointers, ccol = its
// columns): the row's columns are put into the table first, sums are written
// in place and rows longer than MAXU are listed.
template <int G, int CAP, int MAXU>
struct GroupRows {
  double hval[32 / G][CAP];
  int hkey[32 / G][CAP];
  unsigned short ulist[32 / G][MAXU + G];  // slots in order of arrival
  int cnt[32 / G];
};

template <int G, int CAP, int MAXU, int WARPS, bool KNOWN>
__global__ void __launch_bounds__(32 * WARPS) k_spgemm_group(
    int n, const int* __restrict__ list, const int* __restrict__ nlist, int ub_max,
    const int* __restrict__ Arp, const int* __restrict__ Acol, const double* __restrict__ Aval,
    const int* __restrict__ Brp, const int* __restrict__ Bcol, const double* __restrict__ Bval,
    const int* __restrict__ off, const int* __restrict__ ub, int* __restrict__ ccol,
    double* __restrict__ cval, int* __restrict__ cnt, int* __restrict__ olist,
    int* __restrict__ ocnt, int* __restrict__ blist, int* __restrict__ bcnt) {
  using S = GroupRows<G, CAP, MAXU>;
  static_assert((CAP & (CAP - 1)) == 0 && MAXU + G <= CAP, "table");
  constexpr int NG = 32 / G;
  constexpr unsigned kAll = 0xffffffffu;
  extern __shared__ __align__(16) char smem[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = lane / G, gl = lane % G;
  S& s = reinterpret_cast<S*>(smem)[w];
  double* hval = s.hval[grp];
  int* hkey = s.hkey[grp];
  unsigned short* ulist = s.ulist[grp];
  const int count = list ? *nlist : n;
  const long long step = (long long)gridDim.x * WARPS * NG;
  for (long long base = ((long long)blockIdx.x * WARPS + w) * NG; base < count; base += step) {
    const long long q = base + grp;
    int i = q < count ? (list ? list[q] : (int)q) : -1;
    int a0 = 0, na = 0, c0 = 0, clen = 0;
    bool over = false;
    if (i >= 0) {
      a0 = Arp[i];
      na = Arp[i + 1] - a0;
      c0 = off[i];
      if (KNOWN) {
        clen = off[i + 1] - c0;
        over = clen > MAXU;
      } else if (!list && ub[i] > ub_max) {
        i = -1;  // listed by k_spgemm_ub
      }
      if (i < 0 || over) na = clen = 0;
    }
    const int na_max = __reduce_max_sync(kAll, na);
    if (__any_sync(kAll, i >= 0 && !over)) {
#pragma unroll
      for (int h = gl; h < CAP; h += G) hkey[h] = -1;
      if (gl == 0) s.cnt[grp] = 0;
      __syncwarp();
      // slot of column j (claimed when new), -1 when the table has none
      auto find = [&](int j, bool& fresh) -> int {
        unsigned h = ((unsigned)j * 0x9E3779B1u) >> (32 - __popc(CAP - 1));
        fresh = false;
        for (int p = 0; p < CAP; ++p) {
          const int prev = KNOWN ? hkey[h] : atomicCAS(&hkey[h], -1, j);
          if (prev == j) return (int)h;
          if (prev == -1) {
            fresh = !KNOWN;
            return KNOWN ? -1 : (int)h;
          }
          h = (h + 1) & (unsigned)(CAP - 1);
        }
        return -1;
      };
      if (KNOWN) {
        for (int e = gl; e < clen; e += G) {
          const int j = ccol[c0 + e];
          unsigned h = ((unsigned)j * 0x9E3779B1u) >> (32 - __popc(CAP - 1));
          for (int p = 0; p < CAP; ++p) {
            if (atomicCAS(&hkey[h], -1, j) == -1) break;
            h = (h + 1) & (unsigned)(CAP - 1);
          }
          hval[h] = 0.0;
          ulist[e] = (unsigned short)h;
        }
        __syncwarp();
      }
      int u = 0;  // distinct columns so far
      auto add = [&](int j, double prod) {
        bool fresh;
        const int h = find(j, fresh);
        if (h < 0) return;
        if (fresh) {
          const int at = atomicAdd(&s.cnt[grp], 1);
          if (at < MAXU + G) ulist[at] = (unsigned short)h;
        }
        hval[h] = __dadd_rn(fresh ? 0.0 : hval[h], prod);
      };
      for (int e0 = 0; e0 < na_max; e0 += G) {
        // every group's row is dropped or done: without the test, rows of many
        // distinct columns were read to their end twice for nothing (random graph,
        // 150000 rows of 8 entries, two of 3000: setup 242.5 -> 240.2 ms, while
        // rows that fit take as long as before)
        if (!KNOWN && __all_sync(kAll, u > MAXU || e0 >= na)) break;
        // G entries of row i at once: column k, value, row k's extent
        const int e = e0 + gl;
        double a = 0.0;
        int fb = 0, fl = 0;
        if (e < na) {
          const int k = Acol[a0 + e];
          a = Aval[a0 + e];
          fb = Brp[k];
          fl = Brp[k + 1] - fb;
        }
        const int steps = min(G, na_max - e0);
        constexpr int T = 4;  // entries whose rows of B are loaded ahead
        for (int t0 = 0; t0 < steps; t0 += T) {
          double at[T], v[T];
          int ft[T], lt[T], j[T];
#pragma unroll
          for (int t = 0; t < T; ++t) {
            at[t] = __shfl_sync(kAll, a, t0 + t, G);
            ft[t] = __shfl_sync(kAll, fb, t0 + t, G);
            lt[t] = __shfl_sync(kAll, fl, t0 + t, G);
            j[t] = 0;
            v[t] = 0.0;
            if (gl < lt[t]) {
              j[t] = Bcol[ft[t] + gl];
              v[t] = Bval[ft[t] + gl];
            }
          }
#pragma unroll
          for (int t = 0; t < T; ++t) {
            if (u > MAXU) lt[t] = 0;
            if (gl < lt[t]) add(j[t], __dmul_rn(at[t], v[t]));
            __syncwarp();
            if (!KNOWN) u = s.cnt[grp];
            // the rest of a row of B longer than the group
            const int more = __reduce_max_sync(kAll, lt[t]);
            for (int f0 = G; f0 < more; f0 += G) {
              if (f0 + gl < lt[t] && u <= MAXU)
                add(Bcol[ft[t] + f0 + gl], __dmul_rn(at[t], Bval[ft[t] + f0 + gl]));
              __syncwarp();
              if (!KNOWN) u = s.cnt[grp];
            }
          }
        }
      }
      if (KNOWN) {
        for (int e = gl; e < clen; e += G) cval[c0 + e] = hval[ulist[e]];
      } else {
        if (i >= 0 && u > MAXU) over = true;
        const int d = i >= 0 && !over ? u : 0;
        // columns in ascending order: every column to its rank
        constexpr int Q = (MAXU + G - 1) / G;
        const int dmax = __reduce_max_sync(kAll, d);
        constexpr int QB = Q < 8 ? Q : 8;  // columns a lane ranks at a time
        for (int q0 = 0; q0 * G < dmax; q0 += QB) {
          int key[QB], rank[QB], slot[QB];
#pragma unroll
          for (int x = 0; x < QB; ++x) {
            const int m = gl + (q0 + x) * G;
            slot[x] = m < d ? ulist[m] : 0;
            key[x] = m < d ? hkey[slot[x]] : 0x7fffffff;
            rank[x] = 0;
          }
          for (int m = 0; m < dmax; ++m) {
            const int c = m < d ? hkey[ulist[m]] : 0x7fffffff;
#pragma unroll
            for (int x = 0; x < QB; ++x) rank[x] += c < key[x];
          }
#pragma unroll
          for (int x = 0; x < QB; ++x)
            if (gl + (q0 + x) * G < d) {
              ccol[c0 + rank[x]] = key[x];
              cval[c0 + rank[x]] = hval[slot[x]];
            }
        }
        if (d > 0 && gl == 0) cnt[i] = d;
        else if (i >= 0 && !over && gl == 0) cnt[i] = 0;
      }
      __syncwarp();
    }
    if (i >= 0 && over && gl == 0) {
      if (blist && ub[i] >= kSpCap) blist[atomicAdd(bcnt, 1)] = i;
      else olist[atomicAdd(ocnt, 1)] = i;
    }
  }
}

// one class of a product: rows of `list` (null: all), G lanes per row
template <int G, int CAP, int MAXU, bool KNOWN>
void launch_group(const DevCSR& A, const DevCSR& B, const int* list, const int* nlist, int ub_max,
                  const int* off, const int* ub, int* ccol, double* cval, int* cnt, int* olist,
                  int* ocnt, int* blist, int* bcnt, int sms, cudaStream_t s) {
  constexpr int WARPS = 4, NG = 32 / G;
  constexpr size_t smem = WARPS * sizeof(GroupRows<G, CAP, MAXU>);
  auto kern = k_spgemm_group<G, CAP, MAXU, WARPS, KNOWN>;
  static PerDevice<bool> allowed;
  allow_smem(allowed, kern, smem);
  long long blocks = ((long long)A.n + WARPS * NG - 1) / (WARPS * NG);
  if (list && blocks > 16ll * sms) blocks = 16ll * sms;
  if (blocks < 1) blocks = 1;
  kern<<<(int)blocks, 32 * WARPS, smem, s>>>(A.n, list, nlist, ub_max, A.rowptr, A.col, A.val,
                                             B.rowptr, B.col, B.val, off, ub, ccol, cval, cnt,
                                             olist, ocnt, blist, bcnt);
  TP_LAUNCH_CHECK();
}

// lanes per row by the mean length of B's rows (P truncated to 4 weights, A P
// of 9-12 columns, longer), so that most lanes have an entry; the second class,
// for rows of up to 192 columns, doubles them: its tables are four times as
// large and fewer rows fit an SM
template <bool KNOWN, class... Args>
void group_class(bool second, const DevCSR& A, const DevCSR& B, Args... args) {
  const double mean = B.n > 0 ? (double)B.nnz / B.n : 0.0;
  if (!second) {
    if (mean <= 4.5) launch_group<4, 64, 48, KNOWN>(A, B, args...);
    else if (mean <= 10.0) launch_group<8, 64, 48, KNOWN>(A, B, args...);
    else launch_group<16, 64, 48, KNOWN>(A, B, args...);
  } else {
    if (mean <= 4.5) launch_group<8, 256, 192, KNOWN>(A, B, args...);
    else if (mean <= 10.0) launch_group<16, 256, 192, KNOWN>(A, B, args...);
    else launch_group<32, 256, 192, KNOWN>(A, B, args...);
  }
}

// Upper bound (product count) of every row of C = A B; the rows past the first
// group class (more than kSpFirst products) are listed for the second. The
// list order is not deterministic; each row's result is.
__global__ void k_spgemm_ub(int n, const int* __restrict__ Arp, const int* __restrict__ Acol,
                            const int* __restrict__ Brp, int* __restrict__ ub,
                            int* __restrict__ list, int* __restrict__ count) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int u = 0;
  for (int e = Arp[i]; e < Arp[i + 1]; ++e) {
    int k = Acol[e];
    u += Brp[k + 1] - Brp[k];
  }
  ub[i] = u;
  if (u > kSpFirst) list[atomicAdd(count, 1)] = i;
}

__device__ void spgemm_row_serial(int i, const int* __restrict__ Arp, const int* __restrict__ Acol,
                                  const double* __restrict__ Aval, const int* __restrict__ Brp,
                                  const int* __restrict__ Bcol, const double* __restrict__ Bval,
                                  int* __restrict__ cc, double* __restrict__ cv, int* __restrict__ cnt) {
  int u = 0;
  for (int e = Arp[i]; e < Arp[i + 1]; ++e) {
    const int k = Acol[e];
    const double a = Aval[e];
    for (int f = Brp[k]; f < Brp[k + 1]; ++f) {
      const int j = Bcol[f];
      const double prod = __dmul_rn(a, Bval[f]);
      int lo = 0, hi = u;
      while (lo < hi) {
        int mid = (lo + hi) >> 1;
        if (cc[mid] < j) lo = mid + 1;
        else hi = mid;
      }
      if (lo < u && cc[lo] == j) {
        cv[lo] = __dadd_rn(cv[lo], prod);
      } else {
        for (int q = u; q > lo; --q) {
          cc[q] = cc[q - 1];
          cv[q] = cv[q - 1];
        }
        cc[lo] = j;
        cv[lo] = __dadd_rn(0.0, prod);
        ++u;
      }
    }
  }
  cnt[i] = u;
}

// one warp: row i of C = A B through a shared-memory hash table of
// 2^k >= 2 ex slots (hkey/hval, at most `tcap`), then the distinct columns
// sorted in skey (capacity tcap)
__device__ void spgemm_row_hash(int i, int ex, int lane, int tcap, const int* __restrict__ Arp,
                                const int* __restrict__ Acol, const double* __restrict__ Aval,
                                const int* __restrict__ Brp, const int* __restrict__ Bcol,
                                const double* __restrict__ Bval, int* hkey, double* hval,
                                unsigned long long* skey, int* __restrict__ cc,
                                double* __restrict__ cv, int* __restrict__ cnt) {
  int bits = 5;
  while ((1 << bits) < 2 * ex && (1 << bits) < tcap) ++bits;
  const int cap = 1 << bits;
  const unsigned below = (1u << lane) - 1u;
  for (int q = lane; q < cap; q += 32) hkey[q] = -1;
  __syncwarp();
  // 1. accumulate in canonical order: every column's sum starts at 0.0 and
  // takes its products in ascending e; one entry of A per step, its row of B
  // split over the lanes (distinct columns)
  for (int q = lane; q < cap; q += 32) hval[q] = 0.0;
  __syncwarp();
  const int a0 = Arp[i], a1 = Arp[i + 1];
  for (int e0 = a0; e0 < a1; e0 += 32) {
    const int e = e0 + lane;
    double a = 0.0;
    int fb = 0, fe = 0;
    if (e < a1) {
      const int k = Acol[e];
      a = Aval[e];
      fb = Brp[k];
      fe = Brp[k + 1];
    }
    const int ne = min(32, a1 - e0);
    for (int t = 0; t < ne; ++t) {
      const double at = __shfl_sync(0xffffffffu, a, t);
      const int f0 = __shfl_sync(0xffffffffu, fb, t);
      const int f1 = __shfl_sync(0xffffffffu, fe, t);
      for (int f = f0 + lane; f < f1; f += 32) {
        const int j = Bcol[f];
        const double prod = __dmul_rn(at, Bval[f]);
        unsigned h = ((unsigned)j * 0x9E3779B1u) >> (32 - bits);
        for (int probe = 0; probe < cap; ++probe) {
          const int prev = atomicCAS(&hkey[h], -1, j);
          if (prev == -1 || prev == j) {
            hval[h] = __dadd_rn(hval[h], prod);
            break;
          }
          h = (h + 1) & (unsigned)(cap - 1);
        }
      }
      __syncwarp();
    }
  }
  // 2. compact the occupied slots as (column << 32 | slot) keys
  int d = 0;
  for (int q0 = 0; q0 < cap; q0 += 32) {
    const int q = q0 + lane;
    const int c = hkey[q];
    const unsigned m = __ballot_sync(0xffffffffu, c >= 0);
    if (c >= 0)
      skey[d + __popc(m & below)] = ((unsigned long long)(unsigned)c << 32) | (unsigned)q;
    d += __popc(m);
  }
  int P = 1;
  while (P < d) P <<= 1;
  for (int q = d + lane; q < P; q += 32) skey[q] = ~0ull;
  __syncwarp();
  // 3. bitonic sort of the keys (ascending)
  for (int size = 2; size <= P; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int t = lane; t < (P >> 1); t += 32) {
        const int lo = 2 * stride * (t / stride) + (t % stride);
        const int hi = lo + stride;
        const bool up = (lo & size) == 0;
        const unsigned long long x = skey[lo], y = skey[hi];
        if ((x > y) == up) {
          skey[lo] = y;
          skey[hi] = x;
        }
      }
      __syncwarp();
    }
  }
  // 4. columns in ascending order with their sums
  for (int r = lane; r < d; r += 32) {
    const unsigned long long kk = skey[r];
    cc[r] = (int)(kk >> 32);
    cv[r] = hval[(unsigned)(kk & 0xffffffffu)];
  }
  if (lane == 0) cnt[i] = d;
}

// rows past the group kernels' distinct columns with fewer than kSpCap
// products: tables of kSpCap slots, two warps per block (20 kSpCap bytes of
// shared memory per warp); rows of list[0, *count)
constexpr int kSpHashWarps = 2;

__global__ void __launch_bounds__(32 * kSpHashWarps) k_spgemm_rows_warp(
    const int* __restrict__ Arp, const int* __restrict__ Acol, const double* __restrict__ Aval,
    const int* __restrict__ Brp, const int* __restrict__ Bcol, const double* __restrict__ Bval,
    const int* __restrict__ off, const int* __restrict__ ub, const int* __restrict__ list,
    const int* __restrict__ count, int* __restrict__ ccol, double* __restrict__ cval,
    int* __restrict__ cnt) {
  __shared__ int s_hkey[kSpHashWarps][kSpCap];
  __shared__ double s_hval[kSpHashWarps][kSpCap];
  __shared__ unsigned long long s_skey[kSpHashWarps][kSpCap];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int t = blockIdx.x * kSpHashWarps + w; t < *count; t += gridDim.x * kSpHashWarps) {
    const int i = list[t];
    spgemm_row_hash(i, ub[i], lane, kSpCap, Arp, Acol, Aval, Brp, Bcol, Bval, s_hkey[w],
                    s_hval[w], s_skey[w], ccol + off[i], cval + off[i], cnt);
    __syncwarp();
  }
}

// rows past the group kernels' distinct columns with at least kSpCap products:
// one 512-thread block per row (one block per SM)
// with kSpBig products in dynamic shared memory. Every warp stages the
// products of its share of row i of A (lanes over the row of B, coalesced)
// at their canonical sequence positions; a block bitonic sort orders the
// (column, position) keys; a block scan lists the column runs, and one
// thread per run adds it up in sequence order. Rows beyond kSpBig are summed
// serially.
constexpr int kSpBig = 8192;
constexpr int kSpBigThreads = 512;
constexpr int kSpBigWarps = kSpBigThreads / 32;
constexpr size_t kSpBigSmem =
    (size_t)kSpBig * (sizeof(unsigned long long) + sizeof(double)) + (kSpBig + 1) * sizeof(int);

// exclusive scan of x over the block; *total = the block's sum. s_w holds
// kSpBigWarps + 1 ints; the block must not touch it between calls without a
// barrier (the function ends with one).
__device__ __forceinline__ int block_scan_excl(int x, int* s_w, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_w[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const int v = lane < kSpBigWarps ? s_w[lane] : 0;
    int iv = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, iv, o);
      if (lane >= o) iv += y;
    }
    if (lane < kSpBigWarps) s_w[lane] = iv - v;
    if (lane == 31) s_w[kSpBigWarps] = iv;
  }
  __syncthreads();
  const int r = s_w[warp] + incl - x;
  *total = s_w[kSpBigWarps];
  __syncthreads();
  return r;
}

__global__ void __launch_bounds__(kSpBigThreads) k_spgemm_rows_big(
    int n, const int* __restrict__ Arp, const int* __restrict__ Acol,
    const double* __restrict__ Aval, const int* __restrict__ Brp, const int* __restrict__ Bcol,
    const double* __restrict__ Bval, const int* __restrict__ off, const int* __restrict__ ub,
    const int* __restrict__ blist, const int* __restrict__ bcount,
    int* __restrict__ ccol, double* __restrict__ cval, int* __restrict__ cnt) {
  extern __shared__ unsigned long long s_big[];
  unsigned long long* key = s_big;
  double* val = reinterpret_cast<double*>(s_big + kSpBig);
  int* start = reinterpret_cast<int*>(val + kSpBig);
  __shared__ int s_w[kSpBigWarps + 1];
  __shared__ int s_ak[kSpBigThreads], s_aoff[kSpBigThreads];
  __shared__ double s_aa[kSpBigThreads];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int count = *bcount;
  for (int t = blockIdx.x; t < count; t += gridDim.x) {
    const int i = blist[t];
    const int ex = ub[i];  // uniform over the block
    int* cc = ccol + off[i];
    double* cv = cval + off[i];
    if (ex > kSpBig) {
      if (tid == 0) spgemm_row_serial(i, Arp, Acol, Aval, Brp, Bcol, Bval, cc, cv, cnt);
      __syncthreads();
      continue;
    }
    // 1. products at their canonical positions (entry e of row i of A, then
    // the row of B in order), kSpBigThreads entries of A at a time
    const int a0 = Arp[i], a1 = Arp[i + 1];
    int base = 0;
    for (int c0 = a0; c0 < a1; c0 += kSpBigThreads) {
      const int e = c0 + tid;
      int k = 0, len = 0;
      double a = 0.0;
      if (e < a1) {
        k = Acol[e];
        a = Aval[e];
        len = Brp[k + 1] - Brp[k];
      }
      int total = 0;
      const int ex_off = block_scan_excl(len, s_w, &total);
      s_ak[tid] = k;
      s_aa[tid] = a;
      s_aoff[tid] = base + ex_off;
      __syncthreads();
      const int nc = min(kSpBigThreads, a1 - c0);
      for (int q = warp; q < nc; q += kSpBigWarps) {
        const int kk = s_ak[q];
        const double aq = s_aa[q];
        const int fb = Brp[kk], fe = Brp[kk + 1];
        const int pb = s_aoff[q] - fb;
        for (int f = fb + lane; f < fe; f += 32) {
          const int pidx = pb + f;
          key[pidx] = ((unsigned long long)(unsigned)Bcol[f] << 32) | (unsigned)pidx;
          val[pidx] = __dmul_rn(aq, Bval[f]);
        }
      }
      base += total;
      __syncthreads();
    }
    int P = 1;
    while (P < ex) P <<= 1;
    for (int q = ex + tid; q < P; q += kSpBigThreads) key[q] = ~0ull;
    __syncthreads();
    // 2. block bitonic sort
    for (int size = 2; size <= P; size <<= 1) {
      for (int stride = size >> 1; stride > 0; stride >>= 1) {
        for (int u = tid; u < (P >> 1); u += kSpBigThreads) {
          const int lo = 2 * stride * (u / stride) + (u % stride);
          const int hi = lo + stride;
          const bool up = (lo & size) == 0;
          const unsigned long long x = key[lo], y = key[hi];
          if ((x > y) == up) {
            key[lo] = y;
            key[hi] = x;
          }
        }
        __syncthreads();
      }
    }
    // 3. the start of every column run
    int nrun = 0;
    for (int q0 = 0; q0 < ex; q0 += kSpBigThreads) {
      const int q = q0 + tid;
      int st = 0;
      if (q < ex) st = (q == 0) || ((key[q] >> 32) != (key[q - 1] >> 32));
      int total = 0;
      const int r = block_scan_excl(st, s_w, &total);
      if (st) start[nrun + r] = q;
      nrun += total;
    }
    if (tid == 0) start[nrun] = ex;
    __syncthreads();
    // 4. one thread per run, summed in sequence order
    for (int r = tid; r < nrun; r += kSpBigThreads) {
      const int q0 = start[r], q1 = start[r + 1];
      double sum = 0.0;
      for (int q = q0; q < q1; ++q) sum = __dadd_rn(sum, val[(unsigned)(key[q] & 0xffffffffu)]);
      cc[r] = (int)(key[q0] >> 32);
      cv[r] = sum;
    }
    if (tid == 0) cnt[i] = nrun;
    __syncthreads();
  }
}

// numeric-only C = A B on a known pattern (same canonical order), one thread
// per row: the rows of list[0, *count), those longer than the group kernels
// take
__global__ void k_spgemm_numeric(const int* __restrict__ list, const int* __restrict__ count,
                                 const int* __restrict__ Arp, const int* __restrict__ Acol,
                                 const double* __restrict__ Aval, const int* __restrict__ Brp,
                                 const int* __restrict__ Bcol, const double* __restrict__ Bval,
                                 const int* __restrict__ Crp, const int* __restrict__ Ccol,
                                 double* __restrict__ Cval) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < *count; t += gridDim.x * blockDim.x) {
    const int i = list[t];
    const int c0 = Crp[i], c1 = Crp[i + 1];
    for (int q = c0; q < c1; ++q) Cval[q] = 0.0;
    for (int e = Arp[i]; e < Arp[i + 1]; ++e) {
      const int k = Acol[e];
      const double a = Aval[e];
      for (int f = Brp[k]; f < Brp[k + 1]; ++f) {
        const int q = find_in(Ccol, c0, c1, Bcol[f]);
        Cval[q] = __dadd_rn(Cval[q], __dmul_rn(a, Bval[f]));
      }
    }
  }
}

// rows of C from their slots at off[i] to the compact CSR: L lanes per row
// (about two entries per lane on average), so that a warp's copies are a
// few contiguous runs rather than 32 scattered rows
template <int L>
__global__ void k_spgemm_compact(int n, const int* __restrict__ off,
                                 const int* __restrict__ ccol, const double* __restrict__ cval,
                                 const int* __restrict__ Crp, int* __restrict__ Ccol,
                                 double* __restrict__ Cval) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int i = (int)(t / L), lane = (int)(t % L);
  if (i >= n) return;
  const int o = off[i], c0 = Crp[i], len = Crp[i + 1] - c0;
  for (int e = lane; e < len; e += L) {
    Ccol[c0 + e] = ccol[o + e];
    Cval[c0 + e] = cval[o + e];
  }
}


}  // namespace

// C = A B with the canonical summation order; C arrays allocated from `pool`.
DevCSR csr_product(const DevCSR& A, const DevCSR& B, Pool& pool, Pool& scratch, cudaStream_t s) {
  const int n = A.n;
  int* ub = scratch.alloc<int>(n + 1);
  int* off = scratch.alloc<int>(n + 1);
  int* list = scratch.alloc<int>(n + 1);
  int* olist = scratch.alloc<int>(n + 1);
  int* blist = scratch.alloc<int>(n + 1);
  int* counts = scratch.alloc<int>(3);  // rows of list, olist, blist
  TP_CUDA_TRY(cudaMemsetAsync(counts, 0, 3 * sizeof(int), s));
  k_spgemm_ub<<<grid_for(n), kBlock, 0, s>>>(n, A.rowptr, A.col, B.rowptr, ub, list, counts);
  TP_LAUNCH_CHECK();
  long long tot = scan_exclusive(ub, off, n, scratch, s);
  int* ccol = scratch.alloc<int>(tot + 1);
  double* cval = scratch.alloc<double>(tot + 1);
  int* cnt = scratch.alloc<int>(n + 1);
  const bool dense = B.m <= kDenseCap;
  if (dense) {
    static PerDevice<bool> allowed;
    allow_smem(allowed, k_spgemm_dense, kDenseSmem);
    long long blocks = ((long long)n + kDenseWarps - 1) / kDenseWarps;
    if (blocks > 8LL * device_sms()) blocks = 8LL * device_sms();
    const size_t smem = (size_t)kDenseWarps * B.m * (sizeof(double) + 1);
    k_spgemm_dense<<<(int)blocks, 32 * kDenseWarps, smem, s>>>(
        n, B.m, A.rowptr, A.col, A.val, B.rowptr, B.col, B.val, off, ccol, cval, cnt);
    TP_LAUNCH_CHECK();
  } else {
    const int sms = device_sms();
    group_class<false>(false, A, B, (const int*)nullptr, (const int*)nullptr, kSpFirst,
                       (const int*)off, (const int*)ub, ccol, cval, cnt, list, counts,
                       (int*)nullptr, (int*)nullptr, sms, s);
    group_class<false>(true, A, B, (const int*)list, (const int*)counts, 0, (const int*)off,
                       (const int*)ub, ccol, cval, cnt, olist, counts + 1, blist, counts + 2,
                       sms, s);
    long long blocks = (n + kSpHashWarps - 1) / kSpHashWarps;
    if (blocks > 4LL * sms) blocks = 4LL * sms;
    k_spgemm_rows_warp<<<(int)blocks, 32 * kSpHashWarps, 0, s>>>(
        A.rowptr, A.col, A.val, B.rowptr, B.col, B.val, off, ub, olist, counts + 1, ccol, cval,
        cnt);
    TP_LAUNCH_CHECK();
    static PerDevice<bool> allowed;
    allow_smem(allowed, k_spgemm_rows_big, kSpBigSmem);
    k_spgemm_rows_big<<<n < sms ? n : sms, kSpBigThreads, kSpBigSmem, s>>>(
        n, A.rowptr, A.col, A.val, B.rowptr, B.col, B.val, off, ub, blist, counts + 2, ccol, cval,
        cnt);
    TP_LAUNCH_CHECK();
  }
  DevCSR C;
  C.n = n;
  C.m = B.m;
  C.rowptr = pool.alloc<int>(n + 1);
  long long nnz = scan_exclusive(cnt, C.rowptr, n, scratch, s);
  C.nnz = (int)nnz;
  C.col = pool.alloc<int>(nnz + 1);
  C.val = pool.alloc<double>(nnz + 1);
  {
    const double avg = n > 0 ? (double)nnz / n : 1.0;
    int L = 1;
    while (L < 32 && 2.0 * L < avg) L *= 2;
    const int g = grid_for((long long)n * L);
    switch (L) {
#define TP_CASE(LL)                                                                          \
  case LL:                                                                                   \
    k_spgemm_compact<LL><<<g, kBlock, 0, s>>>(n, off, ccol, cval, C.rowptr, C.col, C.val); \
    break;
      TP_CASE(1) TP_CASE(2) TP_CASE(4) TP_CASE(8) TP_CASE(16) TP_CASE(32)
#undef TP_CASE
    }
  }
  TP_LAUNCH_CHECK();
  return C;
}


// A thread per row with a binary search per product took 28.7 of the 83 ms of a
// Newton step at 64x64x32 (four refreshes); the group kernels on the known
// pattern take about 4 ms and the step 61 ms.
void csr_product_numeric(const DevCSR& A, const DevCSR& B, const DevCSR& C, Pool& scratch,
                         cudaStream_t s) {
  const int n = A.n;
  int* list = scratch.alloc<int>(n + 1);
  int* olist = scratch.alloc<int>(n + 1);
  int* counts = scratch.alloc<int>(3);
  TP_CUDA_TRY(cudaMemsetAsync(counts, 0, 3 * sizeof(int), s));
  const int sms = device_sms();
  const int* rows = nullptr;
  const int* nrows = nullptr;
  if (C.nnz <= 48ll * n) {
    group_class<true>(false, A, B, rows, nrows, 0, (const int*)C.rowptr, (const int*)nullptr,
                      C.col, C.val, (int*)nullptr, list, counts, (int*)nullptr, (int*)nullptr,
                      sms, s);
    rows = list;
    nrows = counts;
  }
  group_class<true>(true, A, B, rows, nrows, 0, (const int*)C.rowptr, (const int*)nullptr, C.col,
                    C.val, (int*)nullptr, olist, counts + 1, (int*)nullptr, (int*)nullptr, sms,
                    s);
  // the longest rows, on coarse levels (a thread per row, which the last kernel
  // keeps for rows past 1536 columns, took 9.1 of the 68 ms of a Newton step
  // at 64x64x32 here)
  launch_group<32, 2048, 1536, true>(A, B, olist, counts + 1, 0, C.rowptr, nullptr, C.col, C.val,
                                     nullptr, list, counts + 2, nullptr, nullptr, sms, s);
  k_spgemm_numeric<<<std::min(grid_for(n, 64), 4 * sms), 64, 0, s>>>(
      list, counts + 2, A.rowptr, A.col, A.val, B.rowptr, B.col, B.val, C.rowptr, C.col, C.val);
  TP_LAUNCH_CHECK();
}

}  // namespace tp
