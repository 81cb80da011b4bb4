// AMG setup kernels: strength, PMIS, interpolation, transpose, Galerkin
// product, smoother scaling and the coarsest-level inverse.
//
// The paper inverts A_pp and S~_T approximately with an AMG V-cycle
// (Sec. 3.2) built with classical Ruge-Stueben interpolation and Gaussian
// elimination on the coarsest grid (Sec. 4 solver settings). Here the C/F
// split is PMIS with seeded tie-breaks and the interpolation is classical or
// its distance-two extended+i form; all structure-deciding arithmetic uses
// __dmul_rn / __dadd_rn / __ddiv_rn in a fixed ascending-column order.
#include "amg_dev.cuh"
#include "per_device.cuh"
#include <cmath>
#include <algorithm>

namespace tp {

namespace {

long long resident_threads();

// (d > 0 && a < 0) || (d < 0 && a > 0), decided on the bit patterns: both
// non-zero, neither NaN, signs differ. Integer operations instead of FP64
// comparisons, which on this part share the FP64 pipe (2 per clock per SM)
// with the setup's multiply-adds and divisions.
__device__ __forceinline__ bool opposite(double a, double d) {
  const unsigned long long ua = (unsigned long long)__double_as_longlong(a);
  const unsigned long long ud = (unsigned long long)__double_as_longlong(d);
  const unsigned long long ma = ua & 0x7fffffffffffffffull, md = ud & 0x7fffffffffffffffull;
  const unsigned long long inf = 0x7ff0000000000000ull;
  return ma != 0 && md != 0 && ma <= inf && md <= inf && ((ua ^ ud) >> 63) != 0;
}

__global__ void k_diag_pos(int n, const int* __restrict__ rp, const int* __restrict__ col,
                           int* __restrict__ dpos, int* __restrict__ err) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int p = find_in(col, rp[i], rp[i + 1], i);
  dpos[i] = p;
  if (p < 0) atomicOr(err, 1);
}

__global__ void k_transpose_pos(int n, const int* __restrict__ rp, const int* __restrict__ col,
                                int* __restrict__ tpos, int* __restrict__ err) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  for (int e = rp[i]; e < rp[i + 1]; ++e) {
    int k = col[e];
    int p = (k >= 0 && k < n) ? find_in(col, rp[k], rp[k + 1], i) : -1;
    tpos[e] = p;
    if (p < 0) atomicOr(err, 2);
  }
}

// the same with one warp per row (lanes over the row's entries): for the
// long rows of coarse Galerkin levels
__global__ void k_transpose_pos_warp(int n, const int* __restrict__ rp,
                                     const int* __restrict__ col, int* __restrict__ tpos,
                                     int* __restrict__ err) {
  const int lane = threadIdx.x & 31;
  const int i = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  if (i >= n) return;
  for (int e = rp[i] + lane; e < rp[i + 1]; e += 32) {
    int k = col[e];
    int p = (k >= 0 && k < n) ? find_in(col, rp[k], rp[k + 1], i) : -1;
    tpos[e] = p;
    if (p < 0) atomicOr(err, 2);
  }
}

// mean row length from which row-wise setup kernels take one warp per row
constexpr int kWarpRowMean = 16;

// Strength and PMIS take L lanes per row: 8 on short-row levels (the 7-point
// finest, S~'s first Galerkin levels), a warp where the mean row length is at
// least kWarpRowMean; a row's decision is a maximum, a count or an any over its
// lanes.
//
// strong[e] = 1 iff col != i and -a_e >= theta * max_{k != i}(-a_ik) > 0. The
// magnitudes of the negative entries are compared as integers (their bit
// patterns order like the values): FP64 comparisons would take the FP64 pipe
// for the whole warp (37 M entries of the layered A_pp's first Galerkin level
// 868 us with them, a warp per row).
template <int L>
__global__ void __launch_bounds__(256) k_strength(int n, const int* __restrict__ rp,
                                                  const int* __restrict__ col,
                                                  const double* __restrict__ val, double theta,
                                                  unsigned char* __restrict__ strong) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int i = (int)(t / L), lane = (int)(t % L);
  const int r0 = i < n ? rp[i] : 0, r1 = i < n ? rp[i + 1] : 0;
  // |a| of a negative entry off the diagonal (NaN and the others: 0)
  auto key = [&](int e) -> unsigned long long {
    const unsigned long long u = (unsigned long long)__double_as_longlong(val[e]);
    const unsigned long long m = u & 0x7fffffffffffffffull;
    return (u >> 63) && m <= 0x7ff0000000000000ull && col[e] != i ? m : 0ull;
  };
  unsigned long long mx = 0;
  for (int e = r0 + lane; e < r1; e += L) mx = max(mx, key(e));
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const unsigned long long thr = (unsigned long long)__double_as_longlong(
      __dmul_rn(theta, __longlong_as_double((long long)mx)));
  for (int e = r0 + lane; e < r1; e += L) {
    bool s = false;
    if (mx != 0) {
      s = key(e) >= thr;
      // a threshold that underflowed to zero is met by zeros, and by nothing
      // positive, NaN or on the diagonal
      if (thr == 0) {
        const unsigned long long u = (unsigned long long)__double_as_longlong(val[e]);
        s = col[e] != i && ((u << 1) == 0 || key(e) != 0);
      }
    }
    strong[e] = s ? 1 : 0;
  }
}

template <int L>
__global__ void __launch_bounds__(256) k_pmis_init(int n, const int* __restrict__ rp,
                                                   const int* __restrict__ col,
                                                   const unsigned char* __restrict__ strong,
                                                   const int* __restrict__ tpos,
                                                   int* __restrict__ lam,
                                                   signed char* __restrict__ state,
                                                   unsigned char* __restrict__ newc) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  const int i = (int)(t / L), lane = (int)(t % L);
  int l = 0;
  if (i < n)
    for (int e = rp[i] + lane; e < rp[i + 1]; e += L)
      if (col[e] != i && strong[tpos[e]]) ++l;
#pragma unroll
  for (int o = L / 2; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
  if (i < n && lane == 0) {
    lam[i] = l;
    state[i] = (l == 0) ? kF : kU;
    newc[i] = 0;
  }
}

// The undecided rows among the block's `rows` (at most 256), listed in shared
// memory; returns their number. A round's kernels touch fewer and fewer rows:
// with a lane group per row, decided or not, the rounds of the layered
// 256x256x64 setups took 10.8 ms of kernel time, with the list 6.2.
__device__ __forceinline__ int undecided_rows(int n, int rows,
                                              const signed char* __restrict__ state, int* s_list,
                                              int* s_warp) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * rows + threadIdx.x;
  const bool und = (int)threadIdx.x < rows && i < n && state[i] == kU;
  const unsigned m = __ballot_sync(0xffffffffu, und);
  if (lane == 0) s_warp[warp] = __popc(m);
  __syncthreads();
  int before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    const int c = s_warp[w];
    if (w < warp) before += c;
    total += c;
  }
  if (und) s_list[before + __popc(m & ((1u << lane) - 1u))] = i;
  __syncthreads();
  return total;
}

// newc = 1 where an undecided point beats every undecided neighbour it is
// strongly connected to, either way (decided points keep theirs: 1 for C, 0
// for F)
template <int L>
__global__ void __launch_bounds__(256) k_pmis_select(
    int n, const int* __restrict__ rp, const int* __restrict__ col,
    const unsigned char* __restrict__ strong, const int* __restrict__ tpos,
    const int* __restrict__ lam, const signed char* __restrict__ state, unsigned long long seed,
    int rows, unsigned char* __restrict__ newc, int* __restrict__ undecided) {
  __shared__ int s_list[256], s_warp[8];
  if (blockIdx.x == 0 && threadIdx.x == 0) *undecided = 0;  // set again by k_pmis_update
  const int m = undecided_rows(n, rows, state, s_list, s_warp);
  constexpr int NG = 32 / L;  // rows a warp takes at a time
  const int lane = threadIdx.x & 31, gl = lane % L;
  for (int q0 = (threadIdx.x >> 5) * NG; q0 < m; q0 += 8 * NG) {
    const int q = q0 + lane / L;
    const int i = q < m ? s_list[q] : -1;
    bool bigger = false;
    if (i >= 0) {
      const int li = lam[i];
      const unsigned int hi = pmis_hash(seed, i);
      for (int e = rp[i] + gl; e < rp[i + 1] && !bigger; e += L) {
        const int k = col[e];
        if (k == i || state[k] != kU) continue;
        if (!(strong[e] || strong[tpos[e]])) continue;
        const int lk = lam[k];
        const unsigned int hk = pmis_hash(seed, k);
        bigger = (lk > li) || (lk == li && (hk > hi || (hk == hi && k > i)));
      }
    }
    const unsigned any = __ballot_sync(0xffffffffu, bigger) >> (lane - gl);
    if (i >= 0 && gl == 0) newc[i] = (any & (L == 32 ? 0xffffffffu : (1u << L) - 1u)) ? 0 : 1;
  }
}

// new C points, and F where a point strongly depends on a C point; points left
// undecided set *undecided, once per block
template <int L>
__global__ void __launch_bounds__(256) k_pmis_update(
    int n, const int* __restrict__ rp, const int* __restrict__ col,
    const unsigned char* __restrict__ strong, signed char* __restrict__ state, int rows,
    const unsigned char* __restrict__ newc, int* __restrict__ undecided) {
  __shared__ int s_list[256], s_warp[8];
  const int m = undecided_rows(n, rows, state, s_list, s_warp);
  constexpr int NG = 32 / L;
  const int lane = threadIdx.x & 31, gl = lane % L;
  bool left = false;
  for (int q0 = (threadIdx.x >> 5) * NG; q0 < m; q0 += 8 * NG) {
    const int q = q0 + lane / L;
    const int i = q < m ? s_list[q] : -1;
    const bool isc = i >= 0 && newc[i];
    bool c = false;
    if (i >= 0 && !isc)
      for (int e = rp[i] + gl; e < rp[i + 1] && !c; e += L) {
        const int k = col[e];
        c = strong[e] && (newc[k] || state[k] == kC);
      }
    const unsigned any = (__ballot_sync(0xffffffffu, c) >> (lane - gl)) &
                         (L == 32 ? 0xffffffffu : (1u << L) - 1u);
    if (i >= 0 && gl == 0) {
      if (isc) state[i] = kC;
      else if (any) state[i] = kF;
      else left = true;
    }
  }
  if (__syncthreads_or(left) && threadIdx.x == 0) *undecided = 1;
}

// Untruncated interpolation. The kernels take the rows list[0, n) (LISTED) or
// rows 0 to n - 1; cnt, ub, off and Prp are indexed by the place in the list.
// (The list is the last parameter: as the second one it cost the unlisted
// k_extpi_fill_warp 1 %, 173.5 -> 175.8 ms on 3000 rows of 700 entries.)
template <bool LISTED>
__device__ __forceinline__ int listed_row(const int* __restrict__ list, int q) {
  return LISTED ? list[q] : q;
}

// ---------------------------------------------------- classical interpolation
__device__ __forceinline__ bool is_strong_c(const int* __restrict__ rp,
                                            const int* __restrict__ col,
                                            const unsigned char* __restrict__ strong,
                                            const signed char* __restrict__ state, int i, int m) {
  int p = find_in(col, rp[i], rp[i + 1], m);
  return p >= 0 && strong[p] && state[m] == kC;
}

template <bool LISTED>
__global__ void k_classical_count(int n, const int* __restrict__ rp, const int* __restrict__ col,
                                  const unsigned char* __restrict__ strong,
                                  const signed char* __restrict__ state, int* __restrict__ cnt,
                                  const int* __restrict__ list) {
  const int at = blockIdx.x * blockDim.x + threadIdx.x;
  if (at >= n) return;
  const int i = listed_row<LISTED>(list, at);
  if (state[i] == kC) {
    cnt[at] = 1;
    return;
  }
  int c = 0;
  for (int e = rp[i]; e < rp[i + 1]; ++e)
    if (strong[e] && state[col[e]] == kC) ++c;
  cnt[at] = c;
}

// rows longer than kClsShort are filled by a warp (k_classical_fill_warp)
constexpr int kClsShort = 8;
constexpr int kClsWarps = 4;

template <bool LISTED>
__global__ void k_classical_fill(int n, const int* __restrict__ rp,
                                 const int* __restrict__ col, const double* __restrict__ val,
                                 const int* __restrict__ dpos,
                                 const unsigned char* __restrict__ strong,
                                 const signed char* __restrict__ state,
                                 const int* __restrict__ cidx, const int* __restrict__ Prp,
                                 int* __restrict__ Pcol, double* __restrict__ Pval,
                                 const int* __restrict__ list) {
  const int at = blockIdx.x * blockDim.x + threadIdx.x;
  if (at >= n) return;
  const int i = listed_row<LISTED>(list, at);
  if (rp[i + 1] - rp[i] > kClsShort) return;  // k_classical_fill_warp
  const int p0 = Prp[at], p1 = Prp[at + 1];
  if (state[i] == kC) {
    Pcol[p0] = cidx[i];
    Pval[p0] = 1.0;
    return;
  }
  if (p0 == p1) return;
  // columns (coarse numbering keeps the fine order) and numerator start a_ij
  int q = p0;
  for (int e = rp[i]; e < rp[i + 1]; ++e)
    if (strong[e] && state[col[e]] == kC) {
      Pcol[q] = cidx[col[e]];
      Pval[q] = val[e];
      ++q;
    }
  double denom = val[dpos[i]];
  for (int e = rp[i]; e < rp[i + 1]; ++e) {
    const int k = col[e];
    if (k == i) continue;
    if (!strong[e]) {
      denom = __dadd_rn(denom, val[e]);
      continue;
    }
    if (state[k] == kC) continue;
    const double akk = val[dpos[k]];
    double s = 0.0;
    for (int f = rp[k]; f < rp[k + 1]; ++f) {
      const int m = col[f];
      if (opposite(val[f], akk) && is_strong_c(rp, col, strong, state, i, m))
        s = __dadd_rn(s, val[f]);
    }
    if (!nonzero_bits(s)) {
      denom = __dadd_rn(denom, val[e]);
      continue;
    }
    const double t = __ddiv_rn(val[e], s);
    for (int f = rp[k]; f < rp[k + 1]; ++f) {
      const int m = col[f];
      if (opposite(val[f], akk) && is_strong_c(rp, col, strong, state, i, m)) {
        int slot = find_in(Pcol, p0, p1, cidx[m]);
        Pval[slot] = __dadd_rn(Pval[slot], __dmul_rn(t, val[f]));
      }
    }
  }
  for (int s = p0; s < p1; ++s) Pval[s] = __ddiv_rn(-Pval[s], denom);
}

// The same weights for long rows, one warp per row and the same arithmetic
// in the same order: the entries of row i are visited in order (the
// denominator is a sequential sum); for a strong F neighbour k the lanes
// evaluate the selection predicate over row k in parallel, the sum s runs
// over the selected values in column order (broadcast lane by lane), and
// each selected entry updates its own weight (distinct columns of row k hit
// distinct weights, so the per-weight order of updates is unchanged).
template <bool LISTED>
__global__ void __launch_bounds__(32 * kClsWarps) k_classical_fill_warp(
    int n, const int* __restrict__ rp, const int* __restrict__ col,
    const double* __restrict__ val, const int* __restrict__ dpos,
    const unsigned char* __restrict__ strong, const signed char* __restrict__ state,
    const int* __restrict__ cidx, const int* __restrict__ Prp, int* __restrict__ Pcol,
    double* __restrict__ Pval, const int* __restrict__ list) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  for (int at = blockIdx.x * kClsWarps + w; at < n; at += gridDim.x * kClsWarps) {
    const int i = listed_row<LISTED>(list, at);
    const int r0 = rp[i], r1 = rp[i + 1];
    if (r1 - r0 <= kClsShort) continue;  // uniform over the warp
    const int p0 = Prp[at], p1 = Prp[at + 1];
    if (state[i] == kC) {
      if (lane == 0) {
        Pcol[p0] = cidx[i];
        Pval[p0] = 1.0;
      }
      continue;
    }
    if (p0 == p1) continue;
    // columns and numerator start a_ij, in row order
    int q = p0;
    for (int e0 = r0; e0 < r1; e0 += 32) {
      const int e = e0 + lane;
      const bool sel = e < r1 && strong[e] && state[col[e]] == kC;
      const unsigned m = __ballot_sync(0xffffffffu, sel);
      if (sel) {
        Pcol[q + __popc(m & below)] = cidx[col[e]];
        Pval[q + __popc(m & below)] = val[e];
      }
      q += __popc(m);
    }
    __syncwarp();
    double denom = val[dpos[i]];
    for (int e = r0; e < r1; ++e) {
      const int k = col[e];
      if (k == i) continue;
      if (!strong[e]) {
        denom = __dadd_rn(denom, val[e]);
        continue;
      }
      if (state[k] == kC) continue;
      const double akk = val[dpos[k]];
      const int f1 = rp[k + 1];
      double sk = 0.0;
      for (int f0 = rp[k]; f0 < f1; f0 += 32) {
        const int f = f0 + lane;
        bool sel = false;
        double v = 0.0;
        if (f < f1) {
          v = val[f];
          sel = opposite(v, akk) && is_strong_c(rp, col, strong, state, i, col[f]);
        }
        const unsigned m = __ballot_sync(0xffffffffu, sel);
        for (unsigned mm = m; mm; mm &= mm - 1u) {
          const int src = __ffs(mm) - 1;
          sk = __dadd_rn(sk, __shfl_sync(0xffffffffu, v, src));
        }
        if (m == 0u) continue;
      }
      if (!nonzero_bits(sk)) {
        denom = __dadd_rn(denom, val[e]);
        continue;
      }
      const double t = __ddiv_rn(val[e], sk);
      for (int f0 = rp[k]; f0 < f1; f0 += 32) {
        const int f = f0 + lane;
        if (f < f1) {
          const int m = col[f];
          if (opposite(val[f], akk) && is_strong_c(rp, col, strong, state, i, m)) {
            const int slot = find_in(Pcol, p0, p1, cidx[m]);
            Pval[slot] = __dadd_rn(Pval[slot], __dmul_rn(t, val[f]));
          }
        }
      }
      __syncwarp();
    }
    for (int sI = p0 + lane; sI < p1; sI += 32) Pval[sI] = __ddiv_rn(-Pval[sI], denom);
    __syncwarp();
  }
}

// ---------------------------------------------------- extended+i interpolation
template <bool LISTED>
__global__ void k_extpi_ub(int n, const int* __restrict__ rp,
                           const int* __restrict__ col, const unsigned char* __restrict__ strong,
                           const signed char* __restrict__ state, int* __restrict__ ub,
                           const int* __restrict__ list) {
  const int at = blockIdx.x * blockDim.x + threadIdx.x;
  if (at >= n) return;
  const int i = listed_row<LISTED>(list, at);
  if (state[i] == kC) {
    ub[at] = 1;
    return;
  }
  int u = rp[i + 1] - rp[i];
  for (int e = rp[i]; e < rp[i + 1]; ++e) {
    int k = col[e];
    if (k != i && strong[e] && state[k] != kC) u += rp[k + 1] - rp[k];
  }
  ub[at] = u;
}

__device__ __forceinline__ void insert_unique(int* __restrict__ buf, int& u, int key) {
  int lo = 0, hi = u;
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (buf[mid] < key) lo = mid + 1;
    else hi = mid;
  }
  if (lo < u && buf[lo] == key) return;
  for (int q = u; q > lo; --q) buf[q] = buf[q - 1];
  buf[lo] = key;
  ++u;
}

// rows whose candidate bound exceeds kSetShort build their set with a warp
constexpr int kSetShort = 48;
constexpr int kSetWarps = 4;
constexpr int kSetCap = 1024;   // candidates sorted in shared memory (else serial)

// interpolatory set C^_i (sorted fine indices) of every F row with at most
// kSetShort candidates: one thread per row, insertion into a sorted list
template <bool LISTED>
__global__ void k_extpi_sets(int n, const int* __restrict__ rp,
                             const int* __restrict__ col, const unsigned char* __restrict__ strong,
                             const signed char* __restrict__ state, const int* __restrict__ off,
                             const int* __restrict__ ub, int* __restrict__ buf,
                             int* __restrict__ cnt, const int* __restrict__ list) {
  const int at = blockIdx.x * blockDim.x + threadIdx.x;
  if (at >= n) return;
  const int i = listed_row<LISTED>(list, at);
  if (state[i] == kC) {
    cnt[at] = 1;
    return;
  }
  if (ub[at] > kSetShort) return;  // k_extpi_sets_warp
  int* b = buf + off[at];
  int u = 0;
  for (int e = rp[i]; e < rp[i + 1]; ++e) {
    const int k = col[e];
    if (k == i || !strong[e]) continue;
    if (state[k] == kC) {
      insert_unique(b, u, k);
    } else {
      for (int f = rp[k]; f < rp[k + 1]; ++f) {
        const int m = col[f];
        if (strong[f] && state[m] == kC && m != k) insert_unique(b, u, m);
      }
    }
  }
  cnt[at] = u;
}

// the same sets for F rows with more than kSetShort candidates, one warp per
// row: candidates (C neighbours, strong C neighbours of strong F neighbours)
// are appended to the row's buffer, then sorted (bitonic, shared memory) and
// made unique; the result is the same sorted set as the serial kernel's
template <bool LISTED>
__global__ void __launch_bounds__(32 * kSetWarps) k_extpi_sets_warp(
    int n, const int* __restrict__ rp, const int* __restrict__ col,
    const unsigned char* __restrict__ strong, const signed char* __restrict__ state,
    const int* __restrict__ off, const int* __restrict__ ub, int* __restrict__ buf,
    int* __restrict__ cnt, const int* __restrict__ list) {
  __shared__ int s_list[kSetWarps][kSetCap];
  __shared__ int s_n[kSetWarps];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  for (int at = blockIdx.x * kSetWarps + w; at < n; at += gridDim.x * kSetWarps) {
    const int i = listed_row<LISTED>(list, at);
    if (state[i] == kC || ub[at] <= kSetShort) continue;  // uniform over the warp
    int* b = buf + off[at];
    if (lane == 0) s_n[w] = 0;
    __syncwarp();
    const int r0 = rp[i], r1 = rp[i + 1];
    for (int e0 = r0; e0 < r1; e0 += 32) {
      const int e = e0 + lane;
      const bool act = e < r1;
      const int k = act ? col[e] : -1;
      const bool st = act && k != i && strong[e];
      const bool isc = st && state[k] == kC;
      const unsigned cm = __ballot_sync(0xffffffffu, isc);
      int base = 0;
      if (lane == 0) {
        base = s_n[w];
        s_n[w] = base + __popc(cm);
      }
      base = __shfl_sync(0xffffffffu, base, 0);
      if (isc) b[base + __popc(cm & below)] = k;
      __syncwarp();
      unsigned fm = __ballot_sync(0xffffffffu, st && !isc);
      while (fm) {
        const int src = __ffs(fm) - 1;
        fm &= fm - 1u;
        const int kk = __shfl_sync(0xffffffffu, k, src);
        const int f1 = rp[kk + 1];
        for (int f0 = rp[kk]; f0 < f1; f0 += 32) {
          const int f = f0 + lane;
          const bool a2 = f < f1;
          const int m = a2 ? col[f] : -1;
          const bool c2 = a2 && m != kk && strong[f] && state[m] == kC;
          const unsigned mm = __ballot_sync(0xffffffffu, c2);
          int b2 = 0;
          if (lane == 0) {
            b2 = s_n[w];
            s_n[w] = b2 + __popc(mm);
          }
          b2 = __shfl_sync(0xffffffffu, b2, 0);
          if (c2) b[b2 + __popc(mm & below)] = m;
          __syncwarp();
        }
      }
    }
    __syncwarp();
    const int total = s_n[w];
    if (total > kSetCap) {
      // rare: the serial insertion rebuilds the set from the row itself
      if (lane == 0) {
        int u = 0;
        for (int e = r0; e < r1; ++e) {
          const int k = col[e];
          if (k == i || !strong[e]) continue;
          if (state[k] == kC) {
            insert_unique(b, u, k);
          } else {
            for (int f = rp[k]; f < rp[k + 1]; ++f) {
              const int m = col[f];
              if (strong[f] && state[m] == kC && m != k) insert_unique(b, u, m);
            }
          }
        }
        cnt[at] = u;
      }
      __syncwarp();
      continue;
    }
    int P = 32;
    while (P < total) P <<= 1;
    int* L = s_list[w];
    for (int t = lane; t < P; t += 32) L[t] = t < total ? b[t] : 0x7fffffff;
    __syncwarp();
    for (int k = 2; k <= P; k <<= 1) {
      for (int j = k >> 1; j > 0; j >>= 1) {
        for (int t = lane; t < P; t += 32) {
          const int u = t ^ j;
          if (u > t) {
            const int a = L[t], c = L[u];
            const bool up = (t & k) == 0;
            if ((a > c) == up) {
              L[t] = c;
              L[u] = a;
            }
          }
        }
        __syncwarp();
      }
    }
    // unique, in order
    int outn = 0;
    for (int t0 = 0; t0 < total; t0 += 32) {
      const int t = t0 + lane;
      const bool keep = t < total && (t == 0 || L[t] != L[t - 1]);
      const unsigned km = __ballot_sync(0xffffffffu, keep);
      if (keep) b[outn + __popc(km & below)] = L[t];
      outn += __popc(km);
    }
    if (lane == 0) cnt[at] = outn;
    __syncwarp();
  }
}

// row i into [p0, p1) of P, its set C^_i in `set`
__device__ void extpi_fill_row_serial(int i, int p0, int p1, const int* __restrict__ set,
                             const int* __restrict__ rp, const int* __restrict__ col,
                             const double* __restrict__ val, const int* __restrict__ dpos,
                             const unsigned char* __restrict__ strong,
                             const signed char* __restrict__ state, const int* __restrict__ cidx,
                             int* __restrict__ Pcol, double* __restrict__ Pval) {
  if (state[i] == kC) {
    Pcol[p0] = cidx[i];
    Pval[p0] = 1.0;
    return;
  }
  if (p0 == p1) return;
  const int ns = p1 - p0;
  for (int s = 0; s < ns; ++s) {
    Pcol[p0 + s] = cidx[set[s]];
    Pval[p0 + s] = 0.0;
  }
  for (int e = rp[i]; e < rp[i + 1]; ++e) {
    int s = find_in(set, 0, ns, col[e]);
    if (s >= 0) Pval[p0 + s] = val[e];
  }
  double denom = val[dpos[i]];
  for (int e = rp[i]; e < rp[i + 1]; ++e) {
    const int k = col[e];
    if (k == i) continue;
    if (strong[e] && state[k] != kC) {
      const double akk = val[dpos[k]];
      double s = 0.0;
      double aki = 0.0;
      bool has_ki = false;
      for (int f = rp[k]; f < rp[k + 1]; ++f) {
        const int m = col[f];
        if ((m == i || find_in(set, 0, ns, m) >= 0) && opposite(val[f], akk))
          s = __dadd_rn(s, val[f]);
        if (m == i) {
          aki = val[f];
          has_ki = true;
        }
      }
      if (!nonzero_bits(s)) {
        denom = __dadd_rn(denom, val[e]);
      } else {
        const double t = __ddiv_rn(val[e], s);
        if (has_ki && opposite(aki, akk)) denom = __dadd_rn(denom, __dmul_rn(t, aki));
        for (int f = rp[k]; f < rp[k + 1]; ++f) {
          const int m = col[f];
          if (!opposite(val[f], akk)) continue;
          int slot = find_in(set, 0, ns, m);
          if (slot >= 0) Pval[p0 + slot] = __dadd_rn(Pval[p0 + slot], __dmul_rn(t, val[f]));
        }
      }
    } else if (find_in(set, 0, ns, k) >= 0) {
      // interpolated directly
    } else {
      denom = __dadd_rn(denom, val[e]);
    }
  }
  for (int s = p0; s < p1; ++s) Pval[s] = __ddiv_rn(-Pval[s], denom);
}


// Warp-per-row extended+i fill with the arithmetic order of the serial form:
// lanes evaluate the strong F neighbours' sums s_k (and t_k = a_ik / s_k)
// independently, lane 0 accumulates the denominator over row i ascending,
// and each lane owns interpolation slots, adding t_k * ahat_km over k
// ascending. Rows longer than kFillMaxE use the serial form.
constexpr int kFillMaxE = 256;
constexpr int kFillWarps = 4;
constexpr int kFillShort = 8;  // rows up to this length: one thread per row

template <bool LISTED>
__global__ void k_extpi_fill_short(int n, const int* __restrict__ rp, const int* __restrict__ col,
                                   const double* __restrict__ val, const int* __restrict__ dpos,
                                   const unsigned char* __restrict__ strong,
                                   const signed char* __restrict__ state,
                                   const int* __restrict__ cidx, const int* __restrict__ off,
                                   const int* __restrict__ buf, const int* __restrict__ Prp,
                                   int* __restrict__ Pcol, double* __restrict__ Pval,
                                 const int* __restrict__ list) {
  const int at = blockIdx.x * blockDim.x + threadIdx.x;
  if (at >= n) return;
  const int i = listed_row<LISTED>(list, at);
  if (rp[i + 1] - rp[i] > kFillShort) return;
  extpi_fill_row_serial(i, Prp[at], Prp[at + 1], buf + off[at], rp, col, val, dpos, strong, state,
                        cidx, Pcol, Pval);
}

template <bool LISTED>
__global__ void __launch_bounds__(32 * kFillWarps) k_extpi_fill_warp(
    int n, const int* __restrict__ rp, const int* __restrict__ col,
    const double* __restrict__ val, const int* __restrict__ dpos,
    const unsigned char* __restrict__ strong, const signed char* __restrict__ state,
    const int* __restrict__ cidx, const int* __restrict__ off, const int* __restrict__ buf,
    const int* __restrict__ Prp, int* __restrict__ Pcol, double* __restrict__ Pval,
    const int* __restrict__ list) {
  __shared__ double s_t[kFillWarps][kFillMaxE];
  __shared__ double s_term[kFillWarps][kFillMaxE];
  __shared__ unsigned char s_flag[kFillWarps][kFillMaxE];
  __shared__ unsigned char s_akc[kFillWarps][kFillMaxE];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int at = blockIdx.x * kFillWarps + w;
  if (at >= n) return;
  const int i = listed_row<LISTED>(list, at);
  if (rp[i + 1] - rp[i] <= kFillShort) return;  // done by k_extpi_fill_short
  const int p0 = Prp[at], p1 = Prp[at + 1];
  if (state[i] == kC) {
    if (lane == 0) {
      Pcol[p0] = cidx[i];
      Pval[p0] = 1.0;
    }
    return;
  }
  if (p0 == p1) return;
  const int r0 = rp[i], r1 = rp[i + 1];
  if (r1 - r0 > kFillMaxE) {
    if (lane == 0)
      extpi_fill_row_serial(i, p0, p1, buf + off[at], rp, col, val, dpos, strong, state, cidx, Pcol,
                            Pval);
    return;
  }
  const int* set = buf + off[at];
  const int ns = p1 - p0;
  double* t = s_t[w];
  double* term = s_term[w];
  unsigned char* flag = s_flag[w];
  unsigned char* akc = s_akc[w];
  // flags: 0 skip (diagonal or interpolated directly), 1 lump a_ie into the
  // denominator, 3 strong F neighbour with t_k (term = t_k ahat_ki or 0)
  for (int e = r0 + lane; e < r1; e += 32) {
    const int q = e - r0;
    const int k = col[e];
    unsigned char fl = 0, kc = 0;
    double tk = 0.0, tm = 0.0;
    if (k == i) {
      fl = 0;
    } else if (strong[e] && state[k] != kC) {
      kc = sign_class(val[dpos[k]]);
      double sk = 0.0, aki = 0.0;
      bool has_ki = false;
      for (int f = rp[k]; f < rp[k + 1]; ++f) {
        const int m = col[f];
        const double v = val[f];
        // the sign test first: it skips most of the set searches
        if (opposite_class(v, kc) && (m == i || find_in(set, 0, ns, m) >= 0)) sk = __dadd_rn(sk, v);
        if (m == i) {
          aki = v;
          has_ki = true;
        }
      }
      if (!nonzero_bits(sk)) {
        fl = 1;
      } else {
        fl = 3;
        tk = __ddiv_rn(val[e], sk);
        if (has_ki && opposite_class(aki, kc)) tm = __dmul_rn(tk, aki);
      }
    } else if (find_in(set, 0, ns, k) >= 0) {
      fl = 0;
    } else {
      fl = 1;
    }
    flag[q] = fl;
    t[q] = tk;
    term[q] = tm;
    akc[q] = kc;
  }
  __syncwarp();
  double denom = 0.0;
  if (lane == 0) {
    denom = val[dpos[i]];
    for (int e = r0; e < r1; ++e) {
      const int q = e - r0;
      if (flag[q] == 1) denom = __dadd_rn(denom, val[e]);
      else if (flag[q] == 3 && nonzero_bits(term[q])) denom = __dadd_rn(denom, term[q]);
    }
  }
  denom = __shfl_sync(0xffffffffu, denom, 0);
  for (int sl = lane; sl < ns; sl += 32) {
    const int m = set[sl];
    const int pe = find_in(col, r0, r1, m);
    double num = pe >= 0 ? val[pe] : 0.0;
    for (int e = r0; e < r1; ++e) {
      const int q = e - r0;
      if (flag[q] != 3) continue;
      const int k = col[e];
      const int f = find_in(col, rp[k], rp[k + 1], m);
      if (f >= 0 && opposite_class(val[f], akc[q])) num = __dadd_rn(num, __dmul_rn(t[q], val[f]));
    }
    Pcol[p0 + sl] = cidx[m];
    Pval[p0 + sl] = __ddiv_rn(-num, denom);
  }
}

// --------------------------------------------------- interpolation truncation
constexpr int kPmaxLimit = 16;

__global__ void k_trunc_count(int n, const int* __restrict__ Prp, int pmax, int* __restrict__ cnt) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int len = Prp[i + 1] - Prp[i];
  cnt[i] = len < pmax ? len : pmax;
}

// keep the pmax largest |w| (ties to the lower column) and scale them by
// (sum of all) / (sum of kept), sums over the row ascending from 0.0; the result
// at Trp[i], or for listed rows at list[i] * pmax with its length in Tcnt[list[i]]
__global__ void k_trunc_fill(int n, const int* __restrict__ list, const int* __restrict__ Prp,
                             const int* __restrict__ Pcol, const double* __restrict__ Pval,
                             int pmax, const int* __restrict__ Trp, int* __restrict__ Tcnt,
                             int* __restrict__ Tcol, double* __restrict__ Tval) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int p0 = Prp[i], p1 = Prp[i + 1], len = p1 - p0;
  const long long t0 = list ? (long long)list[i] * pmax : Trp[i];
  if (list) Tcnt[list[i]] = len < pmax ? len : pmax;
  if (len <= pmax) {
    for (int q = 0; q < len; ++q) {
      Tcol[t0 + q] = Pcol[p0 + q];
      Tval[t0 + q] = Pval[p0 + q];
    }
    return;
  }
  int keep[kPmaxLimit];
  int nk = 0;
  for (int r = 0; r < pmax; ++r) {
    int best = -1;
    unsigned long long bw = 0;
    for (int q = 0; q < len; ++q) {
      bool taken = false;
      for (int u = 0; u < nk; ++u) taken |= keep[u] == q;
      if (taken) continue;
      const unsigned long long a = mag_key(Pval[p0 + q]);
      if (best < 0 || a > bw) {  // first maximum in column order wins ties
        bw = a;
        best = q;
      }
    }
    keep[nk++] = best;
  }
  for (int a = 1; a < nk; ++a) {  // ascending position = ascending column
    int v = keep[a], b = a - 1;
    while (b >= 0 && keep[b] > v) {
      keep[b + 1] = keep[b];
      --b;
    }
    keep[b + 1] = v;
  }
  double s_all = 0.0, s_keep = 0.0;
  for (int q = 0; q < len; ++q) s_all = __dadd_rn(s_all, Pval[p0 + q]);
  for (int u = 0; u < nk; ++u) s_keep = __dadd_rn(s_keep, Pval[p0 + keep[u]]);
  const double f = s_keep != 0.0 ? __ddiv_rn(s_all, s_keep) : 1.0;
  for (int u = 0; u < nk; ++u) {
    Tcol[t0 + u] = Pcol[p0 + keep[u]];
    Tval[t0 + u] = s_keep != 0.0 ? __dmul_rn(Pval[p0 + keep[u]], f) : Pval[p0 + keep[u]];
  }
}

// ------------------------------------------------------------- transpose
// entries per column, and every entry's place among its column's (in no
// particular order)
__global__ void k_count_cols(int n, const int* __restrict__ rp, const int* __restrict__ col,
                             int* __restrict__ cnt, int* __restrict__ place) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  for (int e = rp[i]; e < rp[i + 1]; ++e) place[e] = atomicAdd(&cnt[col[e]], 1);
}

__global__ void k_fill_transpose(int n, const int* __restrict__ rp, const int* __restrict__ col,
                                 const double* __restrict__ val, const int* __restrict__ Trp,
                                 const int* __restrict__ place, int* __restrict__ Tcol,
                                 double* __restrict__ Tval) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  for (int e = rp[i]; e < rp[i + 1]; ++e) {
    const int q = Trp[col[e]] + place[e];
    Tcol[q] = i;
    Tval[q] = val[e];
  }
}

// Rows of [rp] with distinct columns, reordered by column from (col, val)
// into (ocol, oval): each entry goes to its rank, the number of entries of
// its row with a smaller column. One warp per row of more than 32 entries
// (the lanes rank the row's entries in parallel), one thread per shorter
// row.
__global__ void k_rank_rows(int n, const int* __restrict__ rp, const int* __restrict__ col,
                            const double* __restrict__ val, int* __restrict__ ocol,
                            double* __restrict__ oval) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int r0 = rp[i], r1 = rp[i + 1];
  if (r1 - r0 > 32) return;  // k_rank_rows_warp
  for (int e = r0; e < r1; ++e) {
    const int c = col[e];
    int rank = 0;
    for (int f = r0; f < r1; ++f) rank += col[f] < c;
    ocol[r0 + rank] = c;
    oval[r0 + rank] = val[e];
  }
}

__global__ void k_rank_rows_warp(int n, const int* __restrict__ rp, const int* __restrict__ col,
                                 const double* __restrict__ val, int* __restrict__ ocol,
                                 double* __restrict__ oval) {
  const int lane = threadIdx.x & 31;
  const int i = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  if (i >= n) return;
  const int r0 = rp[i], r1 = rp[i + 1];
  if (r1 - r0 <= 32) return;  // k_rank_rows
  for (int e = r0 + lane; e < r1; e += 32) {
    const int c = col[e];
    int rank = 0;
    for (int f = r0; f < r1; ++f) rank += col[f] < c;
    ocol[r0 + rank] = c;
    oval[r0 + rank] = val[e];
  }
}

// ------------------------------------------------------------ smoother scaling
// l1-Jacobi scaling d_i = sign(a_ii) (|a_ii| + sum_{j != i} |a_ij|): coarse
// Galerkin operators of the advective S~_T can have a few negative diagonals
__global__ void k_l1_dinv(int n, const int* __restrict__ rp, const int* __restrict__ col,
                          const double* __restrict__ val, double* __restrict__ dinv,
                          float* __restrict__ dinvf, int* __restrict__ err) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double diag = 0.0, off = 0.0;
  for (int e = rp[i]; e < rp[i + 1]; ++e) {
    if (col[e] == i) diag = val[e];
    else off += fabs(val[e]);
  }
  double s = diag >= 0.0 ? diag + off : diag - off;
  if (s == 0.0 || !isfinite(s)) {
    atomicOr(err, 4);
    s = 1.0;
  }
  dinv[i] = 1.0 / s;
  if (dinvf) dinvf[i] = (float)(1.0 / s);
}

__global__ void k_to_float(long long n, const double* __restrict__ a, float* __restrict__ b) {
  long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) b[i] = (float)a[i];
}

// round to nearest even BF16 (interpolation weights of precision 2)
__global__ void k_to_bf16(long long n, const double* __restrict__ a,
                          __nv_bfloat16* __restrict__ b) {
  long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) b[i] = __float2bfloat16_rn((float)a[i]);
}

// ------------------------------------------------ vertical-line smoother
// Thomas factorisation of each column's tridiagonal part (Gaussian
// elimination without pivoting on a tridiagonal matrix): m_0 = d_0,
// m_k = d_k - l_k (u_{k-1} / m_{k-1}); stores l_k, 1 / m_k and u_k / m_k.
// Correctly rounded operations in the oracle's order (no FMA contraction).
// Twisted factorisation of each column's tridiagonal part (diagonal d_k,
// lower l_k, upper u_k; layer k of column c is cell c + nxy k), so that two
// threads can solve a column from both ends at once (k_line_block). With
// mid = nz / 2: the top rows k < mid are eliminated downwards (m_k = d_k -
// l_k cp_{k-1}, cp_k = u_k / m_k), the bottom rows k > mid upwards (q_k =
// d_k - u_k cq_{k+1}, cq_k = l_k / q_k), and the middle row takes both sides
// (pivot d - l cp_{mid-1} - u cq_{mid+1}). Stored per cell: lo = the
// coupling to the row eliminated before it (l_k on top, u_k below, l_mid in
// the middle), minv = 1 / pivot, cp = cp_k on top, cq_k below, u_mid in the
// middle.
__device__ __forceinline__ void line_row(int i, int nxy, const int* __restrict__ rp,
                                         const int* __restrict__ col,
                                         const double* __restrict__ val, double& d, double& l,
                                         double& u, bool& has_lo, bool& has_up) {
  d = l = u = 0.0;
  has_lo = has_up = false;
  for (int e = rp[i]; e < rp[i + 1]; ++e) {
    const int j = col[e];
    if (j == i) d = val[e];
    else if (j == i - nxy) { l = val[e]; has_lo = true; }
    else if (j == i + nxy) { u = val[e]; has_up = true; }
  }
}

__global__ void k_line_factor(int nxy, int nz, const int* __restrict__ rp,
                              const int* __restrict__ col, const double* __restrict__ val,
                              double* __restrict__ lo, double* __restrict__ minv,
                              double* __restrict__ cp, float* __restrict__ lof,
                              float* __restrict__ minvf, float* __restrict__ cpf,
                              int* __restrict__ err) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= nxy) return;
  const int mid = nz >> 1;
  auto store = [&](int i, double a, double mi, double q) {
    lo[i] = a;
    minv[i] = mi;
    cp[i] = q;
    if (lof) {
      lof[i] = (float)a;
      minvf[i] = (float)mi;
      cpf[i] = (float)q;
    }
  };
  auto pivot_ok = [&](double m) {
    const bool ok = m != 0.0 && isfinite(m);
    if (!ok) atomicOr(err, 16);
    return ok;
  };
  double d, l, u;
  bool has_lo, has_up;
  double cprev = 0.0;  // top: cp_{k-1}
  for (int k = 0; k < mid; ++k) {
    const int i = c + k * nxy;
    line_row(i, nxy, rp, col, val, d, l, u, has_lo, has_up);
    if (has_lo != (k > 0) || has_up != (k < nz - 1)) atomicOr(err, 16);
    const double m = __dsub_rn(d, __dmul_rn(l, cprev));
    double mi = 0.0, q = 0.0;
    if (pivot_ok(m)) {
      mi = __ddiv_rn(1.0, m);
      q = __ddiv_rn(u, m);
    }
    store(i, l, mi, q);
    cprev = q;
  }
  double cnext = 0.0;  // bottom: cq_{k+1}
  for (int k = nz - 1; k > mid; --k) {
    const int i = c + k * nxy;
    line_row(i, nxy, rp, col, val, d, l, u, has_lo, has_up);
    if (has_lo != (k > 0) || has_up != (k < nz - 1)) atomicOr(err, 16);
    const double m = __dsub_rn(d, __dmul_rn(u, cnext));
    double mi = 0.0, q = 0.0;
    if (pivot_ok(m)) {
      mi = __ddiv_rn(1.0, m);
      q = __ddiv_rn(l, m);
    }
    store(i, u, mi, q);
    cnext = q;
  }
  const int i = c + mid * nxy;
  line_row(i, nxy, rp, col, val, d, l, u, has_lo, has_up);
  if (has_lo != (mid > 0) || has_up != (mid < nz - 1)) atomicOr(err, 16);
  const double m = __dsub_rn(__dsub_rn(d, __dmul_rn(l, cprev)), __dmul_rn(u, cnext));
  double mi = 0.0;
  if (pivot_ok(m)) mi = __ddiv_rn(1.0, m);
  store(i, l, mi, u);
}

void line_setup(Level& v, int nxy, int nz, Pool& pool, bool f32, int* err, bool allocate,
                cudaStream_t s) {
  const int n = v.A.n;
  if ((long long)nxy * nz != n) fail(TP_EINVAL, "line smoother: level is not the grid");
  if (allocate) {
    v.line_lo = pool.alloc<double>(n);
    v.line_minv = pool.alloc<double>(n);
    v.line_cp = pool.alloc<double>(n);
    if (f32) {
      v.line_lof = pool.alloc<float>(n);
      v.line_minvf = pool.alloc<float>(n);
      v.line_cpf = pool.alloc<float>(n);
    }
  }
  k_line_factor<<<grid_for(nxy), kBlock, 0, s>>>(nxy, nz, v.A.rowptr, v.A.col, v.A.val,
                                                 v.line_lo, v.line_minv, v.line_cp, v.line_lof,
                                                 v.line_minvf, v.line_cpf, err);
  TP_LAUNCH_CHECK();
}

// -------------------------------------------------------- sliced-ELL copy
// One block per window of kSellWindow rows: the rows sorted by descending
// length (ties by ascending row) with a block bitonic sort; slice widths
// are the lengths of each slice's first (longest) row.
__global__ void __launch_bounds__(kSellWindow) k_sell_perm(int n, const int* __restrict__ rp,
                                                           int* __restrict__ perm,
                                                           int* __restrict__ width32) {
  __shared__ unsigned long long key[kSellWindow];
  const int t = threadIdx.x;
  const int r = blockIdx.x * kSellWindow + t;
  unsigned long long k = ~0ull;  // slots past n sort last
  if (r < n) {
    const int len = rp[r + 1] - rp[r];
    k = ((unsigned long long)(unsigned)(0x7fffffff - len) << 32) | (unsigned)r;
  }
  key[t] = k;
  __syncthreads();
  for (int size = 2; size <= kSellWindow; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      const int partner = t ^ stride;
      if (partner > t) {
        const bool up = (t & size) == 0;
        const unsigned long long a = key[t], c = key[partner];
        if ((a > c) == up) {
          key[t] = c;
          key[partner] = a;
        }
      }
      __syncthreads();
    }
  }
  const unsigned long long kk = key[t];
  const int row = kk == ~0ull ? -1 : (int)(kk & 0xffffffffu);
  perm[r] = row;
  if ((t & 31) == 0) width32[r >> 5] = row >= 0 ? 32 * (rp[row + 1] - rp[row]) : 0;
}

// slot t of slice s: the entries of its row, padded to the slice width
__global__ void k_sell_fill(int nslots, const int* __restrict__ rp, const int* __restrict__ col,
                            const double* __restrict__ val, const int* __restrict__ perm,
                            const int* __restrict__ ptr, int* __restrict__ scol,
                            double* __restrict__ sval, float* __restrict__ svalf) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nslots) return;
  const int sl = t >> 5, lane = t & 31;
  const int row = perm[t];
  const int w = (ptr[sl + 1] - ptr[sl]) >> 5;
  const int e0 = row >= 0 ? rp[row] : 0, len = row >= 0 ? rp[row + 1] - e0 : 0;
  for (int k = 0; k < w; ++k) {
    const long long q = (long long)ptr[sl] + 32 * k + lane;
    const bool has = k < len;
    if (scol) scol[q] = has ? col[e0 + k] : (row >= 0 ? row : 0);
    const double v = has ? val[e0 + k] : 0.0;
    sval[q] = v;
    if (svalf) svalf[q] = (float)v;
  }
}

// --------------------------------------------------------------- ELL copy
__global__ void k_max_row(int n, const int* __restrict__ rp, int* __restrict__ mx) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) atomicMax(mx, rp[i + 1] - rp[i]);
}

__global__ void k_to_ell(int n, int w, const int* __restrict__ rp, const int* __restrict__ col,
                         const double* __restrict__ val, int* __restrict__ ecol,
                         double* __restrict__ eval, float* __restrict__ evalf) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int r0 = rp[i], len = rp[i + 1] - r0;
  for (int k = 0; k < w; ++k) {
    const long long q = (long long)k * n + i;
    const bool has = k < len;
    if (ecol) ecol[q] = has ? col[r0 + k] : i;
    const double v = has ? val[r0 + k] : 0.0;
    eval[q] = v;
    if (evalf) evalf[q] = (float)v;
  }
}

// ELL copy by grid direction (the finest level of a grid's 7-point operator):
// slot k of row i holds the entry at column i + (-nxy, -nx, -1, 0, +1, +nx,
// +nxy)[k], 0 where the row has none; an entry at any other offset sets
// bit 32 of *err (the level is not the grid's 7-point pattern)
__global__ void k_to_stencil(int n, int nx, int nxy, const int* __restrict__ rp,
                             const int* __restrict__ col, const double* __restrict__ val,
                             double* __restrict__ eval, float* __restrict__ evalf,
                             int* __restrict__ err) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double v[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (int e = rp[i]; e < rp[i + 1]; ++e) {
    const int d = col[e] - i;
    const int k = d == -nxy ? 0 : d == -nx ? 1 : d == -1 ? 2 : d == 0 ? 3 : d == 1 ? 4
                : d == nx ? 5 : d == nxy ? 6 : -1;
    if (k < 0) {
      atomicOr(err, 32);
      continue;
    }
    v[k] = val[e];
  }
#pragma unroll
  for (int k = 0; k < 7; ++k) {
    const long long q = (long long)k * n + i;
    eval[q] = v[k];
    if (evalf) evalf[q] = (float)v[k];
  }
}

// ------------------------------------------------------------ coarsest level
// the entries of a CSR matrix into a zeroed dense one, one warp per row
__global__ void k_to_dense(int n, const int* __restrict__ rp, const int* __restrict__ col,
                           const double* __restrict__ val, double* __restrict__ D) {
  const int i = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  if (i >= n) return;
  for (int e = rp[i] + (threadIdx.x & 31); e < rp[i + 1]; e += 32)
    D[(long long)i * n + col[e]] = 0.0 + val[e];
}

// Gauss-Jordan elimination with partial pivoting on [A | I] (one block):
// leaves A^{-1} in inv. Pivot: largest |a_ik| over rows >= k, lowest row on
// ties. A zero pivot sets err.
__global__ void k_gauss_jordan(int n, double* __restrict__ A, double* __restrict__ inv,
                               int* __restrict__ err) {
  __shared__ double s_val[1024];
  __shared__ int s_idx[1024];
  __shared__ int s_piv;
  const int tid = threadIdx.x, nt = blockDim.x;
  for (long long q = tid; q < (long long)n * n; q += nt) inv[q] = ((q / n) == (q % n)) ? 1.0 : 0.0;
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    double best = -1.0;
    int bi = n;
    for (int i = k + tid; i < n; i += nt) {
      double a = fabs(A[(long long)i * n + k]);
      if (a > best || (a == best && i < bi)) {
        best = a;
        bi = i;
      }
    }
    s_val[tid] = best;
    s_idx[tid] = bi;
    __syncthreads();
    for (int o = nt / 2; o > 0; o >>= 1) {
      if (tid < o) {
        double a = s_val[tid + o];
        int ai = s_idx[tid + o];
        if (a > s_val[tid] || (a == s_val[tid] && ai < s_idx[tid])) {
          s_val[tid] = a;
          s_idx[tid] = ai;
        }
      }
      __syncthreads();
    }
    if (tid == 0) {
      s_piv = s_idx[0];
      if (!(s_val[0] > 0.0)) *err = 1;
    }
    __syncthreads();
    if (*err) return;
    const int p = s_piv;
    if (p != k) {
      for (int j = tid; j < n; j += nt) {
        double t = A[(long long)k * n + j];
        A[(long long)k * n + j] = A[(long long)p * n + j];
        A[(long long)p * n + j] = t;
        t = inv[(long long)k * n + j];
        inv[(long long)k * n + j] = inv[(long long)p * n + j];
        inv[(long long)p * n + j] = t;
      }
    }
    __syncthreads();
    const double piv = A[(long long)k * n + k];
    __syncthreads();
    for (int j = tid; j < n; j += nt) {
      A[(long long)k * n + j] /= piv;
      inv[(long long)k * n + j] /= piv;
    }
    __syncthreads();
    for (long long q = tid; q < (long long)n * n; q += nt) {
      int i = (int)(q / n), j = (int)(q % n);
      if (i == k) continue;
      double f = A[(long long)i * n + k];
      if (j == k) continue;  // column k of A is cleared below
      A[(long long)i * n + j] -= f * A[(long long)k * n + j];
      inv[(long long)i * n + j] -= f * inv[(long long)k * n + j];
    }
    __syncthreads();
    // inv column k and A column k for rows != k
    for (int i = tid; i < n; i += nt) {
      if (i == k) continue;
      double f = A[(long long)i * n + k];
      inv[(long long)i * n + k] -= f * inv[(long long)k * n + k];
      A[(long long)i * n + k] = 0.0;
    }
    __syncthreads();
  }
}

// threads per CSR row in the V-cycle kernels: a power of two giving each
// lane about 4 entries (fewer lanes mean fewer shuffle steps per row, more
// mean more parallelism on short coarse levels), halved while the launch
// would exceed four waves of resident threads, but not below the width that
// leaves each lane at most 12 entries. FGMRES solve time on GB300 (FP64,
// ms; layered 256x256x64 / grf 64x64x32 / channelised 128x128x64): this
// rule 183.4 / 11.5 / 41.5; halving down to one lane (the rule of the
// smaller grids, where level 1 of the layered A_pp, 1.25 M rows of 29.5
// entries, ran with one lane) 200.2 / 11.4 / 42.5; floors of 8 or 16
// entries 186.5-188.8 / 11.4-11.5 / 41.5-42.4.
int pick_lanes(const DevCSR& A) {
  const long long resident = resident_threads();
  const double avg = A.n > 0 ? (double)A.nnz / A.n : 1.0;
  int l = 1;
  while (l * 4.0 <= avg && l < 32) l *= 2;
  int lmin = 1;
  while (lmin < 32 && avg / lmin > 12.0) lmin *= 2;
  while (l > lmin && (long long)A.n * l > 4 * resident) l /= 2;
  // at most 16 lanes: a 32-lane row's five FP64 reduction adds occupy the
  // FP64 pipe for the whole warp (A_pp's level 3 on the layered workload:
  // 34 k rows x 92 entries). Layered 256x256x64 FGMRES 140.4 -> 138.2 ms
  // (FP64), 95.1 -> 94.6 ms (FP32); channelised and grf 64x64x32 within
  // noise; at most 8 lanes: 140.0 ms, grf +0.6 ms
  return l > 16 ? 16 : l;
}

// threads resident on the whole device at full occupancy
long long resident_threads() {
  static PerDevice<long long> threads;
  return threads([] {
    int dev = 0, thr = 0;
    TP_CUDA_TRY(cudaGetDevice(&dev));
    TP_CUDA_TRY(cudaDeviceGetAttribute(&thr, cudaDevAttrMaxThreadsPerMultiProcessor, dev));
    return (long long)device_sms() * thr;
  });
}

int read_int(const int* d, cudaStream_t s) {
  int h = 0;
  TP_CUDA_TRY(cudaMemcpyAsync(&h, d, sizeof(int), cudaMemcpyDeviceToHost, s));
  TP_CUDA_TRY(cudaStreamSynchronize(s));
  return h;
}

DevCSR transpose(const DevCSR& P, Pool& pool, Pool& scratch, cudaStream_t s) {
  DevCSR R;
  R.n = P.m;
  R.m = P.n;
  R.nnz = P.nnz;
  int* cnt = scratch.alloc<int>(R.n + 1);
  int* place = scratch.alloc<int>(R.nnz + 1);
  TP_CUDA_TRY(cudaMemsetAsync(cnt, 0, sizeof(int) * (R.n + 1), s));
  k_count_cols<<<grid_for(P.n), kBlock, 0, s>>>(P.n, P.rowptr, P.col, cnt, place);
  TP_LAUNCH_CHECK();
  R.rowptr = pool.alloc<int>(R.n + 1);
  scan_exclusive(cnt, R.rowptr, R.n, scratch, s);
  R.col = pool.alloc<int>(R.nnz + 1);
  R.val = pool.alloc<double>(R.nnz + 1);
  // atomically placed (unordered) entries, then each row ranked by column
  int* ucol = scratch.alloc<int>(R.nnz + 1);
  double* uval = scratch.alloc<double>(R.nnz + 1);
  k_fill_transpose<<<grid_for(P.n), kBlock, 0, s>>>(P.n, P.rowptr, P.col, P.val, R.rowptr,
                                                    place, ucol, uval);
  TP_LAUNCH_CHECK();
  k_rank_rows<<<grid_for(R.n), kBlock, 0, s>>>(R.n, R.rowptr, ucol, uval, R.col, R.val);
  TP_LAUNCH_CHECK();
  k_rank_rows_warp<<<grid_for((long long)R.n * 32), kBlock, 0, s>>>(R.n, R.rowptr, ucol, uval,
                                                                    R.col, R.val);
  TP_LAUNCH_CHECK();
  return R;
}

}  // namespace

template <bool LISTED>
static DevCSR interpolation_rows(const DevCSR& A, bool extended, const int* dpos,
                                 const unsigned char* strong, const signed char* state,
                                 const int* cidx, int nc, const int* list, int rows, Pool& pool,
                                 Pool& scratch, cudaStream_t s) {
  const auto warp_blocks = [rows](int warps) {
    return (int)std::min(((long long)rows + warps - 1) / warps, 8LL * device_sms());
  };
  DevCSR P;
  P.n = rows;
  P.m = nc;
  P.rowptr = pool.alloc<int>(rows + 1);
  int* cnt = scratch.alloc<int>(rows + 1);
  const int blocks = grid_for(rows), blocks128 = grid_for(rows, 128);
  if (!extended) {
    k_classical_count<LISTED><<<blocks, kBlock, 0, s>>>(rows, A.rowptr, A.col, strong, state, cnt,
                                                        list);
    TP_LAUNCH_CHECK();
    P.nnz = (int)scan_exclusive(cnt, P.rowptr, rows, scratch, s);
    P.col = pool.alloc<int>(P.nnz);
    P.val = pool.alloc<double>(P.nnz);
    k_classical_fill<LISTED><<<blocks128, 128, 0, s>>>(rows, A.rowptr, A.col, A.val, dpos, strong,
                                                       state, cidx, P.rowptr, P.col, P.val, list);
    TP_LAUNCH_CHECK();
    k_classical_fill_warp<LISTED><<<warp_blocks(kClsWarps), 32 * kClsWarps, 0, s>>>(
        rows, A.rowptr, A.col, A.val, dpos, strong, state, cidx, P.rowptr, P.col, P.val, list);
    TP_LAUNCH_CHECK();
    return P;
  }
  int* ub = scratch.alloc<int>(rows + 1);
  int* off = scratch.alloc<int>(rows + 1);
  k_extpi_ub<LISTED><<<blocks, kBlock, 0, s>>>(rows, A.rowptr, A.col, strong, state, ub, list);
  TP_LAUNCH_CHECK();
  const long long tot = scan_exclusive(ub, off, rows, scratch, s);
  int* buf = scratch.alloc<int>(tot + 1);
  k_extpi_sets<LISTED><<<blocks128, 128, 0, s>>>(rows, A.rowptr, A.col, strong, state, off, ub, buf,
                                                 cnt, list);
  TP_LAUNCH_CHECK();
  k_extpi_sets_warp<LISTED><<<warp_blocks(kSetWarps), 32 * kSetWarps, 0, s>>>(
      rows, A.rowptr, A.col, strong, state, off, ub, buf, cnt, list);
  TP_LAUNCH_CHECK();
  P.nnz = (int)scan_exclusive(cnt, P.rowptr, rows, scratch, s);
  P.col = pool.alloc<int>(P.nnz);
  P.val = pool.alloc<double>(P.nnz);
  k_extpi_fill_short<LISTED><<<blocks128, 128, 0, s>>>(rows, A.rowptr, A.col, A.val, dpos, strong,
                                                       state, cidx, off, buf, P.rowptr, P.col,
                                                       P.val, list);
  TP_LAUNCH_CHECK();
  k_extpi_fill_warp<LISTED><<<(rows + kFillWarps - 1) / kFillWarps, 32 * kFillWarps, 0, s>>>(
      rows, A.rowptr, A.col, A.val, dpos, strong, state, cidx, off, buf, P.rowptr, P.col, P.val,
      list);
  TP_LAUNCH_CHECK();
  return P;
}

DevCSR untruncated_interpolation(const DevCSR& A, bool extended, const int* dpos,
                                 const unsigned char* strong, const signed char* state,
                                 const int* cidx, int nc, const int* list, int rows, Pool& pool,
                                 Pool& scratch, cudaStream_t s) {
  return list ? interpolation_rows<true>(A, extended, dpos, strong, state, cidx, nc, list, rows,
                                         pool, scratch, s)
              : interpolation_rows<false>(A, extended, dpos, strong, state, cidx, nc, list, rows,
                                          pool, scratch, s);
}

void truncate_listed_rows(const DevCSR& P, const int* list, int pmax, int* cnt, int* tcol,
                          double* tval, cudaStream_t s) {
  k_trunc_fill<<<grid_for(P.n), kBlock, 0, s>>>(P.n, list, P.rowptr, P.col, P.val, pmax, nullptr,
                                                cnt, tcol, tval);
  TP_LAUNCH_CHECK();
}

// P with its rows cut to the pmax largest weights
static DevCSR truncated(const DevCSR& P, int pmax, Pool& pool, Pool& scratch, cudaStream_t s) {
  DevCSR T;
  T.n = P.n;
  T.m = P.m;
  T.rowptr = pool.alloc<int>(P.n + 1);
  int* cnt = scratch.alloc<int>(P.n + 1);
  k_trunc_count<<<grid_for(P.n), kBlock, 0, s>>>(P.n, P.rowptr, pmax, cnt);
  TP_LAUNCH_CHECK();
  T.nnz = (int)scan_exclusive(cnt, T.rowptr, P.n, scratch, s);
  T.col = pool.alloc<int>(T.nnz + 1);
  T.val = pool.alloc<double>(T.nnz + 1);
  k_trunc_fill<<<grid_for(P.n), kBlock, 0, s>>>(P.n, nullptr, P.rowptr, P.col, P.val, pmax,
                                                T.rowptr, nullptr, T.col, T.val);
  TP_LAUNCH_CHECK();
  return T;
}

void csr_transpose_positions(const DevCSR& A, int* tpos, int* err, cudaStream_t s) {
  if (A.n > 0 && A.nnz >= (long long)kWarpRowMean * A.n)
    k_transpose_pos_warp<<<grid_for((long long)A.n * 32), kBlock, 0, s>>>(A.n, A.rowptr, A.col,
                                                                         tpos, err);
  else
    k_transpose_pos<<<grid_for(A.n), kBlock, 0, s>>>(A.n, A.rowptr, A.col, tpos, err);
  TP_LAUNCH_CHECK();
}

Hierarchy::~Hierarchy() {
  for (cudaEvent_t e : phase_ev) cudaEventDestroy(e);
}

double Hierarchy::operator_complexity() const {
  if (L.empty() || L[0].A.nnz == 0) return 0.0;
  double s = 0.0;
  for (const Level& l : L) s += l.A.nnz;
  return s / L[0].A.nnz;
}

// phase boundaries as events on the setup's stream, read once at its end (a
// host clock would need the stream to drain at each of them)
void Hierarchy::mark_phase(int phase, cudaStream_t s) {
  if (marks.size() == phase_ev.size()) {
    cudaEvent_t e = nullptr;
    TP_CUDA_TRY(cudaEventCreate(&e));
    phase_ev.push_back(e);
  }
  TP_CUDA_TRY(cudaEventRecord(phase_ev[marks.size()], s));
  marks.push_back(phase);
}

void Hierarchy::read_phases() {
  for (double& x : phase_ms) x = 0.0;
  for (size_t q = 1; q < marks.size(); ++q) {
    float ms = 0.f;
    TP_CUDA_TRY(cudaEventElapsedTime(&ms, phase_ev[q - 1], phase_ev[q]));
    phase_ms[marks[q]] += ms;
  }
}

void Hierarchy::setup(const DevCSR& A0, const AmgOpts& o, cudaStream_t s) {
  opts = o;
  marks.clear();
  mark_phase(0, s);
  pool.release();
  scratch.release();
  L.clear();
  coarse_inv = nullptr;
  cheb_partials = nullptr;
  tail_first = -1;
  err = pool.alloc<int>(2);
  TP_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int), s));
  L.emplace_back();
  L[0].A = A0;
  n0 = A0.n;
  while (true) {
    Level& cur = L.back();
    const DevCSR& A = cur.A;
    const int n = A.n;
    cur.dpos = pool.alloc<int>(n);
    k_diag_pos<<<grid_for(n), kBlock, 0, s>>>(n, A.rowptr, A.col, cur.dpos, err);
    TP_LAUNCH_CHECK();
    const bool coarsest = n <= opts.coarse_size || (int)L.size() >= opts.max_levels;
    if (!coarsest) {
      // transpose positions do not depend on the diagonal: both checks are
      // read back with one synchronisation
      cur.tpos = pool.alloc<int>(A.nnz);
      csr_transpose_positions(A, cur.tpos, err, s);
    }
    {
      const int e = read_int(err, s);
      if (e & 1) fail(TP_EINVAL, "AMG: a row has no diagonal entry");
      if (e & 2) fail(TP_EINVAL, "AMG: pattern is not structurally symmetric");
    }
    if (coarsest) break;
    // long rows (coarse Galerkin levels): one warp per row
    const bool wrow = A.nnz >= (long long)kWarpRowMean * n;
    const int gw = grid_for((long long)n * 32);
    cur.strong = pool.alloc<unsigned char>(A.nnz);
    const int g8 = grid_for((long long)n * 8);
    if (wrow)
      k_strength<32><<<gw, kBlock, 0, s>>>(n, A.rowptr, A.col, A.val, opts.theta, cur.strong);
    else
      k_strength<8><<<g8, kBlock, 0, s>>>(n, A.rowptr, A.col, A.val, opts.theta, cur.strong);
    TP_LAUNCH_CHECK();
    // PMIS
    int* lam = scratch.alloc<int>(n);
    unsigned char* newc = scratch.alloc<unsigned char>(n);
    int* undecided = scratch.alloc<int>(1);
    cur.cf = pool.alloc<signed char>(n);
    if (wrow)
      k_pmis_init<32><<<gw, kBlock, 0, s>>>(n, A.rowptr, A.col, cur.strong, cur.tpos, lam, cur.cf,
                                            newc);
    else
      k_pmis_init<8><<<g8, kBlock, 0, s>>>(n, A.rowptr, A.col, cur.strong, cur.tpos, lam, cur.cf,
                                           newc);
    TP_LAUNCH_CHECK();
    // rounds are enqueued in batches (four, then pairs) before the host
    // reads whether points are undecided: a round after the last is a no-op
    // (no point is undecided, so nothing is selected or changed); levels
    // here take about five rounds
    // rows per block of 256 threads: all 256 where that leaves eight blocks per
    // SM, fewer on small levels (at least one per lane group)
    const int rows_min = wrow ? 8 : 32;
    const int rows = std::max(rows_min, std::min(256, n / (8 * device_sms())));
    const int gr = grid_for(n, rows);
    int rounds = 0;
    while (true) {
      if (rounds >= opts.max_pmis_rounds) fail(TP_SETUP_FAILED, "PMIS round cap reached");
      const int batch = rounds == 0 ? 4 : 2;
      for (int r = 0; r < batch; ++r) {
        ++rounds;
        if (wrow) {
          k_pmis_select<32><<<gr, kBlock, 0, s>>>(n, A.rowptr, A.col, cur.strong, cur.tpos, lam,
                                                  cur.cf, opts.seed, rows, newc, undecided);
          TP_LAUNCH_CHECK();
          k_pmis_update<32><<<gr, kBlock, 0, s>>>(n, A.rowptr, A.col, cur.strong, cur.cf, rows,
                                                  newc, undecided);
        } else {
          k_pmis_select<8><<<gr, kBlock, 0, s>>>(n, A.rowptr, A.col, cur.strong, cur.tpos, lam,
                                                 cur.cf, opts.seed, rows, newc, undecided);
          TP_LAUNCH_CHECK();
          k_pmis_update<8><<<gr, kBlock, 0, s>>>(n, A.rowptr, A.col, cur.strong, cur.cf, rows,
                                                 newc, undecided);
        }
        TP_LAUNCH_CHECK();
      }
      if (read_int(undecided, s) == 0) break;
    }
    cur.pmis_rounds = rounds;
    mark_phase(0, s);
    int* cidx = scratch.alloc<int>(n + 1);
    // (one-pass interpolation: whether a row of a long-row level cannot take it
    // comes back with the number of C points)
    const bool ask = opts.pmax > 0 && interp_long_rows(A);
    int* past = undecided;  // 0 by now
    int rows_past = 0;
    if (ask) rows_past_one_pass(A, cur.strong, cur.cf, past, s);
    const int nc = (int)scan_states(cur.cf, kC, cidx, n, scratch, s, ask ? past : nullptr,
                                    &rows_past);
    if (nc == 0 || (double)nc > 0.9 * (double)n) {
      cur.cf = nullptr;  // this level becomes the coarsest
      break;
    }
    // interpolation: in one pass when it is truncated and the rows can take it,
    // else sets, weights and truncation by kernels of their own
    const bool extended = opts.interp != 0;
    DevCSR P;
    if (opts.pmax > 0 && rows_past == 0) {
      P = truncated_interpolation(A, extended, cur.dpos, cur.strong, cur.cf, cidx, nc, opts.pmax,
                                  pool, scratch, s);
    } else {
      P = untruncated_interpolation(A, extended, cur.dpos, cur.strong, cur.cf, cidx, nc, nullptr,
                                    n, pool, scratch, s);
      if (opts.pmax > 0) P = truncated(P, opts.pmax, pool, scratch, s);
    }
    cur.P = P;
    mark_phase(1, s);
    cur.R = transpose(P, pool, scratch, s);
    mark_phase(2, s);
    cur.AP = csr_product(A, P, pool, scratch, s);
    DevCSR Ac = csr_product(cur.R, cur.AP, pool, scratch, s);
    mark_phase(3, s);
    scratch.release();
    L.emplace_back();
    L.back().A = Ac;
  }
  mark_phase(0, s);
  finish_levels(s, true);
  mark_phase(4, s);
  TP_CUDA_TRY(cudaStreamSynchronize(s));
  read_phases();
}

// smoother scaling, FP32 copies, work vectors (allocate = first setup) and
// the coarsest-level inverse
void Hierarchy::finish_levels(cudaStream_t s, bool allocate) {
  const bool f32 = opts.precision >= 1;
  const bool bf16 = opts.precision == 2;
  TP_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int), s));
  if (opts.smoother == 1 && allocate)
    cheb_partials = pool.alloc<double>(2 * chebyshev_norm_parts());
  for (size_t l = 0; l < L.size(); ++l) {
    Level& v = L[l];
    const int n = v.A.n;
    if (allocate) {
      v.dinv = pool.alloc<double>(n);
      v.dinvf = f32 ? pool.alloc<float>(n) : nullptr;
    }
    if (opts.smoother == 1 && l + 1 < L.size()) {
      chebyshev_setup(v, pool, opts.cheb_degree, opts.seed, cheb_partials, err, allocate, s);
    } else {
      k_l1_dinv<<<grid_for(n), kBlock, 0, s>>>(n, v.A.rowptr, v.A.col, v.A.val, v.dinv,
                                               v.dinvf, err);
      TP_LAUNCH_CHECK();
    }
    if (l == 0 && opts.line_nz > 1 && L.size() > 1)
      line_setup(v, opts.line_nxy, opts.line_nz, pool, f32, err, allocate, s);
    if (f32) {
      if (allocate) v.A.valf = pool.alloc<float>(v.A.nnz);
      k_to_float<<<grid_for(v.A.nnz), kBlock, 0, s>>>(v.A.nnz, v.A.val, v.A.valf);
      TP_LAUNCH_CHECK();
      if (v.P.nnz) {
        if (allocate) {
          v.P.valf = pool.alloc<float>(v.P.nnz);
          v.R.valf = pool.alloc<float>(v.R.nnz);
        }
        k_to_float<<<grid_for(v.P.nnz), kBlock, 0, s>>>(v.P.nnz, v.P.val, v.P.valf);
        k_to_float<<<grid_for(v.R.nnz), kBlock, 0, s>>>(v.R.nnz, v.R.val, v.R.valf);
        TP_LAUNCH_CHECK();
        if (bf16) {
          if (allocate) {
            v.Ph = pool.alloc<__nv_bfloat16>(v.P.nnz);
            v.Rh = pool.alloc<__nv_bfloat16>(v.R.nnz);
          }
          k_to_bf16<<<grid_for(v.P.nnz), kBlock, 0, s>>>(v.P.nnz, v.P.val, v.Ph);
          k_to_bf16<<<grid_for(v.R.nnz), kBlock, 0, s>>>(v.R.nnz, v.R.val, v.Rh);
          TP_LAUNCH_CHECK();
        }
      }
    }
    // ELL copy for short-row levels (the 7-point finest level); by grid
    // direction when the level is a known grid's 7-point operator (the column
    // indices, a third of an FP64 sweep's matrix bytes and half an FP32
    // one's, are then implicit)
    const bool stencil = l == 0 && opts.grid_nx > 1 && opts.grid_ny > 1 && opts.grid_nz > 1 &&
                         (long long)opts.grid_nx * opts.grid_ny * opts.grid_nz == n;
    if (allocate && stencil) {
      v.ell_w = 7;
      v.ell_nx = opts.grid_nx;
      v.ell_nxy = opts.grid_nx * opts.grid_ny;
      v.ell_col = nullptr;
      v.ell_val = pool.alloc<double>((size_t)7 * n);
      v.ell_valf = f32 ? pool.alloc<float>((size_t)7 * n) : nullptr;
    } else if (allocate && n >= 4096 && v.A.nnz <= (long long)kEllMaxW * n) {
      // (a longer mean row rules the copy out without the read-back)
      TP_CUDA_TRY(cudaMemsetAsync(err + 1, 0, sizeof(int), s));
      k_max_row<<<grid_for(n), kBlock, 0, s>>>(n, v.A.rowptr, err + 1);
      TP_LAUNCH_CHECK();
      const int w = read_int(err + 1, s);
      if (w <= kEllMaxW) {
        v.ell_w = w;
        v.ell_col = pool.alloc<int>((size_t)w * n);
        v.ell_val = pool.alloc<double>((size_t)w * n);
        v.ell_valf = f32 ? pool.alloc<float>((size_t)w * n) : nullptr;
      }
    }
    if (v.ell_w > 0 && v.ell_nxy > 0) {
      k_to_stencil<<<grid_for(n), kBlock, 0, s>>>(n, v.ell_nx, v.ell_nxy, v.A.rowptr, v.A.col,
                                                  v.A.val, v.ell_val, v.ell_valf, err);
      TP_LAUNCH_CHECK();
    } else if (v.ell_w > 0) {
      k_to_ell<<<grid_for(n), kBlock, 0, s>>>(n, v.ell_w, v.A.rowptr, v.A.col, v.A.val,
                                              allocate ? v.ell_col : nullptr, v.ell_val,
                                              v.ell_valf);
      TP_LAUNCH_CHECK();
    }
    // sliced-ELL copy of the large levels below the finest: one thread per
    // row gives coalesced loads and no cross-lane reduction (the FP64 adds of
    // a split row's reduction compete with its multiply-adds for the FP64
    // pipe). It needs about half a wave of resident threads: on smaller
    // levels the lane-split CSR sweep fills the machine better. Measured FP64
    // / FP32 solve times (ms) without it; from 262,144 rows; from 131,072 or
    // 200,000 rows; on every level of 4096 rows or more: 256x256x64 layered
    // 169.9 / 116.6, 154.6 / 107.4, 151.3 / 107.4, 166.0 / 111.7; 128^2x64
    // channel 41.9 / 26.3, 40.7 / 25.1, 39.8 / 25.3, 49.7 / 28.5.
    const long long sell_min = opts.sell_rows == 0 ? resident_threads() / 2 : opts.sell_rows;
    if (allocate && opts.sell_rows >= 0 && l > 0 && v.ell_w == 0 && n >= sell_min &&
        l + 1 < L.size()) {
      const int windows = (n + kSellWindow - 1) / kSellWindow;
      const int slices = windows * (kSellWindow / 32);
      v.sell_perm = pool.alloc<int>((size_t)windows * kSellWindow);
      int* w32 = scratch.alloc<int>(slices + 1);
      k_sell_perm<<<windows, kSellWindow, 0, s>>>(n, v.A.rowptr, v.sell_perm, w32);
      TP_LAUNCH_CHECK();
      v.sell_ptr = pool.alloc<int>(slices + 1);
      const long long tot = scan_exclusive(w32, v.sell_ptr, slices, scratch, s);
      v.sell_col = pool.alloc<int>(tot + 1);
      v.sell_val = pool.alloc<double>(tot + 1);
      v.sell_valf = f32 ? pool.alloc<float>(tot + 1) : nullptr;
      v.sell_slices = slices;
      v.sell_entries = tot;
    }
    if (v.sell_slices > 0) {
      const int nslots = v.sell_slices * 32;
      k_sell_fill<<<grid_for(nslots), kBlock, 0, s>>>(nslots, v.A.rowptr, v.A.col, v.A.val,
                                                     v.sell_perm, v.sell_ptr,
                                                     allocate ? v.sell_col : nullptr, v.sell_val,
                                                     v.sell_valf);
      TP_LAUNCH_CHECK();
    }
    if (allocate) {
      const size_t es = f32 ? sizeof(float) : sizeof(double);
      v.b = pool.alloc<char>(es * (n + 1));
      v.x = pool.alloc<char>(es * (n + 1));
      v.t = pool.alloc<char>(es * (n + 1));
      v.r = pool.alloc<char>(es * (n + 1));
      if (opts.smoother == 1) {
        v.cw = pool.alloc<char>(es * (n + 1));
        v.cd0 = pool.alloc<char>(es * (n + 1));
        v.cd1 = pool.alloc<char>(es * (n + 1));
        v.cr = pool.alloc<char>(es * (n + 1));
      }
      v.lanes_A = pick_lanes(v.A);
      v.lanes_P = v.P.nnz ? pick_lanes(v.P) : 1;
      v.lanes_R = v.R.nnz ? pick_lanes(v.R) : 1;
    }
  }
  {
    const int e = read_int(err, s);
    if (e & 4) fail(TP_SETUP_FAILED, "AMG: empty, zero-diagonal or non-finite row");
    if (e & 8) fail(TP_SETUP_FAILED, "AMG: Chebyshev power iteration broke down");
    if (e & 16)
      fail(TP_SETUP_FAILED,
           "AMG: vertical-line smoother needs both vertical neighbours and non-zero pivots");
    if (e & 32) fail(TP_SETUP_FAILED, "AMG: level 0 is not the grid's 7-point pattern");
  }
  // coarsest level: explicit inverse by Gauss-Jordan with partial pivoting
  Level& cl = L.back();
  if (allocate) {
    nc = cl.A.n;
    if (nc > opts.max_coarse_dense) fail(TP_SETUP_FAILED, "AMG: coarsest level too large");
    coarse_dense = pool.alloc<double>((size_t)nc * nc);
    coarse_inv = pool.alloc<double>((size_t)nc * nc);
  }
  TP_CUDA_TRY(cudaMemsetAsync(coarse_dense, 0, sizeof(double) * (size_t)nc * nc, s));
  k_to_dense<<<grid_for((long long)nc * 32), kBlock, 0, s>>>(nc, cl.A.rowptr, cl.A.col, cl.A.val, coarse_dense);
  TP_LAUNCH_CHECK();
  TP_CUDA_TRY(cudaMemsetAsync(err, 0, sizeof(int), s));
  // one cluster holds the matrix in shared memory; the single-CTA kernel
  // (matrix in global memory) covers sizes beyond the cluster's capacity
  if (!coarse_inverse_cluster(nc, coarse_dense, coarse_inv, err, s)) {
    k_gauss_jordan<<<1, 1024, 0, s>>>(nc, coarse_dense, coarse_inv, err);
  }
  TP_LAUNCH_CHECK();
  if (read_int(err, s) != 0) fail(TP_SETUP_FAILED, "AMG: singular coarsest operator");
  if (allocate) {
    in = pool.alloc<double>(n0 + 1);
    out = pool.alloc<double>(n0 + 1);
    plan_tail(s);
  }
  TP_CUDA_TRY(cudaStreamSynchronize(s));
}

// Coarse tail: from the first level below level 0 with at most
// opts.tail_rows rows down to the coarsest, when at least one smoothing
// level is in it, the smoother is l1-Jacobi and clusters can be launched.
// The descriptors point at the level buffers, which keep their addresses
// under refresh().
void Hierarchy::plan_tail(cudaStream_t s) {
  tail_first = -1;
  const int nl = (int)L.size();
  if (opts.tail_rows <= 0 || opts.smoother != 0 || nl < 3) return;
  int f = -1;
  for (int l = 1; l < nl - 1; ++l)
    if (L[l].A.n <= opts.tail_rows) {
      f = l;
      break;
    }
  if (f < 0 || nl - f > kMaxTailLevels) return;
  const int cluster = tail_cluster_size();
  if (cluster == 0) return;
  const bool f32 = opts.precision >= 1;
  tail_host.assign(nl, TailLevel{});
  for (int l = 0; l < nl; ++l) {
    const Level& v = L[l];
    TailLevel& d = tail_host[l];
    d.n = v.A.n;
    d.nnext = (l + 1 < nl) ? L[l + 1].A.n : 0;
    d.Arp = v.A.rowptr;
    d.Acol = v.A.col;
    d.Aval = f32 ? (const void*)v.A.valf : (const void*)v.A.val;
    d.dinv = f32 ? (const void*)v.dinvf : (const void*)v.dinv;
    d.Prp = v.P.rowptr;
    d.Pcol = v.P.col;
    d.Pval = f32 ? (const void*)v.P.valf : (const void*)v.P.val;
    d.Ph = v.Ph;
    d.Rrp = v.R.rowptr;
    d.Rcol = v.R.col;
    d.Rval = f32 ? (const void*)v.R.valf : (const void*)v.R.val;
    d.Rh = v.Rh;
    d.b = v.b;
    d.x = v.x;
    d.t = v.t;
    d.r = v.r;
  }
  tail_desc = pool.alloc<TailLevel>(nl);
  TP_CUDA_TRY(cudaMemcpyAsync(tail_desc, tail_host.data(), sizeof(TailLevel) * nl,
                              cudaMemcpyHostToDevice, s));
  tail_first = f;
  tail_cluster = cluster;
}

void Hierarchy::refresh(cudaStream_t s) {
  if (L.empty()) fail(TP_ESTATE, "AMG: refresh before setup");
  for (size_t l = 0; l + 1 < L.size(); ++l) {
    Level& v = L[l];
    csr_product_numeric(v.A, v.P, v.AP, scratch, s);
    Level& c = L[l + 1];
    csr_product_numeric(v.R, v.AP, c.A, scratch, s);
    scratch.release();
  }
  finish_levels(s, false);
}

}  // namespace tp
