// Truncated interpolation in one pass per row: the interpolatory set, the
// classical or extended+i weights and the truncation to the pmax largest, with
// nothing but the truncated row written to memory.
//
// The arithmetic and its order are those of the untruncated kernels followed by
// k_trunc_fill (amg_setup.cu), which stay for untruncated interpolation, for the
// rows past the largest capacities here and for levels of long rows that have
// such a row, so the weights are the same bit for bit.
//
// What bounds it: the rows of the strong F neighbours have to be read (128
// entries per F row on the first Galerkin level of the layered A_pp, 340 on the
// second), while the sets hold about 5 points and about 19 of the entries
// read enter a sum. So the integer work is spread over lanes and the FP64 work
// kept off them: G lanes of a row walk the concatenated rows of its strong F
// neighbours (coalesced, no lane idle at a row's end), look every column up in
// a hash table in shared memory and append the few entries that count, in
// order, to a list; the sums, which are serial in that order, then run for R
// rows of a warp at once (one lane per neighbour, one per row for the
// denominator), because an FP64 instruction occupies this part's FP64 pipe for
// the whole warp however few lanes take part.
//
// Measured on GB300, layered 256x256x64 (kernel time summed over a setup, both
// hierarchies on their streams): sets, weights and truncation of A_pp 29.4 ms
// before, 15.8 ms here; of S~ 13.2 before, 5.6 here; whole step 201.8 ->
// 192.5 ms, 64x64x32 20.8 -> 19.8 ms, 16x16x8 4.37 -> 4.14 ms (fewer launches
// and one host round trip less per level). What bounds it now is latency at
// low occupancy (shared memory and registers leave 19-28 of 64 warps per SM;
// the 8-lane form also keeps the FP64 pipe half busy, mostly divisions).
#include "amg_dev.cuh"
#include "per_device.cuh"

namespace tp {

namespace {

struct InterpWork {
  int* cnt;      // [n + 1] entries of every truncated row
  int* tcol;     // [n * pmax] truncated rows at i * pmax
  double* tval;
  int *olist0, *olist1;  // rows past a tier's capacities
  int* ocnt;             // [3] their counts by tier
};

// Row classes by the level's mean row length (7 on the finest, 10-15 on S~'s
// first Galerkin levels, 29 on A_pp's first): up to kInterpShortMean 8 lanes
// per row, eight rows per warp (FP64 bound: four rows per warp 5.7 ms instead
// of 4.9 on the layered finest level); above it 16 lanes, two rows per warp
// (latency bound: four rows per warp, half the warps in flight, 10.0 ms
// instead of 8.3 on A_pp's Galerkin levels; a warp per row 9.4). Rows past a
// class's capacities go to the next class through a list. Levels of at most
// kInterpFewRows rows that are not short start at the last class, a warp per
// row: the others would leave most SMs without a warp.
// The last class takes rows of up to 128 strong F neighbours, 32 at a time.
constexpr double kInterpShortMean = 20.0;
constexpr int kInterpFewRows = 16384;
// Levels of long rows on the mean are asked first whether a row is past the last
// class (interp_long_rows, rows_past_one_pass), and go to the untruncated kernels
// as a whole if one is: these wait for their longest rows, so the pass over the
// others would come on top (random graph, levels of 4723 rows of 1164 entries and
// of 963 of 907: 1.8 and 5.2 ms untruncated, the pass 0.6 and 1.5 ms more; setup
// 28.9 -> 26.3 ms). Shorter levels, a grid's among them, are not asked: the pass is
// a small part of what the untruncated kernels take there, and the few rows past
// it go to them by a list (150000 rows of 23 entries, two of them with 800 strong F
// neighbours: 1.08 ms untruncated, 0.94 by pass and list; setup 34.5 -> 29.4 ms).
constexpr int kInterpLongMean = 100;
// the last class: strong F neighbours, entries, set members of a row, entries of
// its neighbours' rows that count
constexpr int kInterpKM = 128, kInterpRL = 1024, kInterpSet = 128, kInterpEnt = 1024;

constexpr unsigned kAll = 0xffffffffu;
constexpr unsigned char kSelf = 255;  // list entry a_ki (extended+i), no slot

// shared memory of one warp: R rows
template <int R, int SET, int ENT, int KM, int RL>
struct InterpRows {
  static constexpr int HS = 2 * SET;  // hash slots
  double ev[R][ENT];            // entries a_km that count; then t_k a_km
  double tk[R][KM];             // t_k = a_ik / s_k
  double num[R][SET];           // numerators, then weights
  int setc[R][SET];             // the set, fine columns ascending
  int hkey[R][HS];
  int ns[R], nk[R], nent[R], row[R];  // row: -1 nothing to do
  unsigned short kst[R][KM + 2];      // list positions of neighbour k
  unsigned short ke[R][KM];           // entry of row i of neighbour k
  unsigned short kself[R][KM];        // list position of a_ki, 0xffff none
  unsigned char hslot[R][HS];
  unsigned char eslot[R][ENT];
  unsigned char ek[R][ENT];
  unsigned char flag[R][RL];    // 0 skip, 1 lumped, 2 neighbour lumped, 3 neighbour
};

template <int HS>
__device__ __forceinline__ unsigned hash_of(int key) {
  static_assert((HS & (HS - 1)) == 0, "power of two");
  return (((unsigned)key * 0x9E3779B1u) >> 16) & (unsigned)(HS - 1);
}

// position of key in the table, or -1
template <int HS>
__device__ __forceinline__ int hash_find(const int* hkey, int key) {
  unsigned h = hash_of<HS>(key);
  for (int p = 0; p < HS; ++p) {
    const int k = hkey[h];
    if (k == key) return (int)h;
    if (k < 0) return -1;
    h = (h + 1) & (unsigned)(HS - 1);
  }
  return -1;
}

// key into the table (and, when new, onto the unordered set while it has room)
template <int HS, int SET>
__device__ __forceinline__ void hash_add(int* hkey, int* setc, int* ns, int key) {
  unsigned h = hash_of<HS>(key);
  for (int p = 0; p < HS; ++p) {
    const int prev = atomicCAS(&hkey[h], -1, key);
    if (prev == key) return;
    if (prev == -1) {
      const int q = atomicAdd(ns, 1);
      if (q < SET) setc[q] = key;
      return;
    }
    h = (h + 1) & (unsigned)(HS - 1);
  }
  atomicAdd(ns, SET + 1);  // table full: overflow
}

// EXT: extended+i, else classical. Rows list[0, *nlist) (list null: rows 0 to
// n - 1). A row past a capacity goes to olist (its count in *ocnt).
template <bool EXT, int G, int R, int SET, int ENT, int KM, int RL, int WARPS>
__global__ void __launch_bounds__(32 * WARPS) k_interp(
    int n, const int* __restrict__ list, const int* __restrict__ nlist,
    const int* __restrict__ rp, const int* __restrict__ col, const double* __restrict__ val,
    const int* __restrict__ dpos, const unsigned char* __restrict__ strong,
    const signed char* __restrict__ state, const int* __restrict__ cidx, int pmax,
    int* __restrict__ cnt, int* __restrict__ tcol, double* __restrict__ tval,
    int* __restrict__ olist, int* __restrict__ ocnt) {
  using S = InterpRows<R, SET, ENT, KM, RL>;
  constexpr int HS = S::HS, NG = 32 / G, LR = 32 / R;
  static_assert(KM < 256 && R % NG == 0 && SET < kSelf && ENT < 0xffff, "capacities");
  extern __shared__ __align__(16) char smem[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  S& s = reinterpret_cast<S*>(smem)[w];
  const int grp = lane / G, gl = lane % G;
  const unsigned gmask = (G == 32 ? 0xffffffffu : ((1u << G) - 1u)) << (grp * G);
  const unsigned below = (1u << lane) - 1u;
  const int count = list ? *nlist : n;
  const long long nwarps = (long long)gridDim.x * WARPS;
  for (long long base = ((long long)blockIdx.x * WARPS + w) * R; base < count;
       base += nwarps * R) {
    // ---- the set and the lists, G lanes per row, NG rows at a time. The
    // groups of a warp stay together (trip counts are the warp's largest, a
    // group past its own end idles): left to run apart, their instructions
    // issue group by group (8-lane form on a 1 M-row 7-point level: 686 warp
    // instructions per row at 9.9 threads each, 1.63 ms)
#pragma unroll 1
    for (int r = grp; r < R; r += NG) {
      const long long q = base + r;
      const int i = q < count ? (list ? list[q] : (int)q) : -1;
      bool act = i >= 0;
      int r0 = 0, len = 0;
      if (act) {
        if (state[i] == kC) {
          if (gl == 0) {
            tcol[(long long)i * pmax] = cidx[i];
            tval[(long long)i * pmax] = 1.0;
            cnt[i] = 1;
          }
          act = false;
        } else {
          r0 = rp[i];
          len = rp[i + 1] - r0;
        }
      }
      bool over = act && len > RL;
      if (over || !act) len = 0;
      if (gl == 0) {
        s.ns[r] = 0;
        s.row[r] = -1;
      }
      const int lenmax = __reduce_max_sync(kAll, len);
      if (lenmax > 0) {
        for (int h = gl; h < HS; h += G) s.hkey[r][h] = -1;
        __syncwarp();
        // row i: strong C points into the set, strong F points listed
        int nk = 0;
        for (int e0 = 0; e0 < lenmax; e0 += G) {
          const int e = e0 + gl;
          int k = -1;
          bool st = false, isc = false;
          if (e < len) {
            k = col[r0 + e];
            st = strong[r0 + e] != 0 && k != i;
            isc = st && state[k] == kC;
            s.flag[r][e] = k == i ? 0 : (st ? (isc ? 0 : 3) : 1);
          }
          if (isc) hash_add<HS, SET>(s.hkey[r], s.setc[r], &s.ns[r], k);
          const bool isf = st && !isc;
          const unsigned fm = __ballot_sync(kAll, isf) & gmask;
          if (isf) {
            const int p = nk + __popc(fm & below);
            if (p < KM) s.ke[r][p] = (unsigned short)e;
          }
          nk += __popc(fm);
        }
        if (nk > KM) {
          over = true;
          nk = 0;
        }
        __syncwarp();
        // G neighbours at a time, one on each lane: its row, its diagonal's sign
        const int nk_max = __reduce_max_sync(kAll, nk);
        int kk = -1, kb = 0, klen = 0, excl = 0, rel = 0, total = 0, total_max = 0;
        unsigned kc = 0;
        auto load = [&](int k0) {
          kk = -1;
          kb = klen = 0;
          kc = 0;
          if (k0 + gl < nk) {
            kk = col[r0 + s.ke[r][k0 + gl]];
            kb = rp[kk];
            klen = rp[kk + 1] - kb;
            kc = sign_class(val[dpos[kk]]);
          }
          int incl = klen;
#pragma unroll
          for (int o = 1; o < G; o <<= 1) {
            const int y = __shfl_up_sync(kAll, incl, o, G);
            if (gl >= o) incl += y;
          }
          excl = incl - klen;
          rel = kb - excl;
          total = __shfl_sync(kAll, incl, G - 1, G);
          total_max = __reduce_max_sync(kAll, total);
        };
        load(0);
        // position p of the concatenated rows: owning neighbour and entry
        auto locate = [&](int p, int& own) -> int {
          int lo = 0;
#pragma unroll
          for (int step = G / 2; step > 0; step >>= 1)
            if (__shfl_sync(kAll, excl, lo + step, G) <= p) lo += step;
          own = lo;
          return __shfl_sync(kAll, rel, lo, G) + p;
        };
        if (EXT) {
          for (int k0 = 0; k0 < nk_max; k0 += G) {
            if (k0 > 0) load(k0);
            for (int p0 = 0; p0 < total_max; p0 += G) {
              const int p = p0 + gl;
              int own;
              const int f = locate(p, own);
              const int kown = __shfl_sync(kAll, kk, own, G);
              if (p < total && strong[f]) {
                const int m = col[f];
                if (m != kown && state[m] == kC)
                  hash_add<HS, SET>(s.hkey[r], s.setc[r], &s.ns[r], m);
              }
            }
          }
        }
        __syncwarp();
        int ns = s.ns[r];
        if (ns > SET) over = true;
        if (over || !act) ns = 0;
        const int ns_max = __reduce_max_sync(kAll, ns);
        // the set in ascending order, every key's slot beside it
        constexpr int Q = (SET + G - 1) / G;
        int key[Q], rank[Q];
#pragma unroll
        for (int u = 0; u < Q; ++u) {
          const int a = gl + u * G;
          key[u] = a < ns ? s.setc[r][a] : 0x7fffffff;
          rank[u] = 0;
        }
        for (int j = 0; j < ns_max; ++j) {
          const int c = j < ns ? s.setc[r][j] : 0x7fffffff;
#pragma unroll
          for (int u = 0; u < Q; ++u) rank[u] += c < key[u];
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < Q; ++u)
          if (gl + u * G < ns) {
            s.setc[r][rank[u]] = key[u];
            s.num[r][gl + u * G] = 0.0;
            s.hslot[r][hash_find<HS>(s.hkey[r], key[u])] = (unsigned char)rank[u];
          }
        for (int k = gl; k < nk; k += G) s.kself[r][k] = 0xffff;
        __syncwarp();
        // numerators start at a_im; a weak neighbour in the set is not lumped
        for (int e = gl; e < len; e += G) {
          const int h = over ? -1 : hash_find<HS>(s.hkey[r], col[r0 + e]);
          if (h >= 0) {
            s.num[r][s.hslot[r][h]] = val[r0 + e];
            s.flag[r][e] = 0;
          }
        }
        // the entries of the neighbours' rows that count, in order
        int ne = 0;
        for (int k0 = 0; k0 < nk_max; k0 += G) {
          if (nk_max > G) load(k0);
          const int ne0 = ne;
          int mine = 0;
          for (int p0 = 0; p0 < total_max; p0 += G) {
            const int p = p0 + gl;
            int own;
            const int f = locate(p, own);
            const unsigned char okc = (unsigned char)__shfl_sync(kAll, kc, own, G);
            bool sel = false;
            double v = 0.0;
            unsigned char slot = kSelf;
            if (p < total && !over) {
              v = val[f];
              if (opposite_class(v, okc)) {
                const int m = col[f];
                if (EXT && m == i) {
                  sel = true;
                } else {
                  const int h = hash_find<HS>(s.hkey[r], m);
                  if (h >= 0) {
                    sel = true;
                    slot = s.hslot[r][h];
                  }
                }
              }
            }
            const unsigned bal = __ballot_sync(kAll, sel) & gmask;
            if (sel) {
              const int at = ne + __popc(bal & below);
              if (at < ENT) {
                s.ev[r][at] = v;
                s.eslot[r][at] = slot;
                s.ek[r][at] = (unsigned char)(k0 + own);
                if (slot == kSelf) s.kself[r][k0 + own] = (unsigned short)at;
              }
            }
            ne += __popc(bal);
            // entries of this lane's neighbour among the group's positions
            const int lo = max(excl - p0, 0), hi = min(excl + klen - p0, G);
            if (hi > lo) {
              const unsigned bits = (bal >> (grp * G)) >> lo;
              mine += __popc(hi - lo == 32 ? bits : bits & ((1u << (hi - lo)) - 1u));
            }
          }
          int kincl = mine;
#pragma unroll
          for (int o = 1; o < G; o <<= 1) {
            const int y = __shfl_up_sync(kAll, kincl, o, G);
            if (gl >= o) kincl += y;
          }
          if (k0 + gl < nk) s.kst[r][k0 + gl] = (unsigned short)min(ne0 + kincl - mine, ENT);
        }
        if (ne > ENT) over = true;
        if (act && !over) {
          if (gl == 0) {
            s.kst[r][nk] = (unsigned short)ne;
            s.nk[r] = nk;
            s.nent[r] = ne;
            s.row[r] = i;
            cnt[i] = min(ns, pmax);
          }
        }
      }
      if (over && gl == 0) {
        olist[atomicAdd(ocnt, 1)] = i;
        cnt[i] = 0;
      }
      __syncwarp();
    }
    // ---- the sums, all R rows at once: (row, neighbour), (row, entry) and
    // (row, slot) pairs flat over the lanes, so that a division, ten or so
    // FP64 instructions, is issued once per 32 of them
    const int r = lane / LR, sub = lane % LR;
    const int i = s.row[r];
    const int ns = i >= 0 ? s.ns[r] : 0, nk = i >= 0 ? s.nk[r] : 0;
    const int nent = i >= 0 ? s.nent[r] : 0;
    const int r0 = i >= 0 ? rp[i] : 0;
    // fn(row, index) for index < count of the row
    auto flat = [&](int count_of_r, auto fn) {
      int incl = sub == 0 ? count_of_r : 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kAll, incl, o);
        if (lane >= o) incl += y;
      }
      const int excl = incl - count_of_r;  // of this lane's row
      const int total = __shfl_sync(kAll, incl, 31);
      for (int t0 = 0; t0 < total; t0 += 32) {
        const int t = t0 + lane;
        int lo = 0;
#pragma unroll
        for (int step = R / 2; step > 0; step >>= 1)
          if (__shfl_sync(kAll, excl, (lo + step) * LR) <= t) lo += step;
        const int first = __shfl_sync(kAll, excl, lo * LR);
        const int start = __shfl_sync(kAll, r0, lo * LR);
        if (t < total) fn(lo, t - first, start);
      }
      __syncwarp();
    };
    // s_k in list order; t_k = a_ik / s_k, or a_ik lumped when s_k is zero
    flat(nk, [&](int row, int k, int start) {
      double sk = 0.0;
      for (int q = s.kst[row][k]; q < s.kst[row][k + 1]; ++q) sk = __dadd_rn(sk, s.ev[row][q]);
      const int e = s.ke[row][k];
      if (nonzero_bits(sk)) s.tk[row][k] = __ddiv_rn(val[start + e], sk);
      else s.flag[row][e] = 2;
    });
    flat(nent, [&](int row, int q, int) {
      const int k = s.ek[row][q];
      if (s.flag[row][s.ke[row][k]] == 3) s.ev[row][q] = __dmul_rn(s.tk[row][k], s.ev[row][q]);
    });
    // numerators: neighbours in order, the entries of one hit distinct slots
    const int kmax = __reduce_max_sync(kAll, nk);
    for (int k = 0; k < kmax; ++k) {
      if (k < nk && s.flag[r][s.ke[r][k]] == 3)
        for (int q = s.kst[r][k] + sub; q < s.kst[r][k + 1]; q += LR) {
          const unsigned char slot = s.eslot[r][q];
          if (slot != kSelf) s.num[r][slot] = __dadd_rn(s.num[r][slot], s.ev[r][q]);
        }
      __syncwarp();
    }
    // denominator over row i in order, one lane per row
    double denom = 0.0;
    if (sub == 0 && ns > 0) {
      denom = val[dpos[i]];
      const int len = rp[i + 1] - r0;
      int k = 0;
      constexpr int U = 8;
      for (int e0 = 0; e0 < len; e0 += U) {
        double v[U];
        unsigned char fl[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          fl[u] = e0 + u < len ? s.flag[r][e0 + u] : 0;
          v[u] = (fl[u] == 1 || fl[u] == 2) ? val[r0 + e0 + u] : 0.0;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          bool add = fl[u] == 1 || fl[u] == 2;
          if (fl[u] >= 2) {
            if (EXT && fl[u] == 3) {
              const unsigned short at = s.kself[r][k];
              if (at != 0xffff) {
                v[u] = s.ev[r][at];
                add = nonzero_bits(v[u]);
              }
            }
            ++k;
          }
          if (add) denom = __dadd_rn(denom, v[u]);
        }
      }
    }
    if (sub == 0) s.tk[r][0] = denom;  // the t_k are done with
    __syncwarp();
    flat(ns, [&](int row, int a, int) { s.num[row][a] = __ddiv_rn(-s.num[row][a], s.tk[row][0]); });
    // truncation: the pmax largest |w| (ties to the lower column) scaled by
    // (sum of all) / (sum of kept), sums over the row ascending from 0.0
    const bool cut = ns > pmax;
    double f = 1.0, s_keep = 0.0;
    // kept slots of this row as a bit set over the lanes' slots
    for (int a = sub; a < ns; a += LR) {
      int rank = 0;
      if (cut) {
        const unsigned long long m = mag_key(s.num[r][a]);
        for (int j = 0; j < ns; ++j) {
          const unsigned long long mj = mag_key(s.num[r][j]);
          rank += mj > m || (mj == m && j < a);
        }
      }
      s.eslot[r][a] = rank < pmax ? 1 : 0;  // the lists are done with
    }
    __syncwarp();
    if (cut && sub == 0) {
      double s_all = 0.0;
      for (int a = 0; a < ns; ++a) {
        s_all = __dadd_rn(s_all, s.num[r][a]);
        if (s.eslot[r][a]) s_keep = __dadd_rn(s_keep, s.num[r][a]);
      }
      f = nonzero_bits(s_keep) ? __ddiv_rn(s_all, s_keep) : 1.0;
    }
    f = __shfl_sync(kAll, f, r * LR);
    s_keep = __shfl_sync(kAll, s_keep, r * LR);
    for (int a = sub; a < ns; a += LR) {
      if (!s.eslot[r][a]) continue;
      int at = 0;
      for (int j = 0; j < a; ++j) at += s.eslot[r][j];
      const double v = s.num[r][a];
      tcol[(long long)i * pmax + at] = cidx[s.setc[r][a]];
      tval[(long long)i * pmax + at] = cut && nonzero_bits(s_keep) ? __dmul_rn(v, f) : v;
    }
    __syncwarp();
  }
}

// sets *past when an F row has more entries, strong F neighbours or strong C
// neighbours (its classical set, a part of its extended+i one) than the last class
// holds, or, if the level's entries (a share `fill` of n^2) lie evenly, more
// entries of the neighbours' rows in the set (a warp per row)
__global__ void k_rows_past(int n, float fill, const int* __restrict__ rp,
                            const int* __restrict__ col,
                            const unsigned char* __restrict__ strong,
                            const signed char* __restrict__ state, int* __restrict__ past) {
  const int i = (int)((blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= n || state[i] == kC) return;
  const int r0 = rp[i], r1 = rp[i + 1];
  int nk = 0, ns = 0;
  if (r1 - r0 <= kInterpRL)
    for (int e = r0 + lane; e < r1; e += 32)
      if (strong[e]) (state[col[e]] == kC ? ns : nk) += 1;
  nk = __reduce_add_sync(kAll, nk);
  ns = __reduce_add_sync(kAll, ns);
  if (lane == 0 && (r1 - r0 > kInterpRL || nk > kInterpKM || ns > kInterpSet ||
                    fill * (float)nk * (float)ns > (float)kInterpEnt))
    *past = 1;
}

// rows of at most pmax entries at i * pmax to the compact CSR
__global__ void k_interp_compact(int n, int pmax, const int* __restrict__ tcol,
                                 const double* __restrict__ tval, const int* __restrict__ Prp,
                                 int* __restrict__ Pcol, double* __restrict__ Pval) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int i = (int)(t / pmax), q = (int)(t % pmax);
  if (i >= n) return;
  const int p0 = Prp[i];
  if (p0 + q < Prp[i + 1]) {
    Pcol[p0 + q] = tcol[t];
    Pval[p0 + q] = tval[t];
  }
}

template <bool EXT, int G, int R, int SET, int ENT, int KM, int RL, int WARPS>
void launch_tier(int blocks_per_sm, int sms, int n, const int* list, const int* nlist,
                 const DevCSR& A, const int* dpos, const unsigned char* strong,
                 const signed char* state, const int* cidx, int pmax, int* cnt, int* tcol,
                 double* tval, int* olist, int* ocnt, cudaStream_t s) {
  auto kern = k_interp<EXT, G, R, SET, ENT, KM, RL, WARPS>;
  constexpr size_t smem = WARPS * sizeof(InterpRows<R, SET, ENT, KM, RL>);
  static PerDevice<bool> allowed;
  allow_smem(allowed, kern, smem);
  long long blocks = ((long long)n + R * WARPS - 1) / (R * WARPS);
  if (list && blocks > (long long)blocks_per_sm * sms) blocks = (long long)blocks_per_sm * sms;
  kern<<<(int)blocks, 32 * WARPS, smem, s>>>(n, list, nlist, A.rowptr, A.col, A.val, dpos,
                                             strong, state, cidx, pmax, cnt, tcol, tval, olist,
                                             ocnt);
  TP_LAUNCH_CHECK();
}

template <bool EXT>
void interp_tiers(const DevCSR& A, int sms, const int* dpos, const unsigned char* strong,
                  const signed char* state, const int* cidx, int pmax, InterpWork& w,
                  cudaStream_t s) {
  const int n = A.n;
  TP_CUDA_TRY(cudaMemsetAsync(w.ocnt, 0, 3 * sizeof(int), s));
  const double mean = n > 0 ? (double)A.nnz / n : 0.0;
  const int* list = nullptr;
  const int* nlist = nullptr;
  if (mean <= kInterpShortMean) {
    launch_tier<EXT, 8, 8, 16, 32, 8, 32, 4>(8, sms, n, list, nlist, A, dpos, strong, state, cidx,
                                             pmax, w.cnt, w.tcol, w.tval, w.olist0, w.ocnt, s);
    list = w.olist0;
    nlist = w.ocnt;
  }
  if (n > kInterpFewRows || list) {
    launch_tier<EXT, 16, 2, 32, 128, 16, 128, 4>(8, sms, n, list, nlist, A, dpos, strong, state,
                                                 cidx, pmax, w.cnt, w.tcol, w.tval, w.olist1,
                                                 w.ocnt + 1, s);
    list = w.olist1;
    nlist = w.ocnt + 1;
  }
  launch_tier<EXT, 32, 1, kInterpSet, kInterpEnt, kInterpKM, kInterpRL, 2>(
      6, sms, n, list, nlist, A, dpos, strong, state, cidx, pmax, w.cnt, w.tcol, w.tval, w.olist0,
      w.ocnt + 2, s);
}

}  // namespace

bool interp_long_rows(const DevCSR& A) { return A.nnz > (long long)kInterpLongMean * A.n; }

void rows_past_one_pass(const DevCSR& A, const unsigned char* strong, const signed char* state,
                        int* past, cudaStream_t s) {
  const float fill = (float)((double)A.nnz / ((double)A.n * A.n));
  k_rows_past<<<grid_for((long long)A.n * 32), kBlock, 0, s>>>(A.n, fill, A.rowptr, A.col, strong,
                                                              state, past);
  TP_LAUNCH_CHECK();
}

DevCSR truncated_interpolation(const DevCSR& A, bool extended, const int* dpos,
                               const unsigned char* strong, const signed char* state,
                               const int* cidx, int nc, int pmax, Pool& pool, Pool& scratch,
                               cudaStream_t s) {
  const int n = A.n;
  InterpWork w;
  w.cnt = scratch.alloc<int>(n + 1);
  w.tcol = scratch.alloc<int>((size_t)n * pmax);
  w.tval = scratch.alloc<double>((size_t)n * pmax);
  w.olist0 = scratch.alloc<int>(n);
  w.olist1 = scratch.alloc<int>(n);
  w.ocnt = scratch.alloc<int>(3);
  if (extended) interp_tiers<true>(A, device_sms(), dpos, strong, state, cidx, pmax, w, s);
  else interp_tiers<false>(A, device_sms(), dpos, strong, state, cidx, pmax, w, s);
  int over = 0;  // rows past the last capacities
  DevCSR P;
  P.n = n;
  P.m = nc;
  P.rowptr = pool.alloc<int>(n + 1);
  long long total = scan_exclusive(w.cnt, P.rowptr, n, scratch, s, w.ocnt + 2, &over);
  if (over > 0) {
    const DevCSR U = untruncated_interpolation(A, extended, dpos, strong, state, cidx, nc,
                                               w.olist0, over, scratch, scratch, s);
    truncate_listed_rows(U, w.olist0, pmax, w.cnt, w.tcol, w.tval, s);
    total = scan_exclusive(w.cnt, P.rowptr, n, scratch, s);
  }
  P.nnz = (int)total;
  P.col = pool.alloc<int>(P.nnz + 1);
  P.val = pool.alloc<double>(P.nnz + 1);
  k_interp_compact<<<grid_for((long long)n * pmax), kBlock, 0, s>>>(n, pmax, w.tcol, w.tval,
                                                                    P.rowptr, P.col, P.val);
  TP_LAUNCH_CHECK();
  return P;
}

}  // namespace tp
