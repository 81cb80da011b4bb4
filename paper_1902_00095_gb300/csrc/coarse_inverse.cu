// Explicit inverse of the coarsest AMG operator (dense n x n, row-major),
// the coarse-grid solver of the V-cycle (Gaussian elimination on the
// coarsest grid, Sec. 4 solver settings), computed inside one
// thread-block cluster.
//
// The rows are split over the cluster's CTAs and stay in their shared
// memory for the whole elimination. Gauss-Jordan runs in place, without an
// augmented identity: at step k with pivot row p (column k),
//   rows i != p:  f_i = a_ik / a_pk,  a_ij -= f_i a_pj (j != k),  a_ik = -f_i
//   row p:        a_pj /= a_pk (j != k),  a_pk = 1 / a_pk
// (each division taken as a product with the reciprocal 1 / a_pk).
// Column k of the identity is e_k until step k, so it can live in the slot
// of column k of A, which step k clears. The pivot is the largest |a_ik|
// over the rows not yet used (ties to the lower row index): each CTA offers
// its best row (a copy of the row, and its value, index and 1 / value stored
// into every CTA's shared memory), every CTA takes the same pivot from the
// offers it holds, copies the pivot row from its
// owner's offer, then updates its own rows. Choosing row p_k at step k is unpivoted elimination of
// B = Pi A (row k of B = row p_k of A) stored in A's row order, so the storage
// ends with B^{-1} = A^{-1} Pi^T, row k of it in storage row p_k, i.e.
// A^{-1}[k][p_j] = M[p_k][j]; the epilogue writes it out in that order.
//
// One cluster barrier per step (a CTA rewrites an offer buffer only after
// the next barrier, which every reader of it has passed); no flag waits.
//
// A step is a chain of latencies beside n^2 / (16 C) FP64 cycles of updates, so
// the chain is kept short: the offers lie in local memory when the barrier
// opens, every warp takes the pivot by itself (integer reductions, no block
// barrier), and while the other warps update their rows warp 0 already forms
// column k + 1 (the same products, so the same bits), picks the next offer
// and its reciprocal. n = 64: 143 -> 109 us, 112: 314 -> 218, 149: 438 -> 340,
// 248: 1103 -> 770, 400: 2557 -> 2135, 640: 7256 -> 6531 (at n = 149 a step is
// some 4300 clocks: 900 the barrier, 1000 the pivot row through its owner's
// shared memory, 1400 the offer, beside which the update is nearly hidden).
// Rows cut into strips of 32 to 256 columns over 15 warps were slower (149: 383
// to 545 us).
// The caller checks and counts the launch.
#include <cooperative_groups.h>
#include <climits>

#include "amg.cuh"
#include "per_device.cuh"

namespace cg = cooperative_groups;

namespace tp {

namespace {

constexpr int kGjThreads = 512;
constexpr int kGjWarps = kGjThreads / 32;

constexpr int kGjMaxCluster = 16;
constexpr int kGjLaneRows = 2;  // rows of a CTA per lane of warp 0: R <= 64, since
                                // R^2 * 8 * (cluster size) bytes fit an SM

// shared-memory layout of one CTA (R rows of n entries), same on both sides
struct GjLayout {
  size_t M, offer, prow, fr, cand_k, cand_inv, perm, pos, cand_i, mine, bytes;
  __host__ __device__ GjLayout(int n, int R) {
    size_t o = 0;
    M = o;        o += sizeof(double) * (size_t)R * n;
    offer = o;    o += sizeof(double) * 2 * (size_t)n;
    prow = o;     o += sizeof(double) * (size_t)n;
    fr = o;       o += sizeof(double) * (size_t)R;
    cand_k = o;   o += sizeof(unsigned long long) * 2 * kGjMaxCluster;
    cand_inv = o; o += sizeof(double) * 2 * kGjMaxCluster;
    perm = o;     o += sizeof(int) * (size_t)n;
    cand_i = o;   o += sizeof(int) * 2 * kGjMaxCluster;
    mine = o;     o += sizeof(int) * 2;
    pos = cand_k;  // after the last step (R ints)
    bytes = o;
  }
};

// Ordering key of |a|: for non-negative IEEE doubles the bit patterns,
// read as unsigned integers, order like the values; NaN maps to 0 (never a
// pivot, as a zero).
__device__ __forceinline__ unsigned long long abs_key(double a) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(a) & 0x7fffffffffffffffull;
  return u > 0x7ff0000000000000ull ? 0ull : u;
}

// Largest key over the warp's lanes, equal keys to the lower index: returns that
// index on every lane and leaves the key in `key` (integer reductions; the FP64
// pipe is narrow on this part).
__device__ __forceinline__ int warp_best(unsigned long long& key, int idx) {
  const unsigned hi = (unsigned)(key >> 32), lo = (unsigned)key;
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
  key = (unsigned long long)mh << 32 | ml;
  return __reduce_min_sync(0xffffffffu, hi == mh && lo == ml ? idx : INT_MAX);
}

__global__ void __launch_bounds__(kGjThreads) k_gj_cluster(int n, int R,
                                                           const double* __restrict__ A,
                                                           double* __restrict__ inv,
                                                           int* __restrict__ err) {
  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)cluster.num_blocks();
  const int c = (int)cluster.block_rank();
  extern __shared__ __align__(16) unsigned char smem[];
  const GjLayout lay(n, R);
  double* M = reinterpret_cast<double*>(smem + lay.M);
  double* prow = reinterpret_cast<double*>(smem + lay.prow);
  double* fr = reinterpret_cast<double*>(smem + lay.fr);
  unsigned long long* cand_k = reinterpret_cast<unsigned long long*>(smem + lay.cand_k);
  double* cand_inv = reinterpret_cast<double*>(smem + lay.cand_inv);
  double* offer = reinterpret_cast<double*>(smem + lay.offer);
  int* perm = reinterpret_cast<int*>(smem + lay.perm);
  int* pos = reinterpret_cast<int*>(smem + lay.pos);
  int* cand_i = reinterpret_cast<int*>(smem + lay.cand_i);
  int* mine = reinterpret_cast<int*>(smem + lay.mine);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = c * R;
  const int rc = max(0, min(R, n - r0));  // rows this CTA owns
  for (int r = warp; r < rc; r += kGjWarps)
    for (int j = lane; j < n; j += 32) M[(size_t)r * n + j] = A[(size_t)(r0 + r) * n + j];
  bool used[kGjLaneRows] = {};  // warp 0: rows lane + 32 q taken as pivots
  // all CTAs of the cluster run before one stores into another
  cluster.sync();

  // warp 0: the offer for a step from v, that step's column in rows lane + 32 q
  auto make_offer = [&](int b, const double (&v)[kGjLaneRows]) {
    unsigned long long key = 0ull;
    int bi = INT_MAX;
    double vb = 0.0;
#pragma unroll
    for (int q = 0; q < kGjLaneRows; ++q) {
      const int r = lane + 32 * q;
      const unsigned long long ok = abs_key(v[q]);
      if (r < rc && !used[q] && (ok > key || bi == INT_MAX)) {
        key = ok;
        bi = r0 + r;
        vb = v[q];
      }
    }
    bi = warp_best(key, bi);
    const double inv_v = 1.0 / __shfl_sync(0xffffffffu, vb, bi == INT_MAX ? 0 : (bi - r0) & 31);
    if (lane < C) {
      const int at = b * kGjMaxCluster + c;
      cluster.map_shared_rank(cand_k, (unsigned)lane)[at] = key;
      cluster.map_shared_rank(cand_inv, (unsigned)lane)[at] = inv_v;
      cluster.map_shared_rank(cand_i, (unsigned)lane)[at] = bi;
    }
    if (lane == 0) mine[b] = bi;
  };
  auto copy_offer = [&](int b) {
    const int bi = mine[b];
    if (bi == INT_MAX) return;
    const double* w = M + (size_t)(bi - r0) * n;
    for (int j = tid; j < n; j += kGjThreads) offer[(size_t)b * n + j] = w[j];
  };
  if (warp == 0) {
    double v[kGjLaneRows];
#pragma unroll
    for (int q = 0; q < kGjLaneRows; ++q)
      v[q] = lane + 32 * q < rc ? M[(size_t)(lane + 32 * q) * n] : 0.0;
    make_offer(0, v);
  }
  __syncthreads();
  copy_offer(0);

  for (int k = 0; k < n; ++k) {
    const int b = k & 1;  // offer buffers alternate between steps
    // every offer is visible cluster-wide; the buffers of step k - 1 are no
    // longer read by anyone
    cluster.sync();
    unsigned long long best = lane < C ? cand_k[b * kGjMaxCluster + lane] : 0ull;
    const int p = warp_best(best, lane < C ? cand_i[b * kGjMaxCluster + lane] : INT_MAX);
    // a zero (or NaN-only) column among the unused rows: singular
    if (best == 0ull) {
      if (c == 0 && tid == 0) *err = 1;
      cluster.sync();  // no CTA leaves while another may still read its offer
      return;
    }
    const int owner = p / R;
    const double ipiv = cand_inv[b * kGjMaxCluster + owner];
    const double* src = cluster.map_shared_rank(offer, (unsigned)owner) + (size_t)b * n;
    for (int j = tid; j < n; j += kGjThreads) prow[j] = src[j];
    // FP64 division is slow on this part: the offer brought 1 / a_pk, one warp
    // forms the row factors, the update multiplies
    double f0[kGjLaneRows], next[kGjLaneRows];
    if (warp == 0) {
      if (lane == 0) perm[k] = p;
#pragma unroll
      for (int q = 0; q < kGjLaneRows; ++q) {
        const int r = lane + 32 * q;
        f0[q] = next[q] = 0.0;
        if (r < rc) {
          if (r0 + r == p) used[q] = true;
          else f0[q] = M[(size_t)r * n + k] * ipiv;
          fr[r] = f0[q];
          if (k + 1 < n) next[q] = M[(size_t)r * n + k + 1];
        }
      }
    }
    __syncthreads();
    if (warp == 0 && k + 1 < n) {
      const double pn = prow[k + 1];
#pragma unroll
      for (int q = 0; q < kGjLaneRows; ++q) next[q] = __fma_rn(-f0[q], pn, next[q]);
      make_offer(b ^ 1, next);
    }
    for (int r = warp; r < rc; r += kGjWarps) {
      double* m = M + (size_t)r * n;
      if (r0 + r == p) {
        for (int j = lane; j < n; j += 32) m[j] = (j == k) ? ipiv : prow[j] * ipiv;
      } else {
        const double f = fr[r];
        for (int j = lane; j < n; j += 32) m[j] = (j == k) ? -f : __fma_rn(-f, prow[j], m[j]);
      }
    }
    __syncthreads();
    if (k + 1 < n) copy_offer(b ^ 1);
  }
  cluster.sync();  // the last offers have been read

  // A^{-1}[k][p_j] = M[p_k][j]
  for (int k = tid; k < n; k += kGjThreads) {
    const int g = perm[k];
    if (g >= r0 && g < r0 + rc) pos[g - r0] = k;
  }
  __syncthreads();
  for (int r = warp; r < rc; r += kGjWarps) {
    double* out = inv + (size_t)pos[r] * n;
    for (int j = lane; j < n; j += 32) out[perm[j]] = M[(size_t)r * n + j];
  }
}

struct GjConfig {
  int cluster = 0;   // 0: cluster launch unavailable
  size_t smem_max = 0;
};

// largest cluster (16, else 8) that can be resident with the largest shared
// memory a CTA may take on this device
GjConfig probe_gj() {
  GjConfig g;
  int dev = 0, optin = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) !=
          cudaSuccess) {
    cudaGetLastError();
    return g;
  }
  if (cudaFuncSetAttribute(k_gj_cluster, cudaFuncAttributeMaxDynamicSharedMemorySize, optin) !=
      cudaSuccess) {
    cudaGetLastError();
    return g;
  }
  for (int c : {16, 8}) {
    if (c > 8 && cudaFuncSetAttribute(k_gj_cluster, cudaFuncAttributeNonPortableClusterSizeAllowed,
                                      1) != cudaSuccess) {
      cudaGetLastError();
      continue;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    cfg.gridDim = dim3(c);
    cfg.blockDim = dim3(kGjThreads);
    cfg.dynamicSmemBytes = (size_t)optin;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = c;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int nclusters = 0;
    if (cudaOccupancyMaxActiveClusters(&nclusters, k_gj_cluster, &cfg) == cudaSuccess &&
        nclusters >= 1) {
      g.cluster = c;
      g.smem_max = (size_t)optin;
      return g;
    }
    cudaGetLastError();
  }
  return g;
}

}  // namespace

bool coarse_inverse_cluster(int n, const double* A, double* inv, int* err, cudaStream_t s) {
  static PerDevice<GjConfig> config;
  const GjConfig g = config(probe_gj);
  if (g.cluster == 0 || n < 1) return false;
  const int R = (n + g.cluster - 1) / g.cluster;
  const GjLayout lay(n, R);
  if (lay.bytes > g.smem_max || R > 32 * kGjLaneRows) return false;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  cfg.gridDim = dim3(g.cluster);
  cfg.blockDim = dim3(kGjThreads);
  cfg.dynamicSmemBytes = lay.bytes;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = g.cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  TP_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_gj_cluster, n, R, A, inv, err));
  return true;
}

}  // namespace tp
