// Device scans and deterministic reductions used by assembly and AMG setup.
#include "common.cuh"
#include <atomic>
#include <climits>

namespace tp {

static std::atomic<long long> g_launches{0};
thread_local bool g_capturing = false;

void count_launch(long long n) {
  if (!g_capturing) g_launches.fetch_add(n, std::memory_order_relaxed);
}

long long launches_total() { return g_launches.load(); }

namespace {

// Exclusive scans of per-row counts. The setup runs seven per level, most on
// levels of a few thousand rows, where launches and not bandwidth cost time:
// one block scans up to kScanOneMax values tile by tile in one launch; longer
// arrays take two launches, tile sums and then the scan itself, whose blocks
// each add up the sums of the tiles before theirs (at most a few thousand
// numbers from L2; no block waits for another). The kernel that knows the total
// also puts a second value beside it for the same read-back. (A recursive scan
// through 64-bit temporaries took five to seven operations.)
constexpr int kScanThreads = 1024;
constexpr int kScanOneMax = 32768;
constexpr int kScanLong = 1 << 24;  // from here tiles of four times the size

// values to scan: counts, or 1 where a point's state is the given one
struct ScanCounts {
  const int* in;
  __device__ __forceinline__ int operator()(int i) const { return in[i]; }
};
struct ScanStates {
  const signed char* state;
  signed char what;
  __device__ __forceinline__ int operator()(int i) const { return state[i] == what ? 1 : 0; }
};

// sum over the block, in every thread; s: 33 values of shared memory
__device__ __forceinline__ long long block_total(long long v, long long* s) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) s[wid] = v;
  __syncthreads();
  if (wid == 0) {
    long long t = s[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) s[32] = t;
  }
  __syncthreads();
  const long long r = s[32];
  __syncthreads();
  return r;
}

// scans the tile of ITEMS values per thread that starts at `base`, adds
// `before` to it; returns the tile's sum
template <int ITEMS, class L>
__device__ __forceinline__ long long scan_tile(L in, int* __restrict__ out, long long base, int n,
                                               long long before, long long* s) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const long long b = base + (long long)threadIdx.x * ITEMS;
  int v[ITEMS];
  long long run = 0;
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    v[k] = b + k < n ? in((int)(b + k)) : 0;
    run += v[k];
  }
  long long incl = run;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s[wid] = incl;
  __syncthreads();
  if (wid == 0) {
    long long t = s[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    s[lane] = t;
  }
  __syncthreads();
  long long at = before + incl - run + (wid > 0 ? s[wid - 1] : 0);
  const long long total = s[31];
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    if (b + k < n) out[b + k] = (int)at;
    at += v[k];
  }
  __syncthreads();
  return total;
}

// result[0] = total, result[1] = *extra (0 when null)
__device__ __forceinline__ void scan_finish(long long total, int* out, int n,
                                            const int* __restrict__ extra, long long* result) {
  if (threadIdx.x == 0) {
    out[n] = (int)total;
    result[0] = total;
    result[1] = extra ? *extra : 0;
  }
}

template <class L>
__global__ void __launch_bounds__(kScanThreads) k_scan_one(L in, int* out, int n,
                                                           const int* __restrict__ extra,
                                                           long long* __restrict__ result) {
  __shared__ long long s[33];
  constexpr int kItems = 8;
  long long before = 0;
  for (long long base = 0; base < n; base += kScanThreads * kItems)
    before += scan_tile<kItems>(in, out, base, n, before, s);
  scan_finish(before, out, n, extra, result);
}

template <int ITEMS, class L>
__global__ void __launch_bounds__(kScanThreads) k_scan_sums(L in, int n,
                                                            long long* __restrict__ sums) {
  __shared__ long long s[33];
  const long long base = (long long)blockIdx.x * kScanThreads * ITEMS;
  long long v = 0;
#pragma unroll
  for (int k = 0; k < ITEMS; ++k) {
    const long long i = base + (long long)k * kScanThreads + threadIdx.x;
    if (i < n) v += in((int)i);
  }
  v = block_total(v, s);
  if (threadIdx.x == 0) sums[blockIdx.x] = v;
}

template <int ITEMS, class L>
__global__ void __launch_bounds__(kScanThreads) k_scan_apply(L in, int* out, int n,
                                                             const long long* __restrict__ sums,
                                                             const int* __restrict__ extra,
                                                             long long* __restrict__ result) {
  __shared__ long long s[33];
  long long v = 0;
  for (int t = threadIdx.x; t < (int)blockIdx.x; t += kScanThreads) v += sums[t];
  const long long before = block_total(v, s);
  const long long base = (long long)blockIdx.x * kScanThreads * ITEMS;
  const long long tile = scan_tile<ITEMS>(in, out, base, n, before, s);
  if (blockIdx.x == gridDim.x - 1) scan_finish(before + tile, out, n, extra, result);
}

template <int ITEMS, class L>
void scan_two(L in, int* out, int n, const int* extra, long long* result, Pool& scratch,
              cudaStream_t s) {
  const int tiles = grid_for(n, kScanThreads * ITEMS);
  long long* sums = scratch.alloc<long long>(tiles);
  k_scan_sums<ITEMS><<<tiles, kScanThreads, 0, s>>>(in, n, sums);
  TP_LAUNCH_CHECK();
  k_scan_apply<ITEMS><<<tiles, kScanThreads, 0, s>>>(in, out, n, sums, extra, result);
  TP_LAUNCH_CHECK();
}

template <class L>
long long scan_values(L in, int* out, int n, Pool& scratch, cudaStream_t s, const int* extra,
                      int* extra_host) {
  long long* result = scratch.alloc<long long>(2);
  if (n <= kScanOneMax) {
    k_scan_one<<<1, kScanThreads, 0, s>>>(in, out, n, extra, result);
    TP_LAUNCH_CHECK();
  } else if (n < kScanLong) {
    scan_two<4>(in, out, n, extra, result, scratch, s);
  } else {
    scan_two<16>(in, out, n, extra, result, scratch, s);
  }
  long long h[2] = {0, 0};
  TP_CUDA_TRY(cudaMemcpyAsync(h, result, sizeof(h), cudaMemcpyDeviceToHost, s));
  TP_CUDA_TRY(cudaStreamSynchronize(s));
  if (extra_host) *extra_host = (int)h[1];
  if (h[0] > (long long)INT_MAX) fail(TP_ENOMEM, "scan total exceeds 32-bit index range");
  return h[0];
}

__global__ void k_partial_sums(const double* __restrict__ x, int n, double* __restrict__ partials) {
  __shared__ double sh[kBlock];
  double acc = 0.0;
  // block b owns the contiguous chunk [b*chunk, (b+1)*chunk)
  long long chunk = ((long long)n + gridDim.x - 1) / gridDim.x;
  long long lo = chunk * blockIdx.x, hi = lo + chunk;
  if (hi > n) hi = n;
  for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x) acc += x[i];
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) partials[blockIdx.x] = sh[0];
}

__global__ void k_sum_partials(const double* __restrict__ partials, int np, double* __restrict__ out) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < np; ++i) s += partials[i];
    *out = s;
  }
}

}  // namespace

long long scan_exclusive(const int* in, int* out, int n, Pool& scratch, cudaStream_t s,
                         const int* extra, int* extra_host) {
  return scan_values(ScanCounts{in}, out, n, scratch, s, extra, extra_host);
}

long long scan_states(const signed char* state, signed char what, int* out, int n, Pool& scratch,
                      cudaStream_t s, const int* extra, int* extra_host) {
  return scan_values(ScanStates{state, what}, out, n, scratch, s, extra, extra_host);
}

void sum_fixed(const double* x, int n, double* out, double* partials, int nparts, cudaStream_t s) {
  k_partial_sums<<<nparts, kBlock, 0, s>>>(x, n, partials);
  TP_LAUNCH_CHECK();
  k_sum_partials<<<1, 32, 0, s>>>(partials, nparts, out);
  TP_LAUNCH_CHECK();
}

}  // namespace tp
