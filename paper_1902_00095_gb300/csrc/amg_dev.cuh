// Device helpers shared by the AMG setup kernels (internal header).
#pragma once
#include "amg.cuh"

namespace tp {

constexpr signed char kC = 1, kF = -1, kU = 0;

// sign class of a_kk for opposite_class(): 0 when a_kk is zero or NaN (never
// opposite), 1 positive, 2 negative (one byte per entry in shared memory
// instead of the value)
__device__ __forceinline__ unsigned char sign_class(double d) {
  const unsigned long long ud = (unsigned long long)__double_as_longlong(d);
  const unsigned long long md = ud & 0x7fffffffffffffffull;
  if (md == 0 || md > 0x7ff0000000000000ull) return 0;
  return (unsigned char)(1 + (ud >> 63));
}

// (d > 0 && a < 0) || (d < 0 && a > 0) with d given by its sign class, decided
// on the bit patterns: integer operations instead of FP64 comparisons, which
// on this part share the FP64 pipe (2 per clock per SM) with the setup's
// multiply-adds and divisions
__device__ __forceinline__ bool opposite_class(double a, unsigned char dc) {
  const unsigned long long ua = (unsigned long long)__double_as_longlong(a);
  const unsigned long long ma = ua & 0x7fffffffffffffffull;
  return dc != 0 && ma != 0 && ma <= 0x7ff0000000000000ull &&
         (unsigned)(ua >> 63) != (unsigned)(dc - 1);
}

// an FP64 value is non-zero (either sign, or NaN), tested on its bits: FP64
// compares would take the FP64 pipe
__device__ __forceinline__ bool nonzero_bits(double v) {
  return ((unsigned long long)__double_as_longlong(v) << 1) != 0;
}

// |w| as an ordered integer, NaN lowest
__device__ __forceinline__ unsigned long long mag_key(double w) {
  const unsigned long long m =
      (unsigned long long)__double_as_longlong(w) & 0x7fffffffffffffffull;
  return m <= 0x7ff0000000000000ull ? m + 1 : 0;
}

// index of key in a[lo, hi) (ascending), or -1
__device__ __forceinline__ int find_in(const int* __restrict__ a, int lo, int hi, int key) {
  int h = hi;
  while (lo < hi) {
    int mid = (lo + hi) >> 1;
    if (a[mid] < key) lo = mid + 1;
    else hi = mid;
  }
  return (lo < h && a[lo] == key) ? lo : -1;
}

}  // namespace tp
