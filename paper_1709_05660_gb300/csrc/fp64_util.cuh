// Small FP64 helpers shared by the dense coarse-level kernels.  On GB300 the
// FP64 pipe retires two operations per SM and cycle, so comparisons of
// doubles are made on their bit patterns.
#pragma once

namespace fsi {
namespace {
constexpr int kWarp = 32;

// a != 0.0 (either sign of zero fails) as an integer test, off the FP64 pipe
__device__ __forceinline__ bool nonzero(double a) {
  return ((unsigned long long)__double_as_longlong(a) << 1) != 0ull;
}
__device__ __forceinline__ unsigned long long abs_key(double a) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(a) & 0x7FFFFFFFFFFFFFFFull;
  return b > 0x7FF0000000000000ull ? 0ull : b;   // NaN -> 0; +inf stays the largest
}
__device__ __forceinline__ bool key_wins(unsigned long long ok, int oi, unsigned long long k, int i) {
  return (oi >= 0 && i < 0) || (oi >= 0 && (ok > k || (ok == k && oi < i)));
}
}  // namespace
}  // namespace fsi
