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

// ---------------------------------------------------------------------------
// Products of FP64 matrices on the integer pipe.  GB300 retires 62 wide integer
// multiply-adds (32 x 32 + 64 bits) per SM and cycle, against two FP64 ones, so
// sums of products are formed in fixed point: a row of the left factor (a
// column of the right one) is scaled by the power of two above its largest
// entry to X = a 2^(57 - E), split into digits X = hi 2^29 + lo with
// |hi|, |lo| <= 2^28, and
//     sum_k a_k b_k = 2^(Ea + Eb - 56) (HH + MID / 2^29),
//     HH = sum hi_a hi_b,  MID = sum (hi_a lo_b + lo_a hi_b),
// both exact in 64 bits for up to 32 terms.  What is left out (the lo lo
// products, the rounding of X and of MID / 2^29) is below 2^-55 of the product
// of the two largest entries per term, where FP64 rounds each product to
// 2^-53 of itself.  (Exact integer products of a two-digit split, the family of
// Ozaki, Ogita, Oishi and Rump's splittings for accurate matrix products.)  Inverses of
// 73 Schwarz blocks of 204 to 372 unknowns against a refined extended-precision one,
// relative to the sweep with FP64 products: error in the norm 0.91 (worst block 7.5e-15
// against 5.0e-14), worst row 0.89, median entry 0.93.  Entries far below their row's
// largest lose: one solid block of 204 unknowns has its median entry 13 times worse
// (8e-14), with the norm and the rows better.
// ---------------------------------------------------------------------------
constexpr int kFixTerms = 32;

// exponent field of a (0 for zeros and denormals, 2047 for non-finite values)
__device__ __forceinline__ int fix_exp(double a) { return (int)((__double2hiint(a) >> 20) & 0x7FF); }

// digits (x: hi, y: lo) of a scaled by the exponent field emax >= fix_exp(a)
__device__ __forceinline__ int2 fix_digits(double a, int emax) {
  const long long b = __double_as_longlong(a);
  const int e = (int)((b >> 52) & 0x7FF), d = emax - e;
  long long x = e ? (b & 0xFFFFFFFFFFFFFll) | 0x10000000000000ll : 0ll;
  if (d <= 4) x <<= 4 - d;
  else x = d < 66 ? (x + (1ll << (d - 5))) >> (d - 4) : 0ll;
  if (b < 0) x = -x;
  const int hi = (int)((x + (1ll << 28)) >> 29);
  return make_int2(hi, (int)(x - ((long long)hi << 29)));
}

__device__ __forceinline__ void fix_mad(long long& hh, long long& mid, int2 a, int2 b) {
  hh += (long long)a.x * b.x;
  mid += (long long)a.x * b.y;
  mid += (long long)a.y * b.x;
}

// c + the sum of products, for the exponent fields of the two scales (a sum beyond
// the FP64 range is infinite, as the sum of the products would be)
__device__ __forceinline__ double fix_add(double c, long long hh, long long mid, int ea, int eb) {
  const long long s = hh + ((mid + (1ll << 28)) >> 29);
  const int se = ea + eb - 1077;
  const double scale = __hiloint2double(se <= 0 ? 0 : (se < 2047 ? se << 20 : 2047 << 20), 0);
  return s != 0 ? fma((double)s, scale, c) : c;
}
}  // namespace
}  // namespace fsi
