// Grid position of an FP64 coordinate in 2^-32 units, in integer arithmetic.
// Plain C++ (host and device), no CUDA headers, so that a host test can check
// it against exact arithmetic.
//
// t = (x - lo) s is one FP64 subtraction and one multiplication; everything
// after them (the range test, floor t, the fraction and its rounding to 2^-32)
// works on the bits of t.  FP64 instructions run at 2 lanes per clock and SM
// on sm_103, integer ones at 64 or more, and the same steps in FP64 (two
// compares, floor, two conversions, a subtraction, a scaling) were three
// quarters of the binning kernels' time on FP64 samples.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define KDE_FP_HD __host__ __device__ __forceinline__
#else
#define KDE_FP_HD inline
#endif

namespace kde {

// For 0 <= t <= top (bits of t and of top; top < 2^24): *V = t 2^32 rounded
// half to even, so node i = V >> 32 and q = V mod 2^32 (a fraction that
// rounds up to one gives the next node with q = 0).  Returns false, leaving
// *V alone, for t < 0, t > top, infinities and NaN; -0 counts as 0.
// Non-negative doubles order like their bits, and 2^32 floor(t) is even, so
// rounding the whole of t 2^32 rounds the fraction's 2^32 f the same way.
KDE_FP_HD bool fixed_position(uint64_t bits, uint64_t top_bits, uint64_t* V) {
  if (bits == 0x8000000000000000ull) bits = 0;
  if (bits > top_bits) return false;   // negative, above top, infinite or NaN
  const int e = (int)(bits >> 52);
  const uint64_t m = (bits & 0xFFFFFFFFFFFFFull) | (e ? 0x10000000000000ull : 0ull);
  const int shift = 1043 - e;          // t 2^32 = m 2^-shift
  if (shift <= 0) {
    *V = m << -shift;                  // t < 2^24: at most 3 places
  } else if (shift > 53) {
    *V = 0;                            // m < 2^53: below one half
  } else {
    const uint64_t r = m >> shift, rem = m << (64 - shift);
    *V = r + (rem > 0x8000000000000000ull || (rem == 0x8000000000000000ull && (r & 1)) ? 1 : 0);
  }
  return true;
}

}  // namespace kde
