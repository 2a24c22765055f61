// Sums of double-float values in three FP32 words, and their fixed-point values (host and device).
#pragma once

#include <cstring>

#ifdef __CUDACC__
#define VP_HD __host__ __device__
#else
#define VP_HD
#endif

namespace vp {

// s + e = a + b exactly (Knuth's TwoSum, no ordering of |a|, |b| assumed; additions only, so nothing is contracted).
VP_HD inline void two_sum(float a, float b, float& s, float& e) {
  s = a + b;
  const float bb = s - a;
  e = (a - (s - bb)) + (b - bb);
}

VP_HD inline unsigned bits_of(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  unsigned b;
  std::memcpy(&b, &x, sizeof(b));
  return b;
#endif
}

constexpr int kSumZero = -(1 << 28);  // exponent() of zero
constexpr int kFixedBits = 62;        // fixed(e) counts units of 2^(e - kFixedBits)

// A running sum hi + lo + lo2 of double-float values: the errors of hi and of lo are carried exactly, so the sum of n
// values of magnitudes M in all is off by at most 8 n^3 2^-72 M (an FP64 sum by n 2^-53 M, a double-float one by about
// n 2^-47 M) for the 20 additions that a double-float sum takes as well.
struct Sum3 {
  float hi = 0.f, lo = 0.f, lo2 = 0.f;
  VP_HD void add(float h, float l) {
    float e1, e2, e3;
    two_sum(hi, h, hi, e1);
    two_sum(lo, l, lo, e2);
    two_sum(lo, e1, lo, e3);
    lo2 += e2 + e3;
  }
  // hi the sum rounded to FP32, lo and lo2 what it leaves; a sum that has overflowed counts as zero.
  VP_HD void normalise() {
    two_sum(lo, lo2, lo, lo2);
    two_sum(hi, lo, hi, lo);
    two_sum(lo, lo2, lo, lo2);
    if (((bits_of(hi) >> 23) & 255) == 255) hi = lo = lo2 = 0.f;
  }
  // e with 2^(e - 1) <= |sum| < 2^e (after normalise).
  VP_HD int exponent() const {
    const unsigned b = bits_of(hi);
    const int f = (int)((b >> 23) & 255);
    const unsigned m = b & 0x7fffffu;
    if (f == 0) {
      int e = kSumZero;
      for (unsigned v = m; v; v >>= 1) e = e == kSumZero ? -148 : e + 1;
      return e;
    }
    const float below = hi < 0.f ? (lo != 0.f ? lo : lo2) : -(lo != 0.f ? lo : lo2);  // > 0: |sum| < |hi|
    return f - 126 - (m == 0 && below > 0.f ? 1 : 0);
  }
  // The sum in units of 2^(e - kFixedBits) for |sum| < 2^e, to one unit per word (after normalise).
  VP_HD long long fixed(int e) const { return word(hi, e) + word(lo, e) + word(lo2, e); }

 private:
  VP_HD static long long word(float x, int e) {
    const unsigned b = bits_of(x);
    const int f = (int)((b >> 23) & 255), sh = (f ? f : 1) - 150 - e + kFixedBits;
    const long long m = (long long)((b & 0x7fffffu) | (f ? 0x800000u : 0u));
    const long long v = sh >= 0 ? m << (sh & 63) : (sh > -32 ? m >> -sh : 0);
    return (int)b < 0 ? -v : v;
  }
};

}  // namespace vp
