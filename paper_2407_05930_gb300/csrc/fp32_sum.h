// Sums of FP32 numbers to better than FP64's own rounding, in FP32 arithmetic.
#pragma once

#include <cmath>

#ifdef __CUDACC__
#define AMGSYM_HD __host__ __device__ __forceinline__
#else
#define AMGSYM_HD inline
#endif

namespace amgsym {

// An unevaluated sum of three FP32 numbers: Knuth's two-sum leaves the exact
// error of hi + x, a second one the exact error of adding that to mid, and only
// those second errors are summed with rounding, in lo.  With u = 2^-24 and S the
// sum of magnitudes of n numbers, mid stays below n u S, so lo sums errors of
// together at most n^2 u^2 S / 2 and is off by at most n^3 u^3 S / 2: 2^-61 S
// for the 16 numbers a thread adds at most, where n additions in FP64 may be off
// by (n - 1) 2^-53 S.  value() rounds twice in FP64.
struct Fp32Sum {
  float hi = 0.f, mid = 0.f, lo = 0.f;
  AMGSYM_HD static float two_sum(float a, float b, float* err) {
    const float t = a + b;
    const float br = t - a;
    *err = (a - (t - br)) + (b - br);
    return t;
  }
  AMGSYM_HD void add(float x) {
    float e1, e2;
    hi = two_sum(hi, x, &e1);
    mid = two_sum(mid, e1, &e2);
    lo += e2;
  }
  AMGSYM_HD double value() const { return (double)hi + ((double)mid + (double)lo); }
};

// The sum of col[first], col[first + step], ... below col[count].  Numbers of
// 2^90 or more, infinities and NaN are summed in FP64: the FP32 sum could
// overflow, or turn an infinity into a NaN.
AMGSYM_HD double fp32_sum(const float* col, int first, int step, int count) {
  Fp32Sum s;
  bool big = false;
  for (int r = first; r < count; r += step) {
    const float x = col[r];
    big |= !(fabsf(x) < 0x1p90f);
    s.add(x);
  }
  if (!big) return s.value();
  double v = 0.0;
  for (int r = first; r < count; r += step) v += (double)col[r];
  return v;
}

}  // namespace amgsym
