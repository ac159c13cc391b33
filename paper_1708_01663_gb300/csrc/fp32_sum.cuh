// A sum of FP32 values held as three of them: every addition's rounding error, which is an FP32 value itself (Knuth's
// TwoSum), goes into the second, and the second's into the third.  About 70 bits, so that value() is the exact sum
// rounded once where an FP64 sum rounds at every addition, for 13 FP32 additions instead of one in FP64 at 1/64 of
// the rate.  (Two values would keep about 46 bits, fewer than FP64.)  An overflow leaves value() not finite.
#pragma once

namespace cisor {

#ifdef __CUDACC__
#define CISOR_SUM_HD __host__ __device__ __forceinline__
#else
#define CISOR_SUM_HD inline
#endif

struct Fp32Sum {
  float s = 0.f, e = 0.f, c = 0.f;
  // s + p in s; the result is the rounding error
  static CISOR_SUM_HD float two_sum(float& s, float p) {
    const float t = s + p, b = t - s, r = (s - (t - b)) + (p - b);
    s = t;
    return r;
  }
  CISOR_SUM_HD void add(float p) { c += two_sum(e, two_sum(s, p)); }
  CISOR_SUM_HD void add(const Fp32Sum& o) {
    add(o.s);
    c += two_sum(e, o.e);
    c += o.c;
  }
  CISOR_SUM_HD double value() const { return (double)s + ((double)e + (double)c); }
};

}  // namespace cisor
