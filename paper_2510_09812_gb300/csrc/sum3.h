// Sum of FP32 pairs to more than FP64's precision (host and device).
#pragma once

#ifndef GSPM_HD
#ifdef __CUDACC__
#define GSPM_HD __host__ __device__
#else
#define GSPM_HD
#endif
#endif

namespace gspm {

// s + e + f, the rounding errors of s kept in e and those of e in f (Ogita, Rump and Oishi, "Accurate
// sum and dot product", SIAM J. Sci. Comput. 26 (2005), Algorithm SumK with K = 3; TwoSum by Knuth).
struct Sum3 {
  float s = 0.f, e = 0.f, f = 0.f;
  GSPM_HD static float plus(float a, float b) {
#ifdef __CUDA_ARCH__
    return __fadd_rn(a, b);  // (never contracted or reassociated)
#else
    return a + b;
#endif
  }
  GSPM_HD static float two_sum(float& a, float b) {  // a += b, returns the rounding error
    const float t = plus(a, b), z = plus(t, -a);
    const float d = plus(plus(a, -plus(t, -z)), plus(b, -z));
    a = t;
    return d;
  }
  GSPM_HD void add(float bs, float be, float bf) {
    const float a = two_sum(s, bs), b = two_sum(e, be), c = two_sum(e, a);
    f = plus(plus(plus(f, bf), b), c);
  }
  GSPM_HD double value() const { return (double)s + ((double)e + (double)f); }
};

}  // namespace gspm
