// velsum.cuh -- sums of products of double-precision weights and
// single-precision values in single-precision arithmetic, rounded once (the
// velocity v(t_j) = sum_l T_l(2 t_j - 1) v_l of the mixed path, Mang & Biros,
// Sec. 3.3.2). GB300's double-precision unit takes two operations per clock and
// SM: the 19 per value of four 64^3 nodes of three coefficients would hold it for 26 us.
#pragma once
#include <math.h>
#include <string.h>

#ifdef __CUDACC__
#define REG_HD __host__ __device__ __forceinline__
#else
#define REG_HD inline
#endif

namespace reg {

// products and sums that are rounded by themselves (never contracted)
REG_HD float mul_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  return a * b;
#endif
}
REG_HD float add_rn(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  return a + b;
#endif
}
// a + b = s + e exactly (Knuth)
REG_HD void two_sum(float a, float b, float& s, float& e) {
  s = add_rn(a, b);
  const float z = add_rn(s, -a);
  e = add_rn(add_rn(a, -add_rn(s, -z)), add_rn(b, -z));
}

// a double as hi + mid + lo, exactly
struct FloatWeight {
  float hi, mid, lo;
};
inline FloatWeight split_weight(double c) {
  FloatWeight w;
  w.hi = (float)c;
  w.mid = (float)(c - (double)w.hi);
  w.lo = (float)(c - (double)w.hi - (double)w.mid);
  return w;
}

// A sum held as s + e + t: s and e take what is added without error, t what e
// rounds off, with a rounding of 2^-72 of the terms, and the result is rounded to
// nearest. No further off than a sum of doubles rounded at the end (2^-53 of the
// terms), which a pair of floats with weights of 48 bits was by up to 850 units where
// terms cancel.
struct FloatSum {
  float s = 0.f, e = 0.f, t = 0.f;
  REG_HD void put(float x) {
    float f;
    two_sum(e, x, e, f);
    t = add_rn(t, f);
  }
  REG_HD void add(const FloatWeight& w, float u) {
    float d;
    const float p = mul_rn(w.hi, u);
    two_sum(s, p, s, d);
    put(fmaf(w.hi, u, -p));
    put(d);
    if (w.mid != 0.f) {  // the weights of a power of two of time steps have none
      const float q = mul_rn(w.mid, u);
      put(q);
      t = add_rn(t, fmaf(w.lo, u, fmaf(w.mid, u, -q)));
    }
  }
  REG_HD float rounded() const {
    float a, b, c;
    two_sum(s, e, a, b);
    if (!(fabsf(a) <= 3.402823466e38f)) return s;  // an infinity or a NaN
    two_sum(b, t, b, c);
    // b to odd: then a + b rounds as a + b + c would
    unsigned i;
    memcpy(&i, &b, sizeof i);
    if (c != 0.f && !(i & 1)) i += (c > 0.f) == (b > 0.f) ? 1u : ~0u;
    memcpy(&b, &i, sizeof i);
    return add_rn(a, b);
  }
};

}  // namespace reg
