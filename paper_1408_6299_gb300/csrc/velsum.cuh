// velsum.cuh -- sums of products of double-precision weights and
// single-precision values in single-precision arithmetic, rounded once (the
// velocity v(t_j) = sum_l T_l(2 t_j - 1) v_l of the mixed path, Mang & Biros,
// Sec. 3.3.2). GB300's double-precision unit takes two operations per clock and
// SM: the 19 per value of four 64^3 nodes of three coefficients would hold it for
// 26 us. Paired instructions (two floats, sm_100 and later) halve the count of what
// stands here for it.
#pragma once
#include <math.h>
#include <string.h>

#ifdef __CUDACC__
#define REG_HD __host__ __device__ __forceinline__
#else
#define REG_HD inline
#endif

namespace reg {

// one or two values; every result is rounded by itself (never contracted)
REG_HD float splat(float a, float) { return a; }
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
REG_HD float sub_rn(float a, float b) { return add_rn(a, -b); }
// rounded towards zero
REG_HD float add_rz(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rz(a, b);
#else
  const float s = a + b, z = s - a, e = (a - (s - z)) + (b - z);
  return e != 0.f && (e > 0.f) != (s > 0.f) ? nextafterf(s, 0.f) : s;
#endif
}
REG_HD float fma_rn(float a, float b, float c) { return fmaf(a, b, c); }
#ifdef __CUDACC__
__device__ __forceinline__ float2 splat(float a, float2) { return make_float2(a, a); }
__device__ __forceinline__ float2 mul_rn(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add_rn(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub_rn(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }
__device__ __forceinline__ float2 add_rz(float2 a, float2 b) { return __fadd2_rz(a, b); }
__device__ __forceinline__ float2 fma_rn(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
#endif

// a + b = s + e exactly (Knuth)
template <class V>
REG_HD void two_sum(V a, V b, V& s, V& e) {
  s = add_rn(a, b);
  const V z = sub_rn(s, a);
  e = add_rn(sub_rn(a, sub_rn(s, z)), sub_rn(b, z));
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

// one lane of FloatSum::rounded
REG_HD float round_lane(float s, float a, float b, float c, float x, float y, float t) {
  unsigned i;
  memcpy(&i, &c, sizeof i);
  if (x != t || y != b) i |= 1u;
  memcpy(&c, &i, sizeof i);
  return fabsf(a) <= 3.402823466e38f ? add_rn(a, c) : s;  // s: an infinity or a NaN
}
REG_HD void round_lanes(float s, float a, float b, float c, float x, float y, float t, float* r) {
  *r = round_lane(s, a, b, c, x, y, t);
}
#ifdef __CUDACC__
__device__ __forceinline__ void round_lanes(float2 s, float2 a, float2 b, float2 c, float2 x, float2 y, float2 t, float* r) {
  r[0] = round_lane(s.x, a.x, b.x, c.x, x.x, y.x, t.x);
  r[1] = round_lane(s.y, a.y, b.y, c.y, x.y, y.y, t.y);
}
#endif

// A sum held as s + e + t: s and e take what is added without error, t what e
// rounds off, with a rounding of 2^-72 of the terms. No further off than a sum of
// doubles rounded at the end (2^-53 of the terms), which a pair of floats with
// weights of 48 bits was by up to 850 units where terms cancel. The first
// weight is that of T_0, one.
template <class V>
struct FloatSum {
  V s, e, t;
  REG_HD void put(V x) {
    V f;
    two_sum(e, x, e, f);
    t = add_rn(t, f);
  }
  // term l of the sum, in order; SHORT: no weight has a second word
  template <bool SHORT>
  REG_HD void add(int l, const FloatWeight& w, V u) {
    if (l == 0) {
      s = u;
      e = t = splat(0.f, u);
      return;
    }
    const V h = splat(w.hi, u), n = mul_rn(splat(-w.hi, u), u);  // n = -h u
    const V r = sub_rn(s, n), z = sub_rn(r, s);                  // two_sum of s and h u
    const V d = sub_rn(sub_rn(s, sub_rn(r, z)), add_rn(n, z));
    s = r;
    if (l == 1) {
      two_sum(fma_rn(h, u, n), d, e, t);
    } else {
      put(fma_rn(h, u, n));
      put(d);
    }
    if (!SHORT) {
      const V q = mul_rn(splat(w.mid, u), u);
      put(q);
      t = fma_rn(splat(w.lo, u), u, sub_rn(t, fma_rn(splat(-w.mid, u), u, q)));
    }
  }
  // The sum to nearest: with s + e = a + b, b + t is rounded to odd (towards zero,
  // the last bit set where that dropped something), so that its sum with a rounds as
  // the exact one would.
  REG_HD void rounded(float* r) const {
    V a, b;
    two_sum(s, e, a, b);
    const V c = add_rz(b, t);
    round_lanes(s, a, b, c, sub_rn(c, b), sub_rn(c, t), t, r);
  }
};

}  // namespace reg
