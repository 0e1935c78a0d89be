// fixed.cuh -- double-precision lines in 64-bit fixed point.
//
// GB300 issues two double-precision operations per clock and SM, one warp
// instruction every 64 cycles per scheduler, but about sixty 64-bit integer
// additions. A transform is additions with a few multiplications, and its
// values stay within a known factor of the largest input, so a line is scaled
// to 64-bit integers once, transformed in integer arithmetic, and scaled back.
//
// Scaling. All values of a line are below 2^e in magnitude. They become
// integers x 2^(S0 - e), S0 = G - log2 R0: after the first stage (radix R0) a
// value is below sqrt(2) 2^G. Every later forward stage of radix R takes its
// inputs times 1/R (inside the twiddle), so that bound holds throughout, and
// the frequencies come out at 2^(S - e), S = G - log2 L. The inverse stages
// do not scale: their partial sums are bounded by the derivative itself, below
// |D|_1 sqrt(2) 2^S with |D|_1 = sum_k |cot(pi k / L)| / 2 (the absolute row
// sum of the derivative matrix: 406 at L = 256, 924 at L = 512). G = 61, and 60
// at L = 512, keeps every sum below 2^63.
//
// The two real lines of a complex line may have a scale each, since the operator is
// real: rows do (k_rows_line), so that a row keeps its own accuracy beside one of
// another size (with one scale 4e-9 of itself beside a row 10^8 times larger). Neighbouring columns share one: every column meets every row.
//
// Accuracy. The rounding of the inputs to 2^(e - S0) and of the products to one
// unit is below that of double-precision butterflies: on smooth, blob and
// white-noise lines the error against extended precision is 0.1 to 0.45 of the
// double-precision transform's (L = 8 to 512); only a line that is a single
// spike comes out up to 2 times further off (6e-16 against 3e-16).
#pragma once
#include "line.cuh"

namespace reg {

struct __align__(16) FxV {
  long long x, y;
};

__device__ __forceinline__ FxV operator+(FxV a, FxV b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ FxV operator-(FxV a, FxV b) { return {a.x - b.x, a.y - b.y}; }

// low word as a signed number and the matching high word
__device__ __forceinline__ int fx_lo(long long v) { return (int)v; }
__device__ __forceinline__ int fx_hi(long long v) { return (int)(v >> 32) + (int)((unsigned)v >> 31); }

// (a 2^32 + t) >> 30 with t's high word already added into a
__device__ __forceinline__ long long fx_shift30(long long a, unsigned t) {
  const unsigned lo = __funnelshift_r(t, (unsigned)a, 30);
  const unsigned hi = __funnelshift_r((unsigned)a, (unsigned)((unsigned long long)a >> 32), 30);
  return (long long)(((unsigned long long)hi << 32) | lo);
}

// A real factor w = h 2^-30 + l 2^-62 (l signed). Products drop the term of
// both low words (below one unit) and round the rest to the nearest unit.
__device__ __forceinline__ long long fx_mul(long long v, int h, int l) {
  const int vl = fx_lo(v), vh = fx_hi(v);
  long long t = (long long)vl * h + (1LL << 29);
  if (l != 0) t += (long long)vh * l;
  const long long a = (long long)vh * h + (t >> 32);
  return fx_shift30(a, (unsigned)t);
}
// u (h, l) + v (m, n), rounded once
__device__ __forceinline__ long long fx_mul2(int ul, int uh, int h, int l, int vl, int vh, int m, int n) {
  long long t = (long long)ul * h + (1LL << 29);
  t += (long long)uh * l;
  t += (long long)vl * m;
  t += (long long)vh * n;
  long long a = (long long)uh * h + (t >> 32);
  a += (long long)vh * m;
  return fx_shift30(a, (unsigned)t);
}
// times the complex factor (ch, cl) + i (sh, sl)
__device__ __forceinline__ FxV fx_cmul(FxV z, int ch, int cl, int sh, int sl) {
  const int xl = fx_lo(z.x), xh = fx_hi(z.x), yl = fx_lo(z.y), yh = fx_hi(z.y);
  return {fx_mul2(xl, xh, ch, cl, yl, yh, -sh, -sl), fx_mul2(xl, xh, sh, sl, yl, yh, ch, cl)};
}

// cos(pi/8), sin(pi/8), sqrt(1/2) times 2^62, split as h 2^32 + l
constexpr int kFxC1h = 992008094, kFxC1l = 1696238673;
constexpr int kFxS1h = 410903207, kFxS1l = -1364630830;
constexpr int kFxHh = 759250125, kFxHl = -25716447;

// o * exp(-2 pi i k / R), compile-time k < R / 2, R <= 16
template <int R, int k>
__device__ __forceinline__ FxV fx_twid(FxV o) {
  constexpr int q = k * 16 / R;
  if constexpr (q == 0) return o;
  else if constexpr (q == 1) return fx_cmul(o, kFxC1h, kFxC1l, -kFxS1h, -kFxS1l);
  else if constexpr (q == 2) return {fx_mul(o.x + o.y, kFxHh, kFxHl), fx_mul(o.y - o.x, kFxHh, kFxHl)};
  else if constexpr (q == 3) return fx_cmul(o, kFxS1h, kFxS1l, -kFxC1h, -kFxC1l);
  else if constexpr (q == 4) return {o.y, -o.x};
  else if constexpr (q == 5) return fx_cmul(o, -kFxS1h, -kFxS1l, -kFxC1h, -kFxC1l);
  else if constexpr (q == 6) return {fx_mul(o.y - o.x, kFxHh, kFxHl), fx_mul(-o.x - o.y, kFxHh, kFxHl)};
  else return fx_cmul(o, -kFxC1h, -kFxC1l, -kFxS1h, -kFxS1l);
}

template <int R>
struct FxDft {
  template <int k>
  static __device__ __forceinline__ void comb(FxV* v, const FxV* e, const FxV* o) {
    if constexpr (k < R / 2) {
      const FxV t = fx_twid<R, k>(o[k]);
      v[k] = e[k] + t;
      v[k + R / 2] = e[k] - t;
      comb<k + 1>(v, e, o);
    }
  }
  static __device__ __forceinline__ void run(FxV* v) {
    FxV e[R / 2], o[R / 2];
#pragma unroll
    for (int i = 0; i < R / 2; ++i) {
      e[i] = v[2 * i];
      o[i] = v[2 * i + 1];
    }
    FxDft<R / 2>::run(e);
    FxDft<R / 2>::run(o);
    comb<0>(v, e, o);
  }
};
template <>
struct FxDft<1> {
  static __device__ __forceinline__ void run(FxV*) {}
};

// Line arithmetic (see line.cuh). W: the factor's words (ch, cl, sh, sl); the
// tables of the forward stages hold the twiddles times 1/R.
struct LineFixed {
  using V = FxV;
  using W = int4;
  using G = double2;  // what it reads and writes
  static constexpr bool SCALED = true;
  static constexpr int CW = 1, TABLE = 1;
  template <int R>
  static __device__ __forceinline__ void dft(V* v) {
    FxDft<R>::run(v);
  }
  template <int R>
  static __device__ __forceinline__ V twiddle_fwd(V a, W w) {
    return fx_cmul(a, w.x, w.y, w.z, w.w);
  }
  static __device__ __forceinline__ V twiddle_inv(V a, W w) { return fx_cmul(a, w.x, w.y, w.z, w.w); }
  template <int R>
  static __device__ __forceinline__ V pass_fwd(V a) {
    return {(a.x + R / 2) >> ilog2_c(R), (a.y + R / 2) >> ilog2_c(R)};
  }
  template <int L>
  static __device__ __forceinline__ V deriv(V z, int f) {
    const int k = f < L / 2 ? f : (f == L / 2 ? 0 : f - L);
    const int h = -k * (1 << (30 - ilog2_c(L)));  // -k / L, exact
    return {fx_mul(z.y, h, 0), fx_mul(z.x, h, 0)};
  }
};

template <int L>
__host__ __device__ constexpr int fx_headroom() {
  return L == 512 ? 60 : 61;
}

// a magnitude as the high word of a double (ordered as an unsigned number), its
// lowest bit set by low words: subnormal values without a high word are not zero
__device__ __forceinline__ unsigned fx_mag(double x) {
  return ((unsigned)__double2hiint(x) & 0x7fffffffu) | min((unsigned)__double2loint(x), 1u);
}
// the larger one of a pair
__device__ __forceinline__ unsigned fx_mag(double2 x) {
  return max((unsigned)__double2hiint(x.x) & 0x7fffffffu, (unsigned)__double2hiint(x.y) & 0x7fffffffu) |
         min((unsigned)(__double2loint(x.x) | __double2loint(x.y)), 1u);
}

// |x| + |y| to about 2^-20, for magnitudes from 2^-126 to 2^100 (smaller ones
// count as zero), from the high words alone
__device__ __forceinline__ float fx_l1(double2 x) {
  auto f = [](double v) {
    const int h = min(__double2hiint(v) & 0x7fffffff, (1023 + 100) << 20);
    return __int_as_float(max(h - (896 << 20), 0) << 3);
  };
  return f(x.x) + f(x.y);
}

// Scaling of one line from the high word of its largest magnitude. Lines whose
// values are near the ends of the exponent range are first moved by 2^+-300
// (pre) and back (post); a line that holds an infinity or a NaN comes out as NaN.
template <int L, int R0>
struct FxScale {
  static constexpr int S0 = fx_headroom<L>() - ilog2_c(R0), S = fx_headroom<L>() - ilog2_c(L);
  enum Kind { PLAIN, TINY, HUGE_, NONFINITE, ZERO };
  int right, down;  // in1: shift of a value with exponent field 0; exponent shift of the results (high word)
  Kind kind;
  bool plain;
  bool scaled = true;  // the forward stages scale (see Line::forward)
  __device__ __forceinline__ explicit FxScale(unsigned mag) {
    int e = (int)(mag >> 20);
    kind = mag == 0 ? ZERO : (e < 64 ? TINY : (e <= 1990 ? PLAIN : (e < 2047 ? HUGE_ : NONFINITE)));
    plain = kind == PLAIN || kind == ZERO;
    if (kind == ZERO || kind == NONFINITE) e = 1023;
    else if (kind != PLAIN) e = __double2hiint(__hiloint2double((int)mag, -1) * pre()) >> 20;
    right = 63 - S0 + e;
    down = (e - 1022 - S) * (1 << 20);
  }
  __device__ __forceinline__ double pre() const { return kind == TINY ? 0x1p300 : (kind == HUGE_ ? 0x1p-300 : 1.0); }
  __device__ __forceinline__ double post() const {
    return kind == TINY ? 0x1p-300 : (kind == HUGE_ ? 0x1p300 : (kind == NONFINITE ? __hiloint2double(0x7ff80000, 0) : 1.0));
  }
  // Conversions in integer arithmetic: the double-precision unit converts two
  // values per clock and SM, and the epilogues need it. Rounded to nearest.
  __device__ __forceinline__ long long in1(double x) const {
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x);
    // the 53-bit significand times 2^10, shifted right by r >= 1; r counts up for smaller values
    const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
    const unsigned long long m = ((unsigned long long)__funnelshift_l(lo, mh, 10) << 32) | (lo << 10);
    const int r = right - ((hi >> 20) & 0x7ff);
    const unsigned long long v = ((r > 64 ? 0ull : m >> (r - 1)) + 1) >> 1;
    const long long sign = (long long)(hi >> 31);
    return (long long)(v ^ (unsigned long long)sign) - sign;
  }
  // on the double-precision unit: one conversion and an exponent shift
  __device__ __forceinline__ double out1(long long r) const {
    const double d = __ll2double_rn(r);
    return r == 0 ? 0.0 : __hiloint2double(__double2hiint(d) + down, __double2loint(d));
  }
  // on the integer units
  __device__ __forceinline__ double out1i(long long r) const {
    const long long sign = r >> 63;
    const unsigned long long a = (unsigned long long)((r ^ sign) - sign);
    const int lz = __clzll((long long)a);
    // leading one at bit 62, rounded at bit 10; a carry moves into the exponent by itself
    const unsigned long long n = ((a << lz) >> 1) + 0x200;
    const unsigned hi = (unsigned)(n >> 42) + (unsigned)((1085 - lz) * (1 << 20) + down);
    const unsigned lo = __funnelshift_r((unsigned)n, (unsigned)(n >> 32), 10);
    return r == 0 ? 0.0 : __hiloint2double((int)(hi | ((unsigned)(sign >> 32) & 0x80000000u)), (int)lo);
  }
  // A line whose sum of magnitudes l1 (see fx_l1) is far below L times its
  // largest value, as the lines of a decaying spectrum are: no partial sum
  // exceeds l1, so it is scaled by l1 and its stages do not scale, which keeps
  // its rounding at one unit of that sum (256 points, spectrum |k|^-1: error
  // 6e-17 against 4e-16 with the scaling stages and 1.7e-16 in double precision).
  __device__ __forceinline__ void by_sum(unsigned mag, float l1) {
    const int e = (int)(mag >> 20);
    if (e < 1023 - 90 || e > 1023 + 90) return;  // outside fx_l1's range (or inf, NaN)
    const int h = (int)(__float_as_uint(l1 * 1.0001f) >> 23) - 126 - (e - 1022);  // l1 < 2^(e - 1022 + h)
    if (h > ilog2_c(L) - 2) return;
    scaled = false;
    const int s = fx_headroom<L>() - (h > 0 ? h : 0);
    right = 63 - s + e;
    down = (e - 1022 - s) * (1 << 20);
  }
  // results times 2^n as well
  __device__ __forceinline__ void times_pow2(int n) { down += n * (1 << 20); }
  // v = x scaled, for the E values a thread holds of the line; im: the scale of the
  // imaginary parts, a real line of its own
  template <int E>
  __device__ __forceinline__ void in(const double2 (&x)[E], FxV (&v)[E]) const {
    in(*this, x, v);
  }
  template <int E>
  __device__ __forceinline__ void in(const FxScale& im, const double2 (&x)[E], FxV (&v)[E]) const {
    if (plain && im.plain) {
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] = {in1(x[e].x), im.in1(x[e].y)};
    } else {
#pragma unroll
      for (int e = 0; e < E; ++e)
        v[e] = {kind == NONFINITE ? 0 : in1(x[e].x * pre()), im.kind == NONFINITE ? 0 : im.in1(x[e].y * im.pre())};
    }
  }
  __device__ __forceinline__ double back(long long r) const { return plain ? out1(r) : out1(r) * post(); }
  // x = the conjugate of v, scaled back; INT: on the integer units
  template <bool INT, int E>
  __device__ __forceinline__ void out(const FxV (&v)[E], double2 (&x)[E]) const {
    out<INT>(*this, v, x);
  }
  template <bool INT, int E>
  __device__ __forceinline__ void out(const FxScale& im, const FxV (&v)[E], double2 (&x)[E]) const {
#pragma unroll
    for (int e = 0; e < E; ++e)
      x[e] = INT ? make_double2(out1i(v[e].x), im.out1i(-v[e].y)) : make_double2(out1(v[e].x), im.out1(-v[e].y));
    if (!(plain && im.plain)) {
#pragma unroll
      for (int e = 0; e < E; ++e) x[e] = make_double2(x[e].x * post(), x[e].y * im.post());
    }
  }
  // a zero line beside another takes its roundings: none of them is its own
  template <int E>
  __device__ __forceinline__ void keep_zero(const FxScale& im, double2 (&x)[E]) const {
    if (kind == ZERO) {
#pragma unroll
      for (int e = 0; e < E; ++e) x[e].x = 0.0;
    }
    if (im.kind == ZERO) {
#pragma unroll
      for (int e = 0; e < E; ++e) x[e].y = 0.0;
    }
  }
};

}  // namespace reg
