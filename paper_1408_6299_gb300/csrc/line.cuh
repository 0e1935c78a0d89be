// line.cuh -- spectral derivative of periodic lines held in registers and
// shared memory (Mang & Biros, Sec. 3.3.1: first derivatives by Fourier
// spectral methods, the Nyquist mode dropped).
//
// The derivative along an axis is a real linear operator, so it acts on a
// complex line x + i y as it acts on the two real lines x and y. Two
// neighbouring real lines therefore form one complex line: forward FFT,
// times i k~ / L, inverse FFT, and the two real derivatives come back as the
// real and the imaginary part. No field leaves physical space, no spectrum is
// packed or unpacked, and every axis is treated alike.
//
// A line of length L is spread over TS threads, E = L / TS complex values
// each. The stages of the forward plan (radices R(0..S-1)) exchange values
// through shared memory; the last one leaves thread j with the frequencies
// j + r L/R, exactly the inputs of the first stage of an inverse transform
// planned in the reversed order, so the multiplier is applied in registers and
// the line ends in the positions it started from.
#pragma once
#include "fft.cuh"

namespace reg {

// ---------------------------------------------------------------------------
// Plans. Wide: radices 16 and 8, the fewest operations and exchanges per
// point, for fields that fill the GPU. Narrow: radix 4, four values per
// thread, four times the threads and a quarter of the serial work of one
// thread, for fields whose wide form would leave most of the SMs idle.
// ---------------------------------------------------------------------------
template <int L, bool NARROW>
struct LinePlan;
#define REG_LINE_PLAN(LEN, NARROW, S_, R0, R1, R2, R3, R4, E_) \
  template <>                                                   \
  struct LinePlan<LEN, NARROW> {                                \
    static constexpr int S = S_;                                \
    __host__ __device__ static constexpr int R(int s) {         \
      return s == 0 ? R0 : (s == 1 ? R1 : (s == 2 ? R2 : (s == 3 ? R3 : R4))); \
    }                                                           \
    static constexpr int E = E_;                                \
    static constexpr int TS = LEN / E_;                         \
  };
REG_LINE_PLAN(8, false, 1, 8, 1, 1, 1, 1, 8)
REG_LINE_PLAN(16, false, 1, 16, 1, 1, 1, 1, 16)
REG_LINE_PLAN(32, false, 2, 8, 4, 1, 1, 1, 8)
REG_LINE_PLAN(64, false, 2, 8, 8, 1, 1, 1, 8)
REG_LINE_PLAN(128, false, 2, 16, 8, 1, 1, 1, 16)
REG_LINE_PLAN(256, false, 2, 16, 16, 1, 1, 1, 16)
REG_LINE_PLAN(512, false, 3, 8, 8, 8, 1, 1, 16)
REG_LINE_PLAN(8, true, 2, 4, 2, 1, 1, 1, 4)
REG_LINE_PLAN(16, true, 2, 4, 4, 1, 1, 1, 4)
REG_LINE_PLAN(32, true, 3, 4, 4, 2, 1, 1, 4)
REG_LINE_PLAN(64, true, 3, 4, 4, 4, 1, 1, 4)
REG_LINE_PLAN(128, true, 4, 4, 4, 4, 2, 1, 4)
REG_LINE_PLAN(256, true, 4, 4, 4, 4, 4, 1, 4)
REG_LINE_PLAN(512, true, 5, 4, 4, 4, 4, 2, 4)
#undef REG_LINE_PLAN

// threads of a wide line
inline int wide_threads(int L) {
  switch (L) {
    case 8: return LinePlan<8, false>::TS;
    case 16: return LinePlan<16, false>::TS;
    case 32: return LinePlan<32, false>::TS;
    case 64: return LinePlan<64, false>::TS;
    case 128: return LinePlan<128, false>::TS;
    case 256: return LinePlan<256, false>::TS;
    default: return LinePlan<512, false>::TS;
  }
}

// radix of forward stage s, of inverse stage s, and the product of the
// radices before stage s
template <class P>
__host__ __device__ constexpr int line_radix(int s, bool inv) {
  return inv ? P::R(P::S - 1 - s) : P::R(s);
}
template <class P>
__host__ __device__ constexpr int line_ns(int s, bool inv) {
  int n = 1;
  for (int t = 0; t < s; ++t) n *= line_radix<P>(t, inv);
  return n;
}
// Offset of stage s's twiddle block in the table of a plan. Stage s >= 1
// stores W_{Ns R}^{r k} at [r Ns + k]. Block 0: the forward stages, block 1: the
// inverse ones; block 2 (fixed point): the forward stages without their scaling.
template <class P>
__host__ __device__ constexpr int line_tw_block(bool inv) {
  int n = 0;
  for (int t = 1; t < P::S; ++t) n += line_ns<P>(t, inv) * line_radix<P>(t, inv);
  return n;
}
template <class P>
__host__ __device__ constexpr int line_tw_offset(int s, bool inv) {
  int off = inv ? line_tw_block<P>(false) : 0;
  for (int t = 1; t < s; ++t) off += line_ns<P>(t, inv) * line_radix<P>(t, inv);
  return off;
}

// Bytes of the fixed-point tables of the wide plans of every length: 3 blocks of
// 16-byte entries (50,688 bytes).
template <int L = 512>
__host__ __device__ constexpr size_t wide_table_bytes() {
  using P = LinePlan<L, false>;
  const size_t n = (size_t)(2 * line_tw_block<P>(false) + line_tw_block<P>(true)) * 16;
  if constexpr (L > 8) return n + wide_table_bytes<L / 2>();
  else return n;
}

// Real additions and multiplications of one forward transform along the wide
// plan (radix-2 butterflies, general roots and stage twiddles as 6 each).
__host__ __device__ constexpr double dft_flops(int R) {
  if (R <= 1) return 0.0;
  int general = 0;
  for (int k = 0; k < R / 2; ++k)
    if (((k * 16 / R) % 16) % 4 != 0) ++general;
  return 2.0 * dft_flops(R / 2) + 2.0 * R + 6.0 * general;
}
template <int L>
constexpr double fft_flops() {
  using P = LinePlan<L, false>;
  double f = 0.0;
  for (int s = 0; s < P::S; ++s) {
    const int r = line_radix<P>(s, false);
    f += (double)(L / r) * dft_flops(r);
    if (s > 0) f += (double)(L / r) * (r - 1) * 6.0;
  }
  return f;
}

__host__ __device__ constexpr int ilog2_c(int n) { return n <= 1 ? 0 : 1 + ilog2_c(n / 2); }

// ---------------------------------------------------------------------------
// Arithmetic of one complex value. V: the value; W: a table entry.
// ---------------------------------------------------------------------------
template <typename T>
struct LineFloat {
  using V = cx<T>;
  using W = cx<T>;
  using G = cx<T>;                       // what it reads and writes: CW complex columns
  static constexpr int CW = 1;
  static constexpr int TABLE = 0;        // kind of its twiddle table
  static constexpr bool SCALED = false;  // values are taken as they are
  static __device__ __forceinline__ V in(G x) { return x; }
  static __device__ __forceinline__ G out(V z) { return cconj(z); }
  template <int R>
  static __device__ __forceinline__ void dft(V* v) {
    Dft<T, R>::run(v);
  }
  // times a table twiddle of a forward stage of radix R / of an inverse stage
  template <int R>
  static __device__ __forceinline__ V twiddle_fwd(V a, W w) {
    return cmul(a, w);
  }
  static __device__ __forceinline__ V twiddle_inv(V a, W w) { return cmul(a, w); }
  // the untwiddled element r = 0 of a forward stage of radix R
  template <int R>
  static __device__ __forceinline__ V pass_fwd(V a) {
    return a;
  }
  // conj(i k~ z / L) for frequency f < L (f = L/2 dropped)
  template <int L>
  static __device__ __forceinline__ V deriv(V z, int f) {
    const T k = (f < L / 2 ? (T)f : (f == L / 2 ? (T)0 : (T)(f - L))) * ((T)1 / (T)L);
    return mk<V>(-k * z.y, -k * z.x);
  }
};

// Single precision, two neighbouring columns per thread: a float2 holds the
// same quantity of both, and the butterflies run as paired instructions
// (add, fma and mul on float2, sm_100 and later), half the arithmetic
// instructions of one column per thread.
struct __align__(16) P2 {
  float2 re, im;
};
__device__ __forceinline__ P2 p2_add(P2 a, P2 b) { return {__fadd2_rn(a.re, b.re), __fadd2_rn(a.im, b.im)}; }
// a - b as a + (-1) b in one fused operation per half (exact: the product by -1 is not rounded)
__device__ __forceinline__ P2 p2_sub(P2 a, P2 b) {
  const float2 m1 = make_float2(-1.f, -1.f);
  return {__ffma2_rn(b.re, m1, a.re), __ffma2_rn(b.im, m1, a.im)};
}
// times the complex scalar (c, s), given as the duplicated pairs (c, c) and (s, s)
__device__ __forceinline__ P2 p2_mul(P2 a, float2 cc, float2 ss) {
  const float2 nss = __fmul2_rn(ss, make_float2(-1.f, -1.f));
  return {__ffma2_rn(a.re, cc, __fmul2_rn(a.im, nss)), __ffma2_rn(a.re, ss, __fmul2_rn(a.im, cc))};
}
template <int R, int k>
__device__ __forceinline__ P2 p2_twid(P2 o) {
  constexpr int q = (k * 16 / R) % 16;
  if constexpr (q == 0) return o;
  else if constexpr (q == 4) return {o.im, make_float2(-o.re.x, -o.re.y)};  // times -i
  else if constexpr (q == 8) return {make_float2(-o.re.x, -o.re.y), make_float2(-o.im.x, -o.im.y)};
  else if constexpr (q == 12) return {make_float2(-o.im.x, -o.im.y), o.re};  // times i
  else {
    const float2 w = root16<float, q>();
    return p2_mul(o, make_float2(w.x, w.x), make_float2(w.y, w.y));
  }
}
// forward DFT of size R on paired values (radix-2 decimation in time, as Dft)
template <int R>
struct P2Dft {
  template <int k>
  static __device__ __forceinline__ void comb(P2* v, const P2* e, const P2* o) {
    if constexpr (k < R / 2) {
      const P2 t = p2_twid<R, k>(o[k]);
      v[k] = p2_add(e[k], t);
      v[k + R / 2] = p2_sub(e[k], t);
      comb<k + 1>(v, e, o);
    }
  }
  static __device__ __forceinline__ void run(P2* v) {
    P2 e[R / 2], o[R / 2];
#pragma unroll
    for (int i = 0; i < R / 2; ++i) {
      e[i] = v[2 * i];
      o[i] = v[2 * i + 1];
    }
    P2Dft<R / 2>::run(e);
    P2Dft<R / 2>::run(o);
    comb<0>(v, e, o);
  }
};
template <>
struct P2Dft<1> {
  static __device__ __forceinline__ void run(P2*) {}
};

struct LinePair {
  using V = P2;
  using W = float4;  // (c, c, s, s)
  using G = float4;
  static constexpr int CW = 2, TABLE = 1;
  static constexpr bool SCALED = false;
  static __device__ __forceinline__ V in(G x) { return {make_float2(x.x, x.z), make_float2(x.y, x.w)}; }
  static __device__ __forceinline__ G out(V z) { return make_float4(z.re.x, -z.im.x, z.re.y, -z.im.y); }
  template <int R>
  static __device__ __forceinline__ void dft(V* v) {
    P2Dft<R>::run(v);
  }
  template <int R>
  static __device__ __forceinline__ V twiddle_fwd(V a, W w) {
    return p2_mul(a, make_float2(w.x, w.y), make_float2(w.z, w.w));
  }
  static __device__ __forceinline__ V twiddle_inv(V a, W w) {
    return p2_mul(a, make_float2(w.x, w.y), make_float2(w.z, w.w));
  }
  template <int R>
  static __device__ __forceinline__ V pass_fwd(V a) {
    return a;
  }
  template <int L>
  static __device__ __forceinline__ V deriv(V z, int f) {
    const float k = (f < L / 2 ? (float)f : (f == L / 2 ? 0.f : (float)(f - L))) * (1.f / (float)L);
    const float2 nk = make_float2(-k, -k);
    return {__fmul2_rn(z.im, nk), __fmul2_rn(z.re, nk)};
  }
};

// ---------------------------------------------------------------------------
// The derivative. v holds the positions t + r Q (Q = L / R(0)) of the line for
// this thread's tasks t = j + i TS, i < E / R(0), at v[i R(0) + r]; on return
// the conjugate of the derivative, in the same positions. buf(p) is the shared
// slot of position p (free on entry; not synchronised on return); sync()
// separates the exchanges of the threads that share buf.
// ---------------------------------------------------------------------------
template <class A, int L, bool NARROW>
struct Line {
  using P = LinePlan<L, NARROW>;
  using V = typename A::V;
  using W = typename A::W;
  static constexpr int E = P::E, TS = P::TS, S = P::S;
  static constexpr int R0 = P::R(0), Q0 = L / R0;

  // Narrow kernels load a thread's forward twiddles into registers before they
  // wait for their predecessor, and the inverse ones ahead of the inverse
  // stages: a stage would otherwise begin with a miss to L2, as L1 is empty when
  // a kernel starts (128^2 mixed matvec 613 us, without it 680; 512^2 FP64 transport
  // 4709 and 4913). Order: stages s >= 1 of one direction.
  static constexpr bool PRELOAD = NARROW;
  __host__ __device__ static constexpr int tw_index(int s, bool inv) {
    int n = 0;
    for (int t = 1; t < s; ++t) {
      const int R = inv ? P::R(S - 1 - t) : P::R(t);
      n += E / R * (R - 1);
    }
    return n;
  }
  static constexpr int NTW = PRELOAD ? tw_index(S, false) : 0;
  template <int s, bool INV>
  static __device__ __forceinline__ void load_stages(W* w, int j, const W* __restrict__ tw) {
    if constexpr (s < S) {
      constexpr int R = line_radix<P>(s, INV), NS = line_ns<P>(s, INV), TK = E / R;
      const W* t0 = tw + line_tw_offset<P>(s, INV);
#pragma unroll
      for (int i = 0; i < TK; ++i)
#pragma unroll
        for (int r = 1; r < R; ++r)
          w[tw_index(s, INV) + i * (R - 1) + r - 1] = __ldg(&t0[r * NS + ((j + i * TS) & (NS - 1))]);
      load_stages<s + 1, INV>(w, j, tw);
    }
  }
  static __device__ __forceinline__ void preload(W* w, int j, const W* __restrict__ tw) {
    if constexpr (PRELOAD) load_stages<1, false>(w, j, tw);
  }

  // position of v[i * R0 + r]
  static __device__ __forceinline__ int position(int j, int e) { return j + (e / R0) * TS + (e % R0) * Q0; }

  // PRE: tw is the thread's preloaded array
  template <int s, bool INV, bool PRE, class Buf, class Sync>
  static __device__ __forceinline__ void stages(V* v, int j, const Buf& buf, const Sync& sync, const W* tw,
                                                bool scaled = true) {
    constexpr int R = line_radix<P>(s, INV), NS = line_ns<P>(s, INV), Q = L / R, TK = E / R;
    if constexpr (s > 0) {
      const W* t0 = tw + (PRE ? 0 : line_tw_offset<P>(s, INV));
#pragma unroll
      for (int i = 0; i < TK; ++i) {
        const int t = j + i * TS;
#pragma unroll
        for (int r = 0; r < R; ++r) v[i * R + r] = *buf(t + r * Q);
        if constexpr (!INV)
          if (scaled) v[i * R] = A::template pass_fwd<R>(v[i * R]);
#pragma unroll
        for (int r = 1; r < R; ++r) {
          W w;
          if constexpr (PRE) w = t0[tw_index(s, INV) + i * (R - 1) + r - 1];
          else w = __ldg(&t0[r * NS + (t & (NS - 1))]);
          if constexpr (INV) v[i * R + r] = A::twiddle_inv(v[i * R + r], w);
          else v[i * R + r] = A::template twiddle_fwd<R>(v[i * R + r], w);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < TK; ++i) A::template dft<R>(v + i * R);
    if constexpr (s < S - 1) {
      if constexpr (s > 0 || INV) sync();  // every value of the previous exchange has been read
#pragma unroll
      for (int i = 0; i < TK; ++i) {
        const int t = j + i * TS;
        const int base = (t / NS) * (NS * R) + (t & (NS - 1));
#pragma unroll
        for (int r = 0; r < R; ++r) *buf(base + r * NS) = v[i * R + r];
      }
      sync();
      stages<s + 1, INV, PRE>(v, j, buf, sync, tw, scaled);
    }
  }

  // Forward transform: v as in derivative(), on return v[e] is the value of
  // frequency(j, e). buf is left with the last exchange (not synchronised).
  // scaled: fixed-point stages take their inputs times 1/R, as derivative() does.
  static __device__ __forceinline__ int frequency(int j, int e) {
    constexpr int R = line_radix<P>(S - 1, false);
    return j + (e / R) * TS + (e % R) * (L / R);
  }
  template <class Buf, class Sync>
  static __device__ __forceinline__ void forward(V* v, int j, const Buf& buf, const Sync& sync, const W* tw,
                                                 bool scaled) {
    stages<0, false, false>(v, j, buf, sync, scaled ? tw : tw + line_tw_block<P>(false) + line_tw_block<P>(true), scaled);
  }

  // pre: what preload() filled (PRELOAD plans)
  template <class Buf, class Sync>
  static __device__ __forceinline__ void derivative(V* v, int j, const Buf& buf, const Sync& sync,
                                                    const W* __restrict__ tw, const W* pre) {
    stages<0, false, PRELOAD>(v, j, buf, sync, PRELOAD ? pre : tw);
    W inv[PRELOAD ? tw_index(S, true) + 1 : 1];
    if constexpr (PRELOAD) load_stages<1, true>(inv, j, tw);
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = A::template deriv<L>(v[e], frequency(j, e));
    stages<0, true, PRELOAD>(v, j, buf, sync, PRELOAD ? inv : tw);
  }
};

}  // namespace reg
