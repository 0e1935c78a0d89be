// fft.cuh -- device building blocks of the power-of-two FFTs behind the Fourier
// pseudospectral operators (Mang & Biros, Sec. 3.3.1: derivatives by Fourier
// spectral methods on a periodic nodal grid).
//
// Conventions: forward transform X[k] = sum_j x[j] exp(-2 pi i jk/L), inverse
// with exp(+2 pi i jk/L) and 1/L. Inverse transforms are formed as
// conj(FFT(conj(x))), so only forward butterflies exist. Twiddles come from
// tables computed on the host in double precision and rounded once.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace reg {

constexpr int kSMs = 152;

// First statement of a kernel launched by chain() (internal.h): waits until the
// previous kernel of the stream has finished and its writes are visible, then
// lets the next one be set up. No effect under an ordinary launch. Blocks of
// the next kernel that are placed early are spread unevenly, which costs more
// than the launch gap where a kernel fills the GPU and its double-precision
// unit (128^3 FP64 gradient: 47.6 -> 56.3 ms), so only single-precision stages
// (early) and grids of at most one block per SM in x let it in before they end
// (y: the time nodes of k_dot_fields, the one kernel with two dimensions; 128^2 mixed
// matvec 610 us whether they count or not).
__device__ __forceinline__ void chain_enter(bool early = false) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (early || gridDim.x <= kSMs) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename T> struct Cx;
template <> struct Cx<float> { using type = float2; };
template <> struct Cx<double> { using type = double2; };
template <typename T> using cx = typename Cx<T>::type;

template <typename C> __device__ __forceinline__ C mk(decltype(C::x) a, decltype(C::x) b) {
  C c;
  c.x = a;
  c.y = b;
  return c;
}
template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return mk<C>(a.x + b.x, a.y + b.y); }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return mk<C>(a.x - b.x, a.y - b.y); }
template <typename C> __device__ __forceinline__ C cmul(C a, C b) {
  return mk<C>(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
template <typename C> __device__ __forceinline__ C cconj(C a) { return mk<C>(a.x, -a.y); }
// multiply by -i
template <typename C> __device__ __forceinline__ C cmul_mi(C a) { return mk<C>(a.y, -a.x); }
template <typename C> __device__ __forceinline__ C cscale(C a, decltype(C::x) s) { return mk<C>(a.x * s, a.y * s); }

// exp(-2 pi i q/16) for compile-time q in [0,16): the 16th roots of unity.
// cos(pi/8) and sin(pi/8) written out; sqrt(1/2) likewise.
// The constants are rounded to T at compile time, so a single-precision
// butterfly issues no double-precision conversion.
template <typename T, int q> __device__ __forceinline__ cx<T> root16() {
  constexpr T c1 = (T)0.92387953251128675613;  // cos(pi/8)
  constexpr T s1 = (T)0.38268343236508977173;  // sin(pi/8)
  constexpr T h = (T)0.70710678118654752440;   // sqrt(1/2)
  constexpr T o = (T)1, z = (T)0;
  constexpr T re[16] = {o, c1, h, s1, z, -s1, -h, -c1, -o, -c1, -h, -s1, z, s1, h, c1};
  constexpr T im[16] = {z, -s1, -h, -c1, -o, -c1, -h, -s1, z, s1, h, c1, o, c1, h, s1};
  constexpr T a = re[q], b = im[q];
  return mk<cx<T>>(a, b);
}

// o * exp(-2 pi i k / R) with compile-time k, R <= 16; trivial roots skip the multiply.
template <typename T, int R, int k> __device__ __forceinline__ cx<T> twid_const(cx<T> o) {
  constexpr int q = (k * 16 / R) % 16;
  if constexpr (q == 0) return o;
  else if constexpr (q == 4) return cmul_mi(o);
  else if constexpr (q == 8) return mk<cx<T>>(-o.x, -o.y);
  else if constexpr (q == 12) return mk<cx<T>>(-o.y, o.x);
  else return cmul(o, root16<T, q>());
}

// e + t and e - t of one radix-2 butterfly. Single precision issues each as
// one paired instruction (sm_100 and later; e - t as e + (-1) t, exact),
// the same roundings as the componentwise form. Twiddles that are multiples
// of -i (a swap and a sign) keep the componentwise form, where the sign
// folds into the addition.
template <typename T, int q>
__device__ __forceinline__ void bfly(cx<T> e, cx<T> t, cx<T>& a, cx<T>& b) {
  if constexpr (sizeof(T) == 4 && (q == 0 || q % 4 != 0)) {
    a = __fadd2_rn(e, t);
    b = __ffma2_rn(t, make_float2(-1.f, -1.f), e);
  } else {
    a = cadd(e, t);
    b = csub(e, t);
  }
}

// In-register forward DFT of size R (power of two, R <= 16): radix-2
// decimation in time, recursively.
template <typename T, int R> struct Dft {
  template <int k> static __device__ __forceinline__ void comb(cx<T>* v, const cx<T>* e, const cx<T>* o) {
    if constexpr (k < R / 2) {
      cx<T> t = twid_const<T, R, k>(o[k]);
      bfly<T, (k * 16 / R) % 16>(e[k], t, v[k], v[k + R / 2]);
      comb<k + 1>(v, e, o);
    }
  }
  static __device__ __forceinline__ void run(cx<T>* v) {
    cx<T> e[R / 2], o[R / 2];
#pragma unroll
    for (int i = 0; i < R / 2; ++i) {
      e[i] = v[2 * i];
      o[i] = v[2 * i + 1];
    }
    Dft<T, R / 2>::run(e);
    Dft<T, R / 2>::run(o);
    comb<0>(v, e, o);
  }
};
template <typename T> struct Dft<T, 1> {
  static __device__ __forceinline__ void run(cx<T>*) {}
};

}  // namespace reg
