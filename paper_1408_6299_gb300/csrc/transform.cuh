// transform.cuh -- double-precision Fourier transforms of whole fields, in
// 64-bit fixed point per line (fixed.cuh), for the Fourier-diagonal operators
// (Mang & Biros, Sec. 3.3.1, 3.3.3): rows of real values to packed half
// spectra and back, and complex columns.
//
// Two neighbouring real rows a, b form one complex line a + i b with transform
// Z; the half spectra follow from additions alone: A_k = (Z_k + conj Z_{L-k})/2,
// B_k = (Z_k - conj Z_{L-k})/(2i). Slot 0 of a packed row holds the DC and the
// Nyquist value (both real) as its real and imaginary part.
#pragma once
#include "internal.h"
#include "fixed.cuh"

namespace reg {

// the largest mag of the TS threads (c, j), j < TS, of a column; thread c + j TC
// of the block holds (c, j). red: scratch, free again after the next barrier.
template <int TC, int TS>
__device__ __forceinline__ unsigned line_max(unsigned mag, unsigned* red, int c, int j) {
  if constexpr (TS == 1) {
    return mag;
  } else {
#pragma unroll
    for (int o = TC; o < 32; o *= 2) mag = max(mag, __shfl_xor_sync(0xffffffffu, mag, o));
    constexpr int NW = TC >= 32 ? TS : TC * TS / 32;  // partial results per column
    if constexpr (NW > 1) {
      red[(TC >= 32 ? j : (int)threadIdx.x / 32) * TC + c] = mag;  // equal values where lanes share a slot
      __syncthreads();
#pragma unroll
      for (int w = 0; w < NW; ++w) mag = max(mag, red[w * TC + c]);
      __syncthreads();
    }
    return mag;
  }
}

// the largest of two mags over the TS neighbouring threads j < TS of a row line; red: scratch of the line
template <int TS, class Sync>
__device__ __forceinline__ void row_max(unsigned& mx, unsigned& my, unsigned* red, int j, const Sync& sync) {
  if constexpr (TS < 32) {
#pragma unroll
    for (int o = 1; o < TS; o *= 2) {
      mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      my = max(my, __shfl_xor_sync(0xffffffffu, my, o));
    }
  } else {
    mx = __reduce_max_sync(0xffffffffu, mx);
    my = __reduce_max_sync(0xffffffffu, my);
  }
  if constexpr (TS > 32) {  // the line's warps exchange their maxima
    red[j / 32] = mx;
    red[TS / 32 + j / 32] = my;
    sync();
#pragma unroll
    for (int w = 0; w < TS / 32; ++w) {
      mx = max(mx, red[w]);
      my = max(my, red[TS / 32 + w]);
    }
    sync();
  }
}

// the same with the sum of l1
template <int TC, int TS>
__device__ __forceinline__ void line_max_sum(unsigned& mag, float& l1, unsigned* red, int c, int j) {
  if constexpr (TS > 1) {
#pragma unroll
    for (int o = TC; o < 32; o *= 2) {
      mag = max(mag, __shfl_xor_sync(0xffffffffu, mag, o));
      l1 += __shfl_xor_sync(0xffffffffu, l1, o);
    }
    constexpr int NW = TC >= 32 ? TS : TC * TS / 32;
    if constexpr (NW > 1) {
      const int w0 = TC >= 32 ? j : (int)threadIdx.x / 32;
      float* sum = reinterpret_cast<float*>(red + NW * TC);
      red[w0 * TC + c] = mag;
      sum[w0 * TC + c] = l1;
      __syncthreads();
      l1 = 0.f;
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        mag = max(mag, red[w * TC + c]);
        l1 += sum[w * TC + c];
      }
      __syncthreads();
    }
  }
}
template <int TS, class Sync>
__device__ __forceinline__ void row_max_sum(unsigned& mag, float& l1, unsigned* red, int j, const Sync& sync) {
#pragma unroll
  for (int o = 1; o < (TS < 32 ? TS : 32); o *= 2) {
    mag = max(mag, __shfl_xor_sync(0xffffffffu, mag, o));
    l1 += __shfl_xor_sync(0xffffffffu, l1, o);
  }
  if constexpr (TS > 32) {
    float* sum = reinterpret_cast<float*>(red + TS / 32);
    red[j / 32] = mag;
    sum[j / 32] = l1;
    sync();
    l1 = 0.f;
#pragma unroll
    for (int w = 0; w < TS / 32; ++w) {
      mag = max(mag, red[w]);
      l1 += sum[w];
    }
    sync();
  }
}

// threads that transform together: a warp, or the first NFFT threads of the block
template <int TS, int NFFT>
struct RowSync {
  __device__ __forceinline__ void operator()() const {
    if constexpr (TS <= 32) __syncwarp();
    else asm volatile("bar.sync 1, %0;" ::"n"(NFFT) : "memory");
  }
};

}  // namespace reg
