// stage.cuh -- transport stages of the Heun sweeps (Mang & Biros, Eq.
// first-order-forward / first-order-adjoint / gauss-newton, Sec. 3.3.1).
//
// A stage is one launch of column passes and one row pass:
//   columns  the derivatives along the strided axes, each field (or product of
//            two fields) read once and its derivative written once;
//   rows     the derivative along the contiguous last axis, and with it the
//            stage's pointwise epilogue, which reads the column derivatives:
//     advection  k = -v . grad u [- grad m . v~], Heun update, optional store of grad u
//     divergence k = div(v lam),                  Heun update
// Both work on real fields: two neighbouring real lines form one complex line
// (line.cuh). Spectra are never stored.
#pragma once
#include "internal.h"
#include "transform.cuh"

namespace reg {
namespace fused {

// Epilogue parameters of the advection stage (state / incremental state).
template <typename T>
struct AdvEpi {
  const T* a[3];   // velocity components at the stage time
  const T* gm[3];  // source: grad m at the stage time (null: no source)
  const T* w[3];   // source: incremental velocity at the stage time
  const T* y;      // y_j (stage 1: null = 0)
  const T* yh;     // stage 2: the predictor y_j + h k_1, i.e. u
  T* out1;         // stage 1: y_j + h k_1; stage 2: y_{j+1} (null: only keep grad u)
  T* G[3];         // optional: keep grad u (null: not stored)
  const T* src;    // optional precomputed source sum_i gm_i w_i (used instead of gm/w)
  const T* sw[3];  // optional: with Sout, store Sout = sum_i (grad u)_i sw_i
  T* Sout;
  T h;
  int stage;
  int src_from_a;  // two-field stage, second field: the source is the first field's Sout value
  int a_from_a;    // two-field stage, second field: same velocity as the first (reuse its loaded values)
};

// Epilogue parameters of the divergence stage (adjoint / incremental adjoint).
// Stage 0 only evaluates: out1 = div(v lam) (+ src). src (optional) is added
// to the divergence (the div(v~ lam) source of the full Newton incremental
// adjoint).
template <typename T>
struct DivEpi {
  const T* y;   // lam_{j+1}
  const T* yh;  // stage 2: the predictor
  T* out1;
  T h;
  int stage;
  const T* src;  // added to the divergence
};

// Accesses that are not repeated before the next stage: first to leave the
// caches, so that the differentiated field and the derivative along the second
// axis, which the next pass reads, stay in L2 (256^3 mixed matvec 176.4 -> 173.8
// ms, 128^3 FP64 gradient 47.6 -> 45.2 ms).
template <typename C>
__device__ __forceinline__ C ld_stream(const C* p) {
  return __ldcs(p);
}
template <typename C>
__device__ __forceinline__ void st_stream(C* p, C v) {
  __stcs(p, v);
}

// y_{j+1} = y_j + h/2 (k_1 + k_2) from the predictor yh = y_j + h k_1, which
// carries k_1: the first stage stores no second field. yh - y_j is exact while the
// increment is below y_j, else rounded to half a unit of the increment; h k_2 and
// the result are rounded once each (256^3 mixed matvec 166 -> 156 ms against storing
// y_j + h/2 k_1 as well; error of 32 steps against extended precision 3.1e-16,
// 4.1e-16 that way).
template <typename T>
__device__ __forceinline__ T heun_end(T y, T yh, T k, T h) {
  return y + (T)0.5 * ((yh - y) + h * k);
}
template <typename T>
__device__ __forceinline__ cx<T> heun_end(cx<T> y, cx<T> yh, cx<T> k, T h) {
  return mk<cx<T>>(heun_end(y.x, yh.x, k.x, h), heun_end(y.y, yh.y, k.y, h));
}

// Advection epilogue on the point pair q with the gradient components g[0..D)
// (-a.g [- source], Heun update, optional keep of g or of g.sw). srcv, when
// given, is the source value instead of e.src. Returns the Sout value.
// av_in: the velocity values at q (null: load them); av_out: receives the
// loaded velocity values when the Heun update ran.
template <typename T, int D>
__device__ __forceinline__ cx<T> adv_point(const AdvEpi<T>& e, const cx<T>* g, long q, const cx<T>* srcv,
                                           const cx<T>* av_in = nullptr, cx<T>* av_out = nullptr) {
  using C = cx<T>;
  C so = mk<C>(0, 0);
  if (e.G[0]) {
#pragma unroll
    for (int f = 0; f < D; ++f) st_stream(reinterpret_cast<C*>(e.G[f]) + q, g[f]);
  }
  if (e.Sout) {
    T s0 = 0, s1 = 0;
#pragma unroll
    for (int f = 0; f < D; ++f) {
      C w = ld_stream(reinterpret_cast<const C*>(e.sw[f]) + q);
      s0 += g[f].x * w.x;
      s1 += g[f].y * w.y;
    }
    so = mk<C>(s0, s1);
    st_stream(reinterpret_cast<C*>(e.Sout) + q, so);
  }
  if (!e.out1) return so;
  T k0 = 0, k1 = 0;
#pragma unroll
  for (int f = 0; f < D; ++f) {
    C a = av_in ? av_in[f] : ld_stream(reinterpret_cast<const C*>(e.a[f]) + q);
    if (av_out) av_out[f] = a;
    k0 -= a.x * g[f].x;
    k1 -= a.y * g[f].y;
  }
  if (srcv) {
    k0 -= srcv->x;
    k1 -= srcv->y;
  } else if (e.src) {
    C sv = ld_stream(reinterpret_cast<const C*>(e.src) + q);
    k0 -= sv.x;
    k1 -= sv.y;
  } else if (e.gm[0]) {
#pragma unroll
    for (int f = 0; f < D; ++f) {
      C gm = ld_stream(reinterpret_cast<const C*>(e.gm[f]) + q);
      C w = ld_stream(reinterpret_cast<const C*>(e.w[f]) + q);
      k0 -= gm.x * w.x;
      k1 -= gm.y * w.y;
    }
  }
  const C yv = e.y ? ld_stream(reinterpret_cast<const C*>(e.y) + q) : mk<C>(0, 0);
  C r1;
  if (e.stage == 1) {
    r1 = mk<C>(yv.x + e.h * k0, yv.y + e.h * k1);
  } else {
    const C yh = ld_stream(reinterpret_cast<const C*>(e.yh) + q);
    r1 = heun_end<T>(yv, yh, mk<C>(k0, k1), e.h);
  }
  reinterpret_cast<C*>(e.out1)[q] = r1;
  return so;
}

// Divergence epilogue on the point pair q with the divergence value k: Heun
// stage update.
template <typename T>
__device__ __forceinline__ void div_point(const DivEpi<T>& dv, cx<T> k, long q) {
  using C = cx<T>;
  if (dv.src) {
    C sv = ld_stream(reinterpret_cast<const C*>(dv.src) + q);
    k = mk<C>(k.x + sv.x, k.y + sv.y);
  }
  if (dv.stage == 0) {
    reinterpret_cast<C*>(dv.out1)[q] = k;
    return;
  }
  const C yv = ld_stream(reinterpret_cast<const C*>(dv.y) + q);
  C r;
  if (dv.stage == 1) r = mk<C>(yv.x + dv.h * k.x, yv.y + dv.h * k.y);
  else r = heun_end<T>(yv, ld_stream(reinterpret_cast<const C*>(dv.yh) + q), k, dv.h);
  reinterpret_cast<C*>(dv.out1)[q] = r;
}

// ---------------------------------------------------------------------------
// Column passes
// ---------------------------------------------------------------------------
constexpr int kColJobs = 4;
// Up to four derivative passes along axes of the same length L: out = D in, or
// D (in mul). s: distance of two line elements (complex values, a power of
// two); n: complex lines of the field (the pairs of neighbouring real lines).
template <typename T>
struct ColJobs {
  const T* in[kColJobs];
  const T* mul[kColJobs];
  T* out[kColJobs];
  int log2s[kColJobs];
  int start[kColJobs + 1];  // first block of each job; start[nj] = all blocks
  int nj;
  int n;
  int stream[kColJobs];  // write out past the cache (axis-0 passes)
};

// Threads of a block: TS along a line times TC neighbouring lines. VAR: 0, or 1
// for the other block size the autotuner may choose; both give the same bits.
// Wide: 128-byte row segments where the block allows it. Narrow: one warp or
// one line (the most blocks; 512^2 FP64 transport 4700 us, with four lines at least
// 6370, 128^2 mixed matvec 613 and 671), or four lines and at least 128 threads.
template <class A, int L, bool NARROW, int VAR>
struct ColTile {
  static constexpr int TS = LinePlan<L, NARROW>::TS;
  static constexpr int LINE = L * (int)sizeof(typename A::V);  // shared bytes of a line
  static constexpr int NT0 = NARROW ? (VAR ? 128 : 32) : (sizeof(typename A::V) == 8 ? 256 : 128) / (VAR ? 2 : 1);
  static constexpr int MINTC = NARROW ? (VAR ? 4 : 1) : (VAR ? 4 : 8);
  static constexpr int TC1 = NT0 / TS < MINTC ? MINTC : NT0 / TS;
  static constexpr int fit(int tc) { return tc * LINE <= 49152 ? tc : fit(tc / 2); }  // 48 KB of shared memory
  static constexpr int TC = fit(TC1);
  static constexpr int NT = TC * TS;
};

__device__ __forceinline__ float2 gmul(float2 a, float2 b) { return make_float2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ double2 gmul(double2 a, double2 b) { return make_double2(a.x * b.x, a.y * b.y); }
__device__ __forceinline__ float4 gmul(float4 a, float4 b) {
  return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w);
}

// Job q of block tile
template <typename T>
__device__ __forceinline__ int col_job(const ColJobs<T>& J, int& tile) {
  int q = 0;
#pragma unroll
  for (int k = 1; k < kColJobs; ++k)
    if (k < J.nj && tile >= J.start[k]) q = k;
  tile -= J.start[q];
  return q;
}

// TC neighbouring lines of job q; buf: L * TC values
template <class A, typename T, int L, bool NARROW, bool PROD, int TC>
__device__ __forceinline__ void cols_tile(const ColJobs<T>& J, int q, int tile, int n, typename A::V* buf,
                                          const typename A::W* __restrict__ tw) {
  using Ln = Line<A, L, NARROW>;
  using V = typename A::V;
  using G = typename A::G;
  constexpr int E = Ln::E, TS = LinePlan<L, NARROW>::TS;
  const int c = threadIdx.x % TC, j = threadIdx.x / TC;
  typename A::W pre[Ln::NTW + 1];
  Ln::preload(pre, j, tw);
  chain_enter(sizeof(T) == 4);
  const int line = tile * TC + c;
  const int ls = J.log2s[q];
  const long s = 1L << ls;
  const long off = ((long)(line >> ls) * L << ls) + (line & (int)(s - 1));
  const bool ok = line < n;
  G x[E];
  {
    const G* in = reinterpret_cast<const G*>(J.in[q]) + off;
#pragma unroll
    for (int e = 0; e < E; ++e)
      x[e] = ok ? (PROD ? ld_stream(in + Ln::position(j, e) * s) : in[Ln::position(j, e) * s]) : G{};
    if constexpr (PROD) {
      const G* mul = reinterpret_cast<const G*>(J.mul[q]) + off;
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (ok) x[e] = gmul(x[e], mul[Ln::position(j, e) * s]);
    }
  }
  V v[E];
  auto at = [&](int p) { return buf + p * TC + c; };
  auto sync = [] { __syncthreads(); };
  G* out = reinterpret_cast<G*>(J.out[q]) + off;
  if constexpr (A::SCALED) {
    unsigned mag = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) mag = max(mag, fx_mag(x[e]));
    const FxScale<L, Ln::R0> sc(line_max<TC, TS>(mag, reinterpret_cast<unsigned*>(buf), c, j));
    sc.in(x, v);
    Ln::derivative(v, j, at, sync, tw, pre);
    if (!ok) return;
    sc.template out<NARROW>(v, x);
#pragma unroll
    for (int e = 0; e < E; ++e) out[Ln::position(j, e) * s] = x[e];
  } else {
#pragma unroll
    for (int e = 0; e < E; ++e) v[e] = A::in(x[e]);
    Ln::derivative(v, j, at, sync, tw, pre);
    if (!ok) return;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      if (J.stream[q]) st_stream(out + Ln::position(j, e) * s, A::out(v[e]));
      else out[Ln::position(j, e) * s] = A::out(v[e]);
    }
  }
}

template <class A, typename T, int L, bool NARROW, bool PROD, int VAR>
__global__ void __launch_bounds__(ColTile<A, L, NARROW, VAR>::NT) k_cols_line(ColJobs<T> J,
                                                                          const typename A::W* __restrict__ tw) {
  constexpr int TC = ColTile<A, L, NARROW, VAR>::TC;
  __shared__ typename A::V buf[L * TC];
  int tile = blockIdx.x;
  const int q = col_job(J, tile);
  cols_tile<A, T, L, NARROW, PROD, TC>(J, q, tile, J.n, buf, tw);
}

// Jobs along axes of two lengths up to 256 (narrow plans): the length is
// uniform in a block of 64 threads, one or several lines of it. One launch,
// chained to its predecessor and successor, instead of one per length on forked
// streams (one_cols_launch has the figures).
constexpr int kTwoNT = 64;
template <class A>
struct TwoAxes {
  const typename A::W* tw[2];
  int lg[2], n[2];  // log2 of the length, lines of a field
  int axis[kColJobs];
};
template <class A, typename T, bool PROD>
__global__ void __launch_bounds__(kTwoNT) k_cols_two(const __grid_constant__ ColJobs<T> J,
                                                    const __grid_constant__ TwoAxes<A> P) {
  __shared__ typename A::V buf[kTwoNT * 4];
  int tile = blockIdx.x;
  const int q = col_job(J, tile), a = P.axis[q];
  auto go = [&](auto len) {
    constexpr int L = decltype(len)::value;
    static_assert(LinePlan<L, true>::E == 4, "lines of a block fill buf");
    cols_tile<A, T, L, true, PROD, kTwoNT / LinePlan<L, true>::TS>(J, q, tile, P.n[a], buf, P.tw[a]);
  };
  switch (P.lg[a]) {
    case 3: return go(std::integral_constant<int, 8>{});
    case 4: return go(std::integral_constant<int, 16>{});
    case 5: return go(std::integral_constant<int, 32>{});
    case 6: return go(std::integral_constant<int, 64>{});
    case 7: return go(std::integral_constant<int, 128>{});
    default: return go(std::integral_constant<int, 256>{});
  }
}

// ---------------------------------------------------------------------------
// Row pass with the stage epilogue
// ---------------------------------------------------------------------------
// ADV2, ADV3: advection in 2D / 3D; ADV33: two 3D advection stages (fields u[0]
// and u[1]); DIV: divergence (2D and 3D)
enum { EPI_ADV2 = 0, EPI_ADV3 = 1, EPI_ADV33 = 2, EPI_DIV = 3 };

template <typename T>
struct RowArgs {
  const T* u[2];   // differentiated fields (DIV: u[0] times mul)
  const T* mul;
  const T* gx[2];  // derivatives along the first axis (DIV: of the first product)
  const T* gy[2];  // along the second axis (3D)
  AdvEpi<T> adv, advB;
  DivEpi<T> dv;
  long nrows;
  int rev;  // blocks take the rows from the last one
};

// In single precision the two rows of a complex line are brought to one size by
// powers of two, and back: their errors mix, and a row keeps its own accuracy beside
// a larger one (its derivative is its own, where those along strided axes mix all
// rows; without, a row came out 1e-2 of itself wrong beside one 10^6 times its
// size). row_binade: the power of two of a row's largest magnitude, as the bits of a
// float, from the bits of that magnitude; 0 for a zero row, which so stays zero.
__device__ __forceinline__ unsigned row_binade(unsigned mag) {
  return min(max(mag & 0x7f800000u, min(mag, 1u) << 23), 253u << 23);
}

// Rows r and r + 1 (r even) form one complex line; a block holds NSEQ of them.
// FEW (narrow plans): one or two lines per block, transformed by part of its
// threads and their epilogue spread over all of them: the shortest pass where
// lines are few. Else every thread transforms, and a line that fits a warp stays in
// it with the epilogue of its rows, so the warps never wait for one another.
template <int L, bool NARROW, bool FEW, int EPI>
struct RowTile {
  using P = LinePlan<L, NARROW>;
  static constexpr int TS = P::TS;
  static constexpr int NF = EPI == EPI_ADV33 ? 2 : 1;
  static constexpr int MINSEQ = 32 / TS > NF ? 32 / TS : NF;
  static constexpr int FULLSEQ = 128 / TS > NF ? 128 / TS : NF;
  static constexpr int NSEQ = FEW ? MINSEQ : FULLSEQ;
  static constexpr int NFFT = NSEQ * TS;  // transforming threads
  static constexpr int NT = NFFT > 128 ? NFFT : 128;
  static constexpr bool WARP = !FEW && 32 / TS >= NF;  // each warp alone
  static constexpr int PADSH = P::R(0) == 16 ? 4 : (P::R(0) == 8 ? 3 : 2);
  static constexpr int RS = (L + (L >> PADSH) + 1) / 2 * 2;
  static constexpr int ROWS = NSEQ / NF * 2;  // rows of one field per block
  // blocks per SM asked of the compiler (0: its choice). The wide two-field pass in
  // single precision, bound by memory, is held to 56 registers: 256^3 mixed matvec
  // 157.4 ms with 58, 154 so
  static constexpr int min_blocks(int size) { return size == 4 && !NARROW && L <= 256 && EPI == EPI_ADV33 ? 9 : 0; }
};

template <class A, typename T, int L, bool NARROW, bool FEW, int EPI>
__global__ void __launch_bounds__(RowTile<L, NARROW, FEW, EPI>::NT, RowTile<L, NARROW, FEW, EPI>::min_blocks(sizeof(T)))
    k_rows_line(RowArgs<T> a, const typename A::W* __restrict__ tw) {
  using Tile = RowTile<L, NARROW, FEW, EPI>;
  using Ln = Line<A, L, NARROW>;
  typename A::W pre[Ln::NTW + 1];
  if (Tile::NFFT == Tile::NT || threadIdx.x < Tile::NFFT) Ln::preload(pre, threadIdx.x % Tile::TS, tw);
  chain_enter(sizeof(T) == 4);
  using V = typename A::V;
  using C = cx<T>;
  constexpr int E = Ln::E, TS = Tile::TS, RS = Tile::RS, NF = Tile::NF, M = L / 2;
  __shared__ __align__(16) V buf[Tile::NSEQ * RS];
  const long row0 = (long)(a.rev ? gridDim.x - 1 - blockIdx.x : blockIdx.x) * Tile::ROWS;
  if (Tile::NFFT == Tile::NT || threadIdx.x < Tile::NFFT) {
    const int seq = threadIdx.x / TS, j = threadIdx.x % TS;
    const long row = row0 + seq / NF * 2;
    const bool ok = row < a.nrows;
    V* b = buf + seq * RS;
    C x[E];
    {
      const T* u = a.u[0];
      if (NF == 2 && seq % NF) u = a.u[1];
      u += row * L;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int p = Ln::position(j, e);
        x[e] = ok ? mk<C>(u[p], u[L + p]) : mk<C>(0, 0);
      }
      if constexpr (EPI == EPI_DIV) {
        const T* m = a.mul + row * L;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const int p = Ln::position(j, e);
          if (ok) x[e] = mk<C>(x[e].x * m[p], x[e].y * m[L + p]);
        }
      }
    }
    V v[E];
    const RowSync<TS, Tile::NFFT> sync;
    auto at = [&](int p) { return b + p + (p >> Tile::PADSH); };
    if constexpr (A::SCALED) {
      unsigned mx = 0, my = 0;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        mx = max(mx, fx_mag(x[e].x));
        my = max(my, fx_mag(x[e].y));
      }
      row_max<TS>(mx, my, reinterpret_cast<unsigned*>(b), j, sync);
      const FxScale<L, Ln::R0> sx(mx), sy(my);
      sx.in(sy, x, v);
      Ln::derivative(v, j, at, sync, tw, pre);
      sx.template out<true>(sy, v, x);
      sx.keep_zero(sy, x);
    } else {
      float mx = 0.f, my = 0.f;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        mx = fmaxf(mx, fabsf(x[e].x));
        my = fmaxf(my, fabsf(x[e].y));
      }
      unsigned bx = __float_as_uint(mx), by = __float_as_uint(my);
      row_max<TS>(bx, by, reinterpret_cast<unsigned*>(b), j, sync);
      bx = row_binade(bx);
      by = row_binade(by);
      const float2 to_one = make_float2(__uint_as_float(0x7f000000u - bx), __uint_as_float(0x7f000000u - by));
      const float2 back = make_float2(__uint_as_float(bx), -__uint_as_float(by));  // of the conjugate
#pragma unroll
      for (int e = 0; e < E; ++e) v[e] = A::in(__fmul2_rn(x[e], to_one));
      Ln::derivative(v, j, at, sync, tw, pre);
#pragma unroll
      for (int e = 0; e < E; ++e) x[e] = __fmul2_rn(v[e], back);
    }
    // the two real rows of the derivative, in place of the exchanged values
    if constexpr (Ln::S > 1) sync();
    T* ra = reinterpret_cast<T*>(b);
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int p = Ln::position(j, e);
      ra[p] = x[e].x;
      ra[RS + p] = x[e].y;
    }
  }
  if constexpr (Tile::WARP) __syncwarp();
  else __syncthreads();
  constexpr int GT = Tile::WARP ? 32 : Tile::NT;                      // threads that share rows
  constexpr int GROWS = Tile::WARP ? 32 / TS / NF * 2 : Tile::ROWS;  // and those rows
  const int g0 = Tile::WARP ? (int)(threadIdx.x / 32) * GROWS : 0;
  const int gt = Tile::WARP ? threadIdx.x % 32 : threadIdx.x;
#pragma unroll 2
  for (int i = gt; i < GROWS * M; i += GT) {
    const int r = g0 + i / M, jj = i % M;
    const long row = row0 + r;
    if (row >= a.nrows) break;
    const long q = row * M + jj;  // the point pair (2 jj, 2 jj + 1) of the row
    auto dlast = [&](int f) {
      const T* ra = reinterpret_cast<const T*>(buf + (r / 2 * NF + f) * RS) + (r & 1) * RS;
      return reinterpret_cast<const C*>(ra)[jj];
    };
    auto ld = [&](const T* p) { return reinterpret_cast<const C*>(p)[q]; };
    auto lds = [&](const T* p) { return ld_stream(reinterpret_cast<const C*>(p) + q); };
    if constexpr (EPI == EPI_ADV2) {
      const C g[2] = {lds(a.gx[0]), dlast(0)};
      adv_point<T, 2>(a.adv, g, q, nullptr);
    } else if constexpr (EPI == EPI_ADV3) {
      const C g[3] = {lds(a.gx[0]), ld(a.gy[0]), dlast(0)};
      adv_point<T, 3>(a.adv, g, q, nullptr);
    } else if constexpr (EPI == EPI_ADV33) {
      const C g[3] = {lds(a.gx[0]), ld(a.gy[0]), dlast(0)};
      const C h[3] = {lds(a.gx[1]), ld(a.gy[1]), dlast(1)};
      C av[3];
      const C sa = adv_point<T, 3>(a.adv, g, q, nullptr, nullptr, av);
      adv_point<T, 3>(a.advB, h, q, a.advB.src_from_a ? &sa : nullptr, a.advB.a_from_a ? av : nullptr);
    } else {
      C k = dlast(0);
      const C x = lds(a.gx[0]);
      k = mk<C>(k.x + x.x, k.y + x.y);
      if (a.gy[0]) {
        const C y = ld(a.gy[0]);
        k = mk<C>(k.x + y.x, k.y + y.y);
      }
      div_point<T>(a.dv, k, q);
    }
  }
}

}  // namespace fused
}  // namespace reg
