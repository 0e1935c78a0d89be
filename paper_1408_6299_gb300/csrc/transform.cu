// transform.cu -- kernels and launchers of the whole-field transforms (transform.cuh).
#include <type_traits>

#include "transform.cuh"
#include "tune.h"

namespace reg {
namespace {

// Lines of a block of a row transform (VAR 1: half of them).
template <int L, bool NARROW, int VAR>
struct FieldRows {
  using P = LinePlan<L, NARROW>;
  static constexpr int TS = P::TS;
  static constexpr int NSEQ0 = NARROW ? (32 / TS > 1 ? 32 / TS : 1) * 2 : 128 / TS;
  static constexpr int NSEQ = VAR ? NSEQ0 / 2 : NSEQ0;
  static constexpr int NT = NSEQ * TS;
  static constexpr int PADSH = P::R(0) == 16 ? 4 : (P::R(0) == 8 ? 3 : 2);
  static constexpr int RS = L + (L >> PADSH);
};

// Real rows to packed half spectra (unnormalised).
template <int L, bool NARROW, int VAR>
__global__ void __launch_bounds__(FieldRows<L, NARROW, VAR>::NT) k_field_rows_fwd(const double* __restrict__ in,
                                                                                   double2* __restrict__ out,
                                                                                   long nrows,
                                                                                   const int4* __restrict__ tw) {
  chain_enter();
  using F = FieldRows<L, NARROW, VAR>;
  using Ln = Line<LineFixed, L, NARROW>;
  constexpr int E = Ln::E, TS = F::TS, M = L / 2;
  __shared__ FxV buf[F::NSEQ * F::RS];
  const int seq = threadIdx.x / TS, j = threadIdx.x % TS;
  const long row = ((long)blockIdx.x * F::NSEQ + seq) * 2;
  const bool ok = row < nrows;
  FxV* b = buf + seq * F::RS;
  const double* u = in + row * L;
  double2 x[E];
  unsigned mag = 0;
  float l1 = 0.f;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int p = Ln::position(j, e);
    x[e] = ok ? make_double2(u[p], u[L + p]) : make_double2(0, 0);
    mag = max(mag, fx_mag(x[e]));
    l1 += fx_l1(x[e]);
  }
  const RowSync<TS, F::NT> sync;
  row_max_sum<TS>(mag, l1, reinterpret_cast<unsigned*>(b), j, sync);
  FxScale<L, Ln::R0> sc(mag);
  sc.by_sum(mag, l1);
  sc.times_pow2(-1);
  FxV v[E];
  sc.in(x, v);
  auto at = [&](int p) { return b + p + (p >> F::PADSH); };
  Ln::forward(v, j, at, sync, tw, sc.scaled);
  if constexpr (Ln::S > 1) sync();
#pragma unroll
  for (int e = 0; e < E; ++e) *at(Ln::frequency(j, e)) = v[e];
  sync();
  if (!ok) return;
  double2* o = out + row * M;
  for (int k = j; k < M; k += TS) {
    const FxV z = *at(k), w = *at(k == 0 ? M : L - k);
    FxV a, c;
    if (k == 0) {
      a = {2 * z.x, 2 * w.x};
      c = {2 * z.y, 2 * w.y};
    } else {
      a = {z.x + w.x, z.y - w.y};
      c = {z.y + w.y, w.x - z.x};
    }
    o[k] = make_double2(sc.back(a.x), sc.back(a.y));
    o[M + k] = make_double2(sc.back(c.x), sc.back(c.y));
  }
}

// Packed half spectra to real rows, normalised by 1/L.
template <int L, bool NARROW>
__global__ void __launch_bounds__(FieldRows<L, NARROW, 0>::NT) k_field_rows_inv(const double2* __restrict__ in,
                                                                                 double* __restrict__ out, long nrows,
                                                                                 const int4* __restrict__ tw) {
  chain_enter();
  using F = FieldRows<L, NARROW, 0>;
  using Ln = Line<LineFixed, L, NARROW>;
  constexpr int E = Ln::E, TS = F::TS, M = L / 2;
  __shared__ FxV buf[F::NSEQ * F::RS];
  const int seq = threadIdx.x / TS, j = threadIdx.x % TS;
  const long row = ((long)blockIdx.x * F::NSEQ + seq) * 2;
  const bool ok = row < nrows;
  FxV* b = buf + seq * F::RS;
  const double2* ra = in + row * M;
  double2 x[E];  // conj(Z_p), Z_p = A_p + i B_p, with A_{L-k} = conj A_k
  unsigned mag = 0;
  float l1 = 0.f;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int p = Ln::position(j, e);
    const int k = p < M ? p : (p == M ? 0 : L - p);
    const double2 A = ok ? ra[k] : make_double2(0, 0), B = ok ? ra[M + k] : make_double2(0, 0);
    if (p == 0) x[e] = make_double2(A.x, -B.x);
    else if (p == M) x[e] = make_double2(A.y, -B.y);
    else if (p < M) x[e] = make_double2(A.x - B.y, -(A.y + B.x));
    else x[e] = make_double2(A.x + B.y, A.y - B.x);
    mag = max(mag, fx_mag(x[e]));
    l1 += fx_l1(x[e]);
  }
  const RowSync<TS, F::NT> sync;
  row_max_sum<TS>(mag, l1, reinterpret_cast<unsigned*>(b), j, sync);
  FxScale<L, Ln::R0> sc(mag);
  sc.by_sum(mag, l1);
  sc.times_pow2(-ilog2_c(L));
  FxV v[E];
  sc.in(x, v);
  Ln::forward(v, j, [&](int p) { return b + p + (p >> F::PADSH); }, sync, tw, sc.scaled);
  if (!ok) return;
  double* o = out + row * L;
  sc.template out<true>(v, x);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int p = Ln::frequency(j, e);
    o[p] = x[e].x;
    o[L + p] = x[e].y;
  }
}

// Complex lines along a strided axis, in place; inverse: normalised by 1/L.
template <int L, bool NARROW>
struct FieldCols {
  static constexpr int TS = LinePlan<L, NARROW>::TS;
  static constexpr int TC1 = (NARROW ? 64 : 128) / TS < (NARROW ? 4 : 8) ? (NARROW ? 4 : 8) : (NARROW ? 64 : 128) / TS;
  static constexpr int fit(int tc) { return tc * L * 16 <= 49152 ? tc : fit(tc / 2); }
  static constexpr int TC = fit(TC1);
  static constexpr int NT = TC * TS;
};
template <int L, bool NARROW, bool INV>
__global__ void __launch_bounds__(FieldCols<L, NARROW>::NT) k_field_cols(double2* __restrict__ data, int ls, long n,
                                                                          const int4* __restrict__ tw) {
  chain_enter();
  using F = FieldCols<L, NARROW>;
  using Ln = Line<LineFixed, L, NARROW>;
  constexpr int E = Ln::E, TC = F::TC;
  __shared__ FxV buf[L * TC];
  const int c = threadIdx.x % TC, j = threadIdx.x / TC;
  const long line = (long)blockIdx.x * TC + c;
  const long s = 1L << ls;
  double2* d = data + (((line >> ls) * L) << ls) + (line & (s - 1));
  const bool ok = line < n;
  double2 x[E];
  unsigned mag = 0;
  float l1 = 0.f;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    x[e] = ok ? d[Ln::position(j, e) * s] : make_double2(0, 0);
    if (INV) x[e].y = -x[e].y;
    mag = max(mag, fx_mag(x[e]));
    l1 += fx_l1(x[e]);
  }
  line_max_sum<TC, F::TS>(mag, l1, reinterpret_cast<unsigned*>(buf), c, j);
  FxScale<L, Ln::R0> sc(mag);
  sc.by_sum(mag, l1);
  if (INV) sc.times_pow2(-ilog2_c(L));
  FxV v[E];
  sc.in(x, v);
  Ln::forward(v, j, [&](int p) { return buf + p * TC + c; }, [] { __syncthreads(); }, tw, sc.scaled);
  if (!ok) return;
  sc.template out<false>(v, x);  // conjugated
#pragma unroll
  for (int e = 0; e < E; ++e) d[Ln::frequency(j, e) * s] = INV ? x[e] : make_double2(x[e].x, -x[e].y);
}

template <class F>
void by_length(int L, F f) {
  switch (L) {
    case 8: return f(std::integral_constant<int, 8>{});
    case 16: return f(std::integral_constant<int, 16>{});
    case 32: return f(std::integral_constant<int, 32>{});
    case 64: return f(std::integral_constant<int, 64>{});
    case 128: return f(std::integral_constant<int, 128>{});
    case 256: return f(std::integral_constant<int, 256>{});
    case 512: return f(std::integral_constant<int, 512>{});
  }
  throw StatusError{1, "unsupported FFT length " + std::to_string(L)};
}
template <class F>
void by_plan(bool narrow, F f) {
  if (narrow) f(std::true_type{});
  else f(std::false_type{});
}

}  // namespace

FieldTransforms::FieldTransforms(const Grid& g, cudaStream_t s, TableFn tables, bool tuned)
    : g_(g), s_(s), tables_(std::move(tables)), tuned_(tuned) {}

bool FieldTransforms::narrow(int L, long lines) const {
  return tuned_ && narrow_lines(plan_lines(g_, lines, sizeof(double)) * wide_threads(L), sizeof(double));
}

void FieldTransforms::cols(double2* U, int axis, int nf, bool inverse) const {
  long s = g_.M;
  for (int a = axis + 1; a < g_.d - 1; ++a) s *= g_.n[a];
  by_length(g_.n[axis], [&](auto len) {
    constexpr int L = decltype(len)::value;
    const long n = nf * g_.Nc / L;
    ProfScope ps(KK_COLS, s_, 2.0 * n * L * sizeof(double2), (double)n * fft_flops<L>());
    by_plan(narrow(L, n), [&](auto nw) {
      constexpr bool NW = decltype(nw)::value;
      using F = FieldCols<L, NW>;
      const int4* tw = static_cast<const int4*>(tables_(L, NW));
      const unsigned grid = (unsigned)((n + F::TC - 1) / F::TC);
      chain(inverse ? k_field_cols<L, NW, true> : k_field_cols<L, NW, false>, grid, F::NT, s_, U, ilog2_c((int)s), n,
            tw);
    });
  });
}

void FieldTransforms::fwd(const double* u, double2* U, int nf) const {
  by_length(g_.L, [&](auto len) {
    constexpr int L = decltype(len)::value;
    const long rows = nf * g_.rows;
    ProfScope ps(KK_ROWS_R2C, s_, 2.0 * rows * L * sizeof(double), (double)rows / 2 * (fft_flops<L>() + 4.0 * L));
    by_plan(narrow(L, rows / 2), [&](auto nw) {
      constexpr bool NW = decltype(nw)::value;
      const int4* tw = static_cast<const int4*>(tables_(L, NW));
      auto run = [&](int var) {
        using F0 = FieldRows<L, NW, 0>;
        using F1 = FieldRows<L, NW, 1>;
        const long lines = rows / 2;
        if (var == 0)
          chain(k_field_rows_fwd<L, NW, 0>, (unsigned)((lines + F0::NSEQ - 1) / F0::NSEQ), F0::NT, s_, u, U, rows, tw);
        else
          chain(k_field_rows_fwd<L, NW, 1>, (unsigned)((lines + F1::NSEQ - 1) / F1::NSEQ), F1::NT, s_, u, U, rows, tw);
      };
      run(tuned_ ? tuned_choice(NW ? "rows_r2c|narrow" : "rows_r2c|wide", sizeof(double), L, tune_size(rows), 2, s_, run) : 0);
    });
  });
  for (int a = g_.d - 2; a >= 0; --a) cols(U, a, nf, false);
}

void FieldTransforms::inv(double2* U, double* u, int nf) const {
  for (int a = 0; a <= g_.d - 2; ++a) cols(U, a, nf, true);
  by_length(g_.L, [&](auto len) {
    constexpr int L = decltype(len)::value;
    const long rows = nf * g_.rows;
    ProfScope ps(KK_ROWS_C2R, s_, 2.0 * rows * L * sizeof(double), (double)rows / 2 * (fft_flops<L>() + 4.0 * L));
    by_plan(narrow(L, rows / 2), [&](auto nw) {
      constexpr bool NW = decltype(nw)::value;
      using F = FieldRows<L, NW, 0>;
      chain(k_field_rows_inv<L, NW>, (unsigned)((rows / 2 + F::NSEQ - 1) / F::NSEQ), F::NT, s_, U, u, rows,
            static_cast<const int4*>(tables_(L, NW)));
    });
  });
}

}  // namespace reg
