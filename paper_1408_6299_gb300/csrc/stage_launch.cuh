// stage_launch.cuh -- host launchers of the transport stages (stage.cuh),
// instantiated per precision by the stage_*.cu files.
#pragma once
#include <type_traits>

#include "stage.cuh"
#include "tune.h"

namespace reg {
namespace fused {

// line arithmetic per precision
template <typename T>
struct Arith;
template <>
struct Arith<float> {
  using Main = LineFloat<float>;
};
template <>
struct Arith<double> {
  using Main = LineFixed;
};

// One derivative pass along a strided axis: out = D_axis in, or D_axis (in mul)
template <typename T>
struct ColJob {
  int axis;
  const T* in;
  const T* mul;
  T* out;
};

// distance of two elements of a line along `axis` (complex values: pairs of reals)
inline long line_stride(const Grid& g, int axis) {
  long s = g.M;
  for (int a = axis + 1; a < g.d - 1; ++a) s *= g.n[a];
  return s;
}

template <class A, typename T, int L, bool NARROW, bool PROD, int VAR>
void cols_launch(const Spectral<T>& sp, const ColJob<T>* jobs, int nj, cudaStream_t st) {
  using Tile = ColTile<A, L, NARROW, VAR>;
  const Grid& g = sp.grid();
  ColJobs<T> J{};
  J.nj = nj;
  J.n = (int)(g.Nc / L / A::CW);
  const int per = (J.n + Tile::TC - 1) / Tile::TC;
  for (int q = 0; q < nj; ++q) {
    J.in[q] = jobs[q].in;
    J.mul[q] = jobs[q].mul;
    J.out[q] = jobs[q].out;
    J.stream[q] = jobs[q].axis == 0;
    J.log2s[q] = ilog2_c((int)(line_stride(g, jobs[q].axis) / A::CW));
    J.start[q] = q * per;
  }
  J.start[nj] = nj * per;
  ProfScope ps(KK_COLS, st, (double)nj * g.N * sizeof(T) * (PROD ? 3.0 : 2.0),
               (double)nj * g.Nc / L * (2.0 * fft_flops<L>() + 2.0 * L));
  chain(k_cols_line<A, T, L, NARROW, PROD, VAR>, (unsigned)(nj * per), Tile::NT, st, J,
        static_cast<const typename A::W*>(sp.line_table(L, NARROW, A::TABLE)));
}

// Fields up to 16 MB live in L2 between the passes, as in the trials, and the
// double-precision passes are bound by arithmetic; larger single-precision
// fields stream, which a trial on the same buffers does not show: variant 0.
template <class A, typename T, int L, bool NARROW, bool PROD>
void cols_tuned(const Spectral<T>& sp, const ColJob<T>* jobs, int nj, cudaStream_t st) {
  auto run = [&](int v) {
    if (v == 0) cols_launch<A, T, L, NARROW, PROD, 0>(sp, jobs, nj, st);
    else cols_launch<A, T, L, NARROW, PROD, 1>(sp, jobs, nj, st);
  };
  const long n = sp.grid().N;
  if (sizeof(T) == 4 && n * (long)sizeof(T) > (16 << 20)) return run(0);
  const char* kind = NARROW ? (PROD ? "cols|prod|narrow" : "cols|plain|narrow")
                            : A::CW == 2 ? (PROD ? "cols|prod|pair" : "cols|plain|pair")
                                         : (PROD ? "cols|prod|wide" : "cols|plain|wide");
  run(tuned_choice(kind, sizeof(T), L, tune_size(n * nj), 2, st, run));
}

template <typename T, int L, bool PROD>
void cols_L(const Spectral<T>& sp, const ColJob<T>* jobs, int nj, cudaStream_t st) {
  using A = typename Arith<T>::Main;
  const Grid& g = sp.grid();
  const long threads = plan_lines(g, (long)nj * g.Nc / L, sizeof(T)) * LinePlan<L, false>::TS;
  if (narrow_lines(threads, sizeof(T))) return cols_tuned<A, T, L, true, PROD>(sp, jobs, nj, st);
  if constexpr (sizeof(T) == 4)
    if (threads >= 2 * kSMs * 512) return cols_tuned<LinePair, T, L, false, PROD>(sp, jobs, nj, st);
  cols_tuned<A, T, L, false, PROD>(sp, jobs, nj, st);
}

// Whether jobs along axes of two lengths share a launch: where both run narrow
// plans, and in double precision only while every block has an SM to itself,
// since k_cols_two holds the registers of its longest line and does not tune its
// tile (32 x 16 x 8 mixed matvec 287 -> 254 us, 32 x 64 x 128 mixed Newton matvec
// 2506 -> 2422, 64 x 16 x 8 FP64 matvec 967 -> 871; beyond the limit 64 x 128 x
// 16 FP64 transport 1056 -> 1132, 256 x 32 x 64 FP64 matvec 40.8 -> 44.5 ms).
template <typename T>
bool one_cols_launch(const Grid& g, int nj) {
  for (int a = 0; a < 2; ++a) {
    const int L = (int)g.n[a];
    if (L > 256) return false;
    if (!narrow_lines(plan_lines(g, (long)(nj / 2) * g.Nc / L, sizeof(T)) * wide_threads(L), sizeof(T))) return false;
  }
  return sizeof(T) == 4 || nj * g.Nc / 4 <= (long)kSMs * kTwoNT;
}

// jobs along both strided axes, of two lengths, in one launch of narrow plans
template <typename T, bool PROD>
void cols_two(const Spectral<T>& sp, const ColJob<T>* jobs, int nj, cudaStream_t st) {
  using A = typename Arith<T>::Main;
  const Grid& g = sp.grid();
  ColJobs<T> J{};
  TwoAxes<A> P{};
  J.nj = nj;
  double flops = 0;
  for (int a = 0; a < 2; ++a) {
    P.tw[a] = static_cast<const typename A::W*>(sp.line_table((int)g.n[a], true, A::TABLE));
    P.lg[a] = ilog2_c((int)g.n[a]);
    P.n[a] = (int)(g.Nc / g.n[a] / A::CW);
  }
  for (int q = 0; q < nj; ++q) {
    const int a = jobs[q].axis, tc = kTwoNT * 4 / (int)g.n[a];
    J.in[q] = jobs[q].in;
    J.mul[q] = jobs[q].mul;
    J.out[q] = jobs[q].out;
    J.log2s[q] = ilog2_c((int)(line_stride(g, a) / A::CW));
    J.start[q + 1] = J.start[q] + (P.n[a] + tc - 1) / tc;
    P.axis[q] = a;
    flops += (double)g.Nc / g.n[a] * (10.0 * g.n[a] * P.lg[a] + 2.0 * g.n[a]);
  }
  ProfScope ps(KK_COLS, st, (double)nj * g.N * sizeof(T) * (PROD ? 3.0 : 2.0), flops);
  chain(k_cols_two<A, T, PROD>, (unsigned)J.start[nj], kTwoNT, st, J, P);
}

// The column passes of one stage. Axes of two lengths: one launch
// (one_cols_launch) or one launch per length, side by side (each fills the
// other's last wave; 32 x 64 x 128 Newton matvec 3140 -> 2800 us).
template <typename T, bool PROD>
void run_cols(Spectral<T>& sp, const ColJob<T>* jobs, int nj, cudaStream_t st) {
  const Grid& g = sp.grid();
  const bool two = nj > 1 && g.n[0] != g.n[1];
  if (two && one_cols_launch<T>(g, nj)) return cols_two<T, PROD>(sp, jobs, nj, st);
  cudaStream_t st2 = two ? sp.fork() : st;
  for (int axis = 0; axis < (two ? 2 : 1); ++axis) {
    ColJob<T> grp[kColJobs];
    int m = 0;
    for (int q = 0; q < nj; ++q)
      if (!two || jobs[q].axis == axis) grp[m++] = jobs[q];
    if (two) tl_plain_launch = true;
    cudaStream_t s = axis ? st2 : st;
    switch (g.n[axis]) {
      case 8: cols_L<T, 8, PROD>(sp, grp, m, s); break;
      case 16: cols_L<T, 16, PROD>(sp, grp, m, s); break;
      case 32: cols_L<T, 32, PROD>(sp, grp, m, s); break;
      case 64: cols_L<T, 64, PROD>(sp, grp, m, s); break;
      case 128: cols_L<T, 128, PROD>(sp, grp, m, s); break;
      case 256: cols_L<T, 256, PROD>(sp, grp, m, s); break;
      case 512: cols_L<T, 512, PROD>(sp, grp, m, s); break;
      default: throw StatusError{1, "unsupported axis length"};
    }
  }
  if (two) {
    sp.join();
    tl_plain_launch = true;
  }
}

template <typename T, int L, int EPI>
void rows_L(const Spectral<T>& sp, const RowArgs<T>& a, double bytes, cudaStream_t st) {
  using A = typename Arith<T>::Main;
  constexpr int NF = RowTile<L, false, false, EPI>::NF;
  ProfScope ps(KK_ROWS_C2R, st, bytes, (double)a.nrows / 2 * NF * (2.0 * fft_flops<L>() + 2.0 * L));
  auto go = [&](auto narrow, auto few) {
    constexpr bool NARROW = decltype(narrow)::value, FEW = decltype(few)::value;
    using Tile = RowTile<L, NARROW, FEW, EPI>;
    // large fields from the last row on: the column pass left its last planes in
    // L2 (256^3 mixed matvec 158.7 -> 156.3 ms)
    RowArgs<T> b = a;
    b.rev = a.nrows * (long)L * sizeof(T) >= (64 << 20);
    chain(k_rows_line<A, T, L, NARROW, FEW, EPI>, (unsigned)((a.nrows + Tile::ROWS - 1) / Tile::ROWS), Tile::NT, st, b,
          static_cast<const typename A::W*>(sp.line_table(L, NARROW, A::TABLE)));
  };
  const long lines = a.nrows / 2 * NF;
  // few lines, against full blocks at any size, all else equal: 32^2 FP64 matvec 529
  // us (708 full), 128^2 mixed 613 (817), 64^3 mixed 1426 (1627). Double precision,
  // bound by arithmetic, loses earlier: 64^3 gradient (2048 lines) 3940 us (3790)
  const long few = (long)kSMs * (sizeof(T) == 8 ? 8 : 24);
  if (!narrow_lines(plan_lines(sp.grid(), lines, sizeof(T)) * LinePlan<L, false>::TS, sizeof(T))) go(std::false_type{}, std::false_type{});
  else if (lines <= few) go(std::true_type{}, std::true_type{});
  else go(std::true_type{}, std::false_type{});
}

template <typename T, int EPI>
void run_rows(const Spectral<T>& sp, const RowArgs<T>& a, double bytes, cudaStream_t st) {
  switch (sp.grid().L) {
    case 8: return rows_L<T, 8, EPI>(sp, a, bytes, st);
    case 16: return rows_L<T, 16, EPI>(sp, a, bytes, st);
    case 32: return rows_L<T, 32, EPI>(sp, a, bytes, st);
    case 64: return rows_L<T, 64, EPI>(sp, a, bytes, st);
    case 128: return rows_L<T, 128, EPI>(sp, a, bytes, st);
    case 256: return rows_L<T, 256, EPI>(sp, a, bytes, st);
    case 512: return rows_L<T, 512, EPI>(sp, a, bytes, st);
  }
  throw StatusError{1, "unsupported last-axis length"};
}

// Instantiated once per precision and pass (stage_cols_*.cu, stage_rows_*.cu),
// which compile side by side: one file per precision took 105 s.
#define REG_COLS_OF(T)                                                                         \
  template void run_cols<T, false>(Spectral<T>&, const ColJob<T>*, int, cudaStream_t);         \
  template void run_cols<T, true>(Spectral<T>&, const ColJob<T>*, int, cudaStream_t);
#define REG_ROWS_OF(T, EPI) template void run_rows<T, EPI>(const Spectral<T>&, const RowArgs<T>&, double, cudaStream_t);
#define REG_STAGES_OF(T)                                                                       \
  extern template void run_cols<T, false>(Spectral<T>&, const ColJob<T>*, int, cudaStream_t);  \
  extern template void run_cols<T, true>(Spectral<T>&, const ColJob<T>*, int, cudaStream_t);   \
  extern REG_ROWS_OF(T, EPI_ADV2) extern REG_ROWS_OF(T, EPI_ADV3)                              \
  extern REG_ROWS_OF(T, EPI_ADV33) extern REG_ROWS_OF(T, EPI_DIV)
REG_STAGES_OF(float)
REG_STAGES_OF(double)
#undef REG_STAGES_OF

// fields an advection epilogue reads and writes beyond u and its derivatives
// (stage 1 reads y = u itself)
template <typename T>
int adv_fields(const AdvEpi<T>& e, int d, const T* u) {
  int n = (e.G[0] ? d : 0) + (e.Sout ? d + 1 : 0);
  if (e.out1)
    n += d + (e.src ? 1 : (e.gm[0] && !e.src_from_a ? 2 * d : 0)) + (e.y && e.y != u ? 1 : 0) + 1;
  return n;
}

// One advection stage on u; gx, gy: scratch fields (gy in 3D).
template <typename T>
void adv_stage_impl(Spectral<T>& sp, const T* u, const AdvEpi<T>& e, T* gx, T* gy) {
  const Grid& g = sp.grid();
  cudaStream_t s = sp.stream();
  const ColJob<T> jobs[2] = {{0, u, nullptr, gx}, {1, u, nullptr, gy}};
  run_cols<T, false>(sp, jobs, g.d - 1, s);
  RowArgs<T> a{};
  a.u[0] = u;
  a.gx[0] = gx;
  a.gy[0] = g.d == 3 ? gy : nullptr;
  a.adv = e;
  a.nrows = g.rows;
  const double bytes = (double)g.N * sizeof(T) * (g.d + adv_fields(e, g.d, u));
  if (g.d == 3) run_rows<T, EPI_ADV3>(sp, a, bytes, s);
  else run_rows<T, EPI_ADV2>(sp, a, bytes, s);
}

// Two advection stages of 3D fields uA and uB sharing their launches; Z: four
// scratch fields.
template <typename T>
void adv2_stage_impl(Spectral<T>& sp, const T* uA, const AdvEpi<T>& eA, const T* uB, const AdvEpi<T>& eB,
                     T* const* Z) {
  const Grid& g = sp.grid();
  cudaStream_t s = sp.stream();
  const ColJob<T> jobs[4] = {
      {0, uA, nullptr, Z[0]}, {1, uA, nullptr, Z[1]}, {0, uB, nullptr, Z[2]}, {1, uB, nullptr, Z[3]}};
  run_cols<T, false>(sp, jobs, 4, s);
  RowArgs<T> a{};
  a.u[0] = uA;
  a.u[1] = uB;
  for (int f = 0; f < 2; ++f) {
    a.gx[f] = Z[2 * f];
    a.gy[f] = Z[2 * f + 1];
  }
  a.adv = eA;
  a.advB = eB;
  // a velocity read by both epilogues (the same node, or n_c = 1) is read once
  const bool shared_a = eA.out1 && eB.out1 && eA.a[0] == eB.a[0] && eA.a[1] == eB.a[1] && eA.a[2] == eB.a[2];
  a.advB.a_from_a = shared_a ? 1 : 0;
  a.nrows = g.rows;
  const double bytes =
      (double)g.N * sizeof(T) * (6 + adv_fields(eA, 3, uA) + adv_fields(eB, 3, uB) - (shared_a ? 3 : 0));
  run_rows<T, EPI_ADV33>(sp, a, bytes, s);
}

// One divergence stage: div(a lam); kx, ky: scratch fields (ky in 3D).
template <typename T>
void div_stage_impl(Spectral<T>& sp, const T* lam, const T* a, const DivEpi<T>& e, T* kx, T* ky) {
  const Grid& g = sp.grid();
  cudaStream_t s = sp.stream();
  const long N = g.N;
  const ColJob<T> jobs[2] = {{0, a, lam, kx}, {1, a + N, lam, ky}};
  run_cols<T, true>(sp, jobs, g.d - 1, s);
  RowArgs<T> r{};
  r.u[0] = a + (g.d - 1) * N;
  r.mul = lam;
  r.gx[0] = kx;
  r.gy[0] = g.d == 3 ? ky : nullptr;
  r.dv = e;
  r.nrows = g.rows;
  const double f = 2 + g.d - 1 + (e.stage && e.y != lam ? 1 : 0) + 1 + (e.src ? 1 : 0);
  run_rows<T, EPI_DIV>(sp, r, f * N * sizeof(T), s);
}

}  // namespace fused
}  // namespace reg
