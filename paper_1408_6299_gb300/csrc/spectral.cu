// spectral.cu -- Fourier multipliers of the pseudospectral discretisation
// (Mang & Biros, Sec. 3.3.3 the spectral inverse of beta*A; Sec. 3.3.4 / App. B
// the Leray projection K), on packed half spectra, and the launch accounting.
//
// The packed layout stores the DC and Nyquist columns of the last axis
// together in slot 0 (see Grid in internal.h); Leray multipliers treat both
// halves alike (their last-axis wavenumber is 0 for both), while multipliers
// depending on |k| (A and its inverse) pair the mode k' with -k' to act on the
// two halves separately.
//
// The kernels are bound by memory only if they stay off the double-precision
// unit (two operations per clock and SM): wavenumbers and |k|^2 are integers,
// and the reciprocals of |k|^2 (one of sum (n_a/2)^2 values) come from a table.
#include <math.h>

#include <algorithm>
#include <atomic>
#include <stdexcept>
#include <type_traits>

#include "internal.h"

namespace reg {

namespace {

__host__ __device__ inline int kfull(int j, int n) { return j < n / 2 ? j : j - n; }
__host__ __device__ inline int kmask(int j, int n) { return j == n / 2 ? 0 : kfull(j, n); }

// mode index q of the packed spectrum -> per-axis indices (last = slot)
struct ModeIdx {
  int j[3];
};
struct GridArgs {
  int d;
  int n[3];
  int M;
  long Nc;   // all stacked problems
  long Nc1;  // one problem (a power of two)
  int lg1;   // log2 Nc1
  int lg[3];  // log2 n, of the last axis log2 M
};
// D: the dimension where it is a constant (indices then stay in registers), or 0
template <int D = 0>
__device__ inline ModeIdx decode(long q, const GridArgs& g) {
  const int d = D ? D : g.d;
  ModeIdx m;
  int r = (int)(q & (g.Nc1 - 1));
#pragma unroll
  for (int a = d - 1; a >= 0; --a) {
    m.j[a] = r & ((1 << g.lg[a]) - 1);
    r >>= g.lg[a];
  }
  return m;
}
// index of -k' on the slot-0 plane of the problem that holds mode q0
template <int D = 0>
__device__ inline long encode_neg(long q0, const ModeIdx& m, const GridArgs& g) {
  int q = 0;
#pragma unroll
  for (int a = 0; a < (D ? D : g.d) - 1; ++a) q = q * g.n[a] + ((g.n[a] - m.j[a]) & (g.n[a] - 1));
  return (q0 & ~(g.Nc1 - 1)) + (long)q * g.M;
}
template <int D>
__device__ inline int masked_k(const ModeIdx& m, const GridArgs& g, int a) {
  if (a == D - 1) return m.j[a];  // slot 0 -> 0 for both DC and Nyquist halves
  return kmask(m.j[a], g.n[a]);
}
// |k|^2 over the leading axes (full wavenumbers, Nyquist kept)
template <int D = 0>
__device__ inline int lead_k2(const ModeIdx& m, const GridArgs& g) {
  int kk = 0;
#pragma unroll
  for (int a = 0; a < (D ? D : g.d) - 1; ++a) {
    const int k = kfull(m.j[a], g.n[a]);
    kk += k * k;
  }
  return kk;
}
// |k|^2 or |k|^4 (exact: |k|^2 <= 3 256^2)
__device__ inline double sym_pow(int kk, int reg) { return (double)(reg == 1 ? (long long)kk : (long long)kk * kk); }
// p / kk from the rounded reciprocal w = 1 / kk: the remainder corrects the product
__device__ inline double quotient(double p, double w, double kk) {
  const double q = p * w;
  return fma(w, fma(-q, kk, p), q);
}

constexpr int kMaxNc = 16;

// t[m] = 1 / (beta m^reg)
__global__ void k_inv_k2(double* t, long n, double beta, int reg) {
  const long m = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (m < n) t[m] = m ? 1.0 / (beta * sym_pow((int)m, reg)) : 0.0;
}

// NC: n_c where it is 1, 2 or 3 (the coefficients of a component then stay in
// registers), else 0. Bound by the double-precision unit, so products with one
// and sums with zero are left out for n_c = 1, and indices come from shifts with
// the dimension a constant (256^3: 472 -> 243 us, 177 at the copy rate).
template <int NC, int D>
__global__ void __launch_bounds__(256) k_spec_tail(const double2* __restrict__ V, const double2* __restrict__ F,
                                                   double2* __restrict__ out, GridArgs g, int nc_, double beta,
                                                   const double* __restrict__ Cg, int reg, int stokes,
                                                   const double* __restrict__ betas,
                                                   const double* __restrict__ inv_k2) {
  chain_enter();
  const long q = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= g.Nc) return;
  if (betas) beta = betas[q >> g.lg1];
  constexpr int d = D;
  const int nc = NC ? NC : nc_;
  const long Nc = g.Nc;
  const ModeIdx m = decode<D>(q, g);
  const int kk = lead_k2<D>(m, g), kz = m.j[d - 1];
  double alpha, delta = 0.0;
  long qn = q;
  if (kz == 0) {
    const double a0 = sym_pow(kk, reg), aN = sym_pow(kk + g.M * g.M, reg);
    alpha = 0.5 * beta * (a0 + aN);
    delta = 0.5 * beta * (a0 - aN);
    qn = encode_neg<D>(q, m, g);
  } else {
    alpha = beta * sym_pow(kk + kz * kz, reg);
  }
  // masked wavenumber for K
  int kt[d], kt2 = 0;
  if (F && stokes)
#pragma unroll
    for (int a = 0; a < d; ++a) {
      kt[a] = masked_k<D>(m, g, a);
      kt2 += kt[a] * kt[a];
    }
  auto reg_term = [&](int i, int l, const double2* v, const double2* vn) {
    double2 s = make_double2(0, 0), n = make_double2(0, 0);
    for (int lp = 0; lp < nc; ++lp) {
      const double c = __ldg(&Cg[l * nc + lp]);
      if (c == 0.0) continue;  // odd pairs of Chebyshev polynomials are orthogonal
      const double2 x = NC ? v[lp] : V[(lp * d + i) * Nc + q];
      s.x += c * x.x;
      s.y += c * x.y;
      if (kz == 0) {
        const double2 y = NC ? vn[lp] : V[(lp * d + i) * Nc + qn];
        n.x += c * y.x;
        n.y += c * y.y;
      }
    }
    double2 r = make_double2(alpha * s.x, alpha * s.y);
    if (kz == 0) r = make_double2(r.x + delta * n.x, r.y - delta * n.y);  // + delta conj(n)
    return r;
  };
  // k . f_l / |k|^2; out may be F, so it is formed before any component of f_l is overwritten
  const double wk = kt2 > 0 && F && stokes ? (inv_k2 ? __ldg(&inv_k2[kt2]) : 1.0 / (double)kt2) : 0.0;
  auto over_k2 = [&](double2 p) { return make_double2(quotient(p.x, wk, (double)kt2), quotient(p.y, wk, (double)kt2)); };
  auto projection = [&](int l) {
    double2 p = make_double2(0, 0);
    if (!(F && stokes && kt2 > 0)) return p;
    for (int a = 0; a < d; ++a) {
      const double2 fa = F[(l * d + a) * Nc + q];
      p.x += (double)kt[a] * fa.x;
      p.y += (double)kt[a] * fa.y;
    }
    return over_k2(p);
  };
  auto store = [&](int i, int l, double2 r, double2 p) {
    if (F) {
      const double2 f = F[(l * d + i) * Nc + q];
      r = make_double2(r.x + f.x, r.y + f.y);
      if (stokes && kt2 > 0) r = make_double2(r.x - (double)kt[i] * p.x, r.y - (double)kt[i] * p.y);
    }
    out[(l * d + i) * Nc + q] = r;
  };
  if constexpr (NC == 1) {
    // the 1 x 1 Gram matrix is 1; all loads of a mode first
    double2 v[d], f[d], vn[d];
#pragma unroll
    for (int i = 0; i < d; ++i) {
      v[i] = V[i * Nc + q];
      f[i] = F ? F[i * Nc + q] : make_double2(0, 0);
      if (kz == 0) vn[i] = V[i * Nc + qn];
    }
    double2 p = make_double2(0, 0);
    const bool leray = F && stokes && kt2 > 0;
    if (leray) {
#pragma unroll
      for (int a = 0; a < d; ++a) p = make_double2(p.x + (double)kt[a] * f[a].x, p.y + (double)kt[a] * f[a].y);
      p = over_k2(p);
    }
#pragma unroll
    for (int i = 0; i < d; ++i) {
      double2 r = make_double2(alpha * v[i].x, alpha * v[i].y);
      if (kz == 0) r = make_double2(r.x + delta * vn[i].x, r.y - delta * vn[i].y);
      if (F) r = make_double2(r.x + f[i].x, r.y + f[i].y);
      if (leray) r = make_double2(r.x - (double)kt[i] * p.x, r.y - (double)kt[i] * p.y);
      out[i * Nc + q] = r;
    }
  } else if constexpr (NC > 0) {
    double2 p[NC];
#pragma unroll
    for (int l = 0; l < NC; ++l) p[l] = projection(l);
    for (int i = 0; i < d; ++i) {
      double2 v[NC], vn[NC];
#pragma unroll
      for (int lp = 0; lp < NC; ++lp) {
        v[lp] = V[(lp * d + i) * Nc + q];
        vn[lp] = kz == 0 ? V[(lp * d + i) * Nc + qn] : make_double2(0, 0);
      }
#pragma unroll
      for (int l = 0; l < NC; ++l) store(i, l, reg_term(i, l, v, vn), p[l]);
    }
  } else {
    for (int l = 0; l < nc; ++l) {
      const double2 p = projection(l);
      for (int i = 0; i < d; ++i) store(i, l, reg_term(i, l, nullptr, nullptr), p);
    }
  }
}

// inv: 1 / (beta |k|^2) or 1 / (beta |k|^4) by |k|^2; null: divided per mode (with
// the changes named at k_spec_tail the 256^3 preconditioner 2085 -> 1883 us, of
// which this kernel 242; 118 at the copy rate)
template <int NC, int D>
__global__ void __launch_bounds__(256) k_spec_precond(const double2* __restrict__ R, double2* __restrict__ out,
                                                      GridArgs g, int nc_, double beta, const double* __restrict__ Ci,
                                                      int reg, const double* __restrict__ betas,
                                                      const double* __restrict__ inv) {
  chain_enter();
  const long q = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= g.Nc) return;
  if (betas) beta = betas[q >> g.lg1];
  constexpr int d = D;
  const int nc = NC ? NC : nc_;
  const long Nc = g.Nc;
  const ModeIdx m = decode<D>(q, g);
  const int kk = lead_k2<D>(m, g), kz = m.j[d - 1];
  double alpha, delta = 0.0;
  long qn = q;
  auto scale = [&](int k2) { return inv ? __ldg(&inv[k2]) : 1.0 / (beta * sym_pow(k2, reg)); };
  if (kz == 0) {
    const double s0 = kk == 0 ? 1.0 : scale(kk);  // k = 0: the inverse is replaced by one
    const double sN = scale(kk + g.M * g.M);
    alpha = 0.5 * (s0 + sN);
    delta = 0.5 * (s0 - sN);
    qn = encode_neg<D>(q, m, g);
  } else {
    alpha = scale(kk + kz * kz);
  }
  if constexpr (NC == 1) {  // the 1 x 1 Gram matrix is 1; all loads of a mode first
    double2 v[d], vn[d];
#pragma unroll
    for (int i = 0; i < d; ++i) {
      v[i] = R[i * Nc + q];
      if (kz == 0) vn[i] = R[i * Nc + qn];
    }
#pragma unroll
    for (int i = 0; i < d; ++i) {
      double2 r = make_double2(alpha * v[i].x, alpha * v[i].y);
      if (kz == 0) r = make_double2(r.x + delta * vn[i].x, r.y - delta * vn[i].y);
      out[i * Nc + q] = r;
    }
  } else {
    for (int i = 0; i < d; ++i) {
      double2 v[NC ? NC : 1], vn[NC ? NC : 1];
      if (NC) {
#pragma unroll
        for (int lp = 0; lp < NC; ++lp) {
          v[lp] = R[(lp * d + i) * Nc + q];
          if (kz == 0) vn[lp] = R[(lp * d + i) * Nc + qn];
        }
      }
#pragma unroll
      for (int l = 0; l < nc; ++l) {
        double2 s = make_double2(0, 0), n = make_double2(0, 0);
        for (int lp = 0; lp < nc; ++lp) {
          const double c = __ldg(&Ci[l * nc + lp]);
          const double2 x = NC ? v[NC ? lp : 0] : R[(lp * d + i) * Nc + q];
          s.x += c * x.x;
          s.y += c * x.y;
          if (kz == 0) {
            const double2 y = NC ? vn[NC ? lp : 0] : R[(lp * d + i) * Nc + qn];
            n.x += c * y.x;
            n.y += c * y.y;
          }
        }
        double2 r = make_double2(alpha * s.x, alpha * s.y);
        if (kz == 0) r = make_double2(r.x + delta * n.x, r.y - delta * n.y);
        out[(l * d + i) * Nc + q] = r;
      }
    }
  }
}

// Gaussian filter exp(-sigma^2 |k|^2 / 2) on one packed field (full
// wavenumbers, Nyquist kept; slot 0 of the last axis pairs k' with -k' as A does)
__global__ void k_spec_gauss(double2* __restrict__ U, double2* __restrict__ out, GridArgs g, double s2) {
  long q = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= g.Nc) return;
  const int d = g.d;
  ModeIdx m = decode(q, g);
  double kk = (double)lead_k2(m, g);
  int kz = m.j[d - 1];
  double2 v = U[q];
  if (kz == 0) {
    double g0 = exp(-0.5 * s2 * kk), gN = exp(-0.5 * s2 * (kk + 0.25 * (double)g.n[d - 1] * g.n[d - 1]));
    double alpha = 0.5 * (g0 + gN), delta = 0.5 * (g0 - gN);
    double2 vn = U[encode_neg(q, m, g)];
    out[q] = make_double2(alpha * v.x + delta * vn.x, alpha * v.y - delta * vn.y);
  } else {
    double gk = exp(-0.5 * s2 * (kk + (double)kz * kz));
    out[q] = make_double2(gk * v.x, gk * v.y);
  }
}

GridArgs args(const Grid& g) {
  GridArgs a;
  a.d = g.d;
  for (int i = 0; i < 3; ++i) a.n[i] = g.n[i];
  a.M = g.M;
  a.Nc = g.Nc;
  a.Nc1 = g.Nc / g.B;
  a.lg1 = 0;
  while ((1L << a.lg1) < a.Nc1) ++a.lg1;
  for (int i = 0; i < g.d; ++i) {
    a.lg[i] = 0;
    while ((1 << a.lg[i]) < (i == g.d - 1 ? g.M : g.n[i])) ++a.lg[i];
  }
  return a;
}

unsigned blocks_for(long n, int bs = 256) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace

Grid make_grid(int d, const int64_t* n, int batch) {
  Grid g;
  if (batch < 1) throw StatusError{1, "batch must be >= 1"};
  if (d != 2 && d != 3) throw StatusError{1, "d must be 2 or 3"};
  g.d = d;
  g.N = 1;
  for (int a = 0; a < d; ++a) {
    int64_t k = n[a];
    if (k < 8 || k > 512 || (k & (k - 1)) != 0)
      throw StatusError{1, "grid sizes must be powers of two in [8, 512]"};
    g.n[a] = (int)k;
    g.N *= k;
  }
  g.N1 = g.N;
  g.B = batch;
  g.N *= batch;
  g.L = g.n[d - 1];
  g.M = g.L / 2;
  g.Nc = g.N / 2;
  g.rows = g.N / g.L;
  return g;
}

long inv_k2_count(const Grid& g) {
  long n = 1;
  for (int a = 0; a < g.d; ++a) n += (long)(g.n[a] / 2) * (g.n[a] / 2);
  return n;
}

void fill_inv_k2(double* t, long count, double beta, int reg, cudaStream_t s) {
  k_inv_k2<<<blocks_for(count), 256, 0, s>>>(t, count, beta, reg);
  REG_LAUNCH();
}

void spec_tail(const Grid& g, cudaStream_t s, const double2* V, const double2* F, double2* out, int nc, double beta,
               const double* Cg_dev, int reg, int stokes, const double* betas, const double* inv_k2) {
  if (nc > kMaxNc) throw StatusError{1, "n_c too large"};
  auto run = [&](auto k) {
    chain(k, blocks_for(g.Nc), 256, s, V, F, out, args(g), nc, beta, Cg_dev, reg, stokes, betas, inv_k2);
  };
  auto dim = [&](auto d) {
    constexpr int D = decltype(d)::value;
    if (nc == 1) run(k_spec_tail<1, D>);
    else if (nc == 2) run(k_spec_tail<2, D>);
    else if (nc == 3) run(k_spec_tail<3, D>);
    else run(k_spec_tail<0, D>);
  };
  if (g.d == 2) dim(std::integral_constant<int, 2>{});
  else dim(std::integral_constant<int, 3>{});
}

void spec_precond(const Grid& g, cudaStream_t s, const double2* R, double2* out, int nc, double beta,
                  const double* Ci_dev, int reg, const double* betas, const double* inv) {
  auto run = [&](auto k) {
    chain(k, blocks_for(g.Nc), 256, s, R, out, args(g), nc, beta, Ci_dev, reg, betas, inv);
  };
  auto dim = [&](auto d) {
    constexpr int D = decltype(d)::value;
    if (nc == 1) run(k_spec_precond<1, D>);
    else if (nc == 2) run(k_spec_precond<2, D>);
    else if (nc == 3) run(k_spec_precond<3, D>);
    else run(k_spec_precond<0, D>);
  };
  if (g.d == 2) dim(std::integral_constant<int, 2>{});
  else dim(std::integral_constant<int, 3>{});
}

void spec_gauss(const Grid& g, cudaStream_t s, double2* U, double2* out, double sigma) {
  k_spec_gauss<<<blocks_for(g.Nc), 256, 0, s>>>(U, out, args(g), sigma * sigma);
  REG_LAUNCH();
}

// Trigonometric interpolation onto a grid refined per axis: the packed
// spectrum Q of the fine grid f from the packed spectrum P of the coarse grid
// c (nfields fields each; scale = N_f / N_c, so the fine inverse transform
// returns point values). A mode with |k_a| < n_a/2 on every axis keeps its
// coefficient; every other mode is zero, the coarse Nyquist modes included:
// the coarse derivatives treat those as constants (first derivatives and the
// Leray projection use the masked wavenumber), so the interpolated field is
// the part of the velocity that the coarse operators differentiate, and a
// velocity that is divergence-free on the coarse grid stays divergence-free.
// On the last axis the coarse slot 0 (DC + i Nyquist, both Hermitian in the
// other axes) is unpacked and its DC half goes to the fine slot 0.
__global__ void k_spec_upsample(const double2* __restrict__ P, double2* __restrict__ Q, GridArgs c, GridArgs f,
                                int nfields, double scale) {
  const long total = (long)nfields * f.Nc;
  for (long t = (long)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (long)gridDim.x * blockDim.x) {
    const long fld = t / f.Nc, q = t % f.Nc;
    const ModeIdx m = decode(q, f);
    bool zero = m.j[f.d - 1] >= c.M;
    long row = 0, nrow = 0;  // coarse row of k' and of -k'
    for (int a = 0; a < f.d - 1 && !zero; ++a) {
      const long i = m.j[a];
      const long k = i < f.n[a] / 2 ? i : i - f.n[a];
      const long h = c.n[a] / 2;
      if (k >= h || k <= -h) {
        zero = true;
        break;
      }
      const long ci = (k + c.n[a]) % c.n[a];
      row = row * c.n[a] + ci;
      nrow = nrow * c.n[a] + (c.n[a] - ci) % c.n[a];
    }
    double2 out = make_double2(0.0, 0.0);
    if (!zero) {
      const double2* Pf = P + fld * c.Nc;
      const long kz = m.j[f.d - 1];
      if (kz > 0) {
        const double2 z = Pf[row * c.M + kz];
        out = make_double2(scale * z.x, scale * z.y);
      } else {  // the DC half of the coarse slot 0: (z + conj(zn)) / 2
        const double2 z = Pf[row * c.M], zn = Pf[nrow * c.M];
        out = make_double2(0.5 * scale * (z.x + zn.x), 0.5 * scale * (z.y - zn.y));
      }
    }
    Q[fld * f.Nc + q] = out;
  }
}

void spec_upsample(const Grid& c, const Grid& f, cudaStream_t s, const double2* P, double2* Q, int nfields) {
  const long total = (long)nfields * f.Nc;
  const int blocks = (int)std::min<long>((total + 255) / 256, (long)kSMs * 16);
  k_spec_upsample<<<blocks, 256, 0, s>>>(P, Q, args(c), args(f), nfields, (double)f.N / (double)c.N);
  REG_LAUNCH();
}

}  // namespace reg

namespace reg {

static std::atomic<long> g_launches{0};
static thread_local long tl_launches = 0;
void count_launch() {
  g_launches.fetch_add(1, std::memory_order_relaxed);
  ++tl_launches;
}
long thread_launch_count() { return tl_launches; }
void add_launches(long n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
long launch_count() { return g_launches.load(std::memory_order_relaxed); }

thread_local KernelProfiler* tl_prof = nullptr;
thread_local bool tl_plain_launch = false;

KernelProfiler::~KernelProfiler() {
  for (auto& r : recs) {
    cudaEventDestroy(r.a);
    cudaEventDestroy(r.b);
  }
  for (auto e : pool) cudaEventDestroy(e);
}

cudaEvent_t KernelProfiler::take() {
  if (!pool.empty()) {
    cudaEvent_t e = pool.back();
    pool.pop_back();
    return e;
  }
  cudaEvent_t e;
  REG_CUDA(cudaEventCreate(&e));
  return e;
}

void KernelProfiler::collect(double* ms, double* bytes, long* count) {
  for (int k = 0; k < KK_COUNT; ++k) {
    ms[k] = 0;
    bytes[k] = 0;
    count[k] = 0;
    last_flops[k] = 0;
  }
  for (auto& r : recs) {
    REG_CUDA(cudaEventSynchronize(r.b));
    float t = 0;
    REG_CUDA(cudaEventElapsedTime(&t, r.a, r.b));
    ms[r.kind] += t;
    bytes[r.kind] += r.bytes;
    last_flops[r.kind] += r.flops;
    count[r.kind] += 1;
    pool.push_back(r.a);
    pool.push_back(r.b);
  }
  recs.clear();
}

ProfScope::ProfScope(int k, cudaStream_t st, double b, double f) : kind(k), s(st), bytes(b), flops(f) {
  if (tl_prof && (tl_prof->mask & (1u << k))) {
    a = tl_prof->take();
    REG_CUDA(cudaEventRecord(a, s));
  }
}

ProfScope::~ProfScope() {
  if (!a || !tl_prof) return;
  cudaEvent_t b = tl_prof->take();
  if (cudaEventRecord(b, s) != cudaSuccess) return;
  tl_prof->recs.push_back(KernelProfiler::Rec{kind, a, b, bytes, flops});
}

}  // namespace reg
