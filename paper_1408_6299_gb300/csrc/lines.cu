// lines.cu -- twiddle tables of the line transforms (line.cuh, fixed.cuh).
#include <math.h>

#include <algorithm>

#include "internal.h"
#include "line.cuh"

namespace reg {
namespace {

// exp(-2 pi i m / 512) = c - i s, m < 512, from the first octant
struct Circle {
  long double c[512], s[512];
  Circle() {
    long double oc[65], os[65];
    for (int m = 0; m <= 64; ++m) {
      const long double a = acosl(-1.0L) * m / 256;
      oc[m] = cosl(a);
      os[m] = sinl(a);
    }
    for (int m = 0; m < 512; ++m) {
      const int quarter = m / 128, r = m % 128;
      const long double x = r <= 64 ? oc[r] : os[128 - r], y = r <= 64 ? os[r] : oc[128 - r];
      c[m] = quarter == 0 ? x : (quarter == 1 ? -y : (quarter == 2 ? -x : y));
      s[m] = quarter == 0 ? y : (quarter == 1 ? x : (quarter == 2 ? -y : -x));
    }
  }
};
const Circle& circle() {
  static const Circle k;
  return k;
}

// x 2^62, rounded, as h 2^32 + l with l a signed low word
void fixed_words(long double x, int* h, int* l) {
  const long long v = llrintl(ldexpl(x, 62));
  *l = (int)(unsigned)(unsigned long long)v;
  *h = (int)((v - *l) >> 32);
}

void put(std::vector<unsigned char>& out, const void* p, size_t n) {
  const unsigned char* b = static_cast<const unsigned char*>(p);
  out.insert(out.end(), b, b + n);
}

template <typename T, int L, bool NARROW>
void emit(std::vector<unsigned char>& out, int kind) {
  using P = LinePlan<L, NARROW>;
  const Circle& k = circle();
  for (int block = 0; block < (sizeof(T) == 8 ? 3 : 2); ++block)
    for (int s = 1; s < P::S; ++s) {
      const bool inv = block == 1;
      const int R = line_radix<P>(s, inv), ns = line_ns<P>(s, inv);
      for (int r = 0; r < R; ++r)
        for (int t = 0; t < ns; ++t) {
          const int m = r * t * (512 / (ns * R)) % 512;
          const long double c = k.c[m], d = -k.s[m];
          if (sizeof(T) == 4 && kind == 1) {
            const float4 w = make_float4((float)c, (float)c, (float)d, (float)d);
            put(out, &w, sizeof w);
          } else if (sizeof(T) == 4) {
            const float2 w = make_float2((float)c, (float)d);
            put(out, &w, sizeof w);
          } else {  // fixed point; block 0 takes 1/R with the twiddle
            int4 w;
            const long double f = block == 0 ? 1.0L / R : 1.0L;
            fixed_words(c * f, &w.x, &w.y);
            fixed_words(d * f, &w.z, &w.w);
            put(out, &w, sizeof w);
          }
        }
    }
}

template <typename T>
void emit_any(std::vector<unsigned char>& out, int L, bool narrow, int kind) {
  switch (L) {
    case 8: return narrow ? emit<T, 8, true>(out, kind) : emit<T, 8, false>(out, kind);
    case 16: return narrow ? emit<T, 16, true>(out, kind) : emit<T, 16, false>(out, kind);
    case 32: return narrow ? emit<T, 32, true>(out, kind) : emit<T, 32, false>(out, kind);
    case 64: return narrow ? emit<T, 64, true>(out, kind) : emit<T, 64, false>(out, kind);
    case 128: return narrow ? emit<T, 128, true>(out, kind) : emit<T, 128, false>(out, kind);
    case 256: return narrow ? emit<T, 256, true>(out, kind) : emit<T, 256, false>(out, kind);
    case 512: return narrow ? emit<T, 512, true>(out, kind) : emit<T, 512, false>(out, kind);
  }
  throw StatusError{1, "unsupported line length"};
}

int table_slot(int L, bool narrow, int kind) { return (ilog2_c(L) * 2 + (narrow ? 1 : 0)) * 2 + kind; }

}  // namespace

template <typename T>
LineTables<T>::LineTables(const Grid& g) {
  std::vector<unsigned char> h;
  for (long& o : off_) o = -1;
  for (int a = 0; a < g.d; ++a)
    for (int narrow = 0; narrow < 2; ++narrow)
      for (int kind = sizeof(T) == 8; kind < 2; ++kind) {
        long& o = off_[table_slot(g.n[a], narrow, kind)];
        if (o >= 0) continue;
        h.resize((h.size() + 15) / 16 * 16);
        o = (long)h.size();
        emit_any<T>(h, g.n[a], narrow, kind);
      }
  h.resize(h.size() + 16);
  REG_CUDA(cudaMalloc(&dev_, h.size()));
  upload(dev_, h.data(), h.size());
}
template <typename T>
LineTables<T>::~LineTables() {
  if (dev_) cudaFree(dev_);
}
template <typename T>
const void* LineTables<T>::get(int L, bool narrow, int kind) const {
  return dev_ + off_[table_slot(L, narrow, kind)];
}

size_t write_wide_tables(unsigned char* out, long* off) {
  std::vector<unsigned char> h;
  for (int L = 8; L <= 512; L *= 2) {
    off[ilog2_c(L)] = (long)h.size();
    emit_any<double>(h, L, false, 1);
  }
  if (out) std::copy(h.begin(), h.end(), out);
  return h.size();
}

template class LineTables<float>;
template class LineTables<double>;

}  // namespace reg
