// internal.h -- host-side declarations shared by the translation units of the
// registration library (not part of the public C ABI, see include/reg.h).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <functional>
#include <memory>
#include <string>
#include <vector>

#include "fft.cuh"

namespace reg {

// CUDA error -> exception carrying the failing call, caught at the C ABI.
struct CudaError {
  cudaError_t code;
  std::string what;
};
struct StatusError {
  int status;
  std::string what;
};

#define REG_CUDA(call)                                                                      \
  do {                                                                                      \
    cudaError_t e_ = (call);                                                                \
    if (e_ != cudaSuccess) throw ::reg::CudaError{e_, std::string(#call) + ": " +           \
                                                      cudaGetErrorString(e_)};              \
  } while (0)
#define REG_LAUNCH()         \
  do {                       \
    ::reg::count_launch();   \
    REG_CUDA(cudaGetLastError()); \
  } while (0)

// Host data to device memory, complete on return. cudaMemcpy from pageable memory
// may return with the transfer still under way on the NULL stream, and a
// non-blocking stream has no order behind that stream.
inline void upload(void* dst, const void* src, size_t bytes) {
  REG_CUDA(cudaMemcpy(dst, src, bytes, cudaMemcpyHostToDevice));
  REG_CUDA(cudaStreamSynchronize(nullptr));
}

// ---------------------------------------------------------------------------
// Kernel accounting: a process-wide launch counter, and optional CUDA-event
// bracketing of launches by kind (enabled per context through the C ABI).
// ---------------------------------------------------------------------------
enum KernelKind {
  KK_ROWS_R2C = 0,  // real-to-complex rows of whole-field transforms
  KK_ROWS_C2R = 1,  // row pass of a stage with its epilogue, or complex-to-real rows
  KK_COLS = 2,      // strided pass
  KK_MULT = 3,      // Fourier multipliers
  KK_STAGE = 4,     // Heun stage / transport right-hand side
  KK_FORCE = 5,     // body-force accumulation
  KK_OTHER = 6,     // everything else
  KK_COUNT = 7
};
void count_launch();
void add_launches(long n);  // kernels launched by a graph replay
long launch_count();
long thread_launch_count();  // those of count_launch() on this thread

// Launch of a kernel that begins with chain_enter(): it may be set up while its
// predecessor on the stream still runs, and waits there for its results. The
// kernels of a sweep depend on one another and run a few microseconds each on
// small grids, so the launch gap between them counts. (Behind a join of two
// streams the launch is an ordinary one: tl_plain_launch.)
extern thread_local bool tl_plain_launch;
template <typename... P, typename... A>
void chain(void (*kern)(P...), dim3 grid, unsigned block, cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = tl_plain_launch ? 0 : 1;
  tl_plain_launch = false;
  count_launch();
  REG_CUDA(cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...));
}

struct KernelProfiler {
  unsigned mask = 0;
  struct Rec {
    int kind;
    cudaEvent_t a, b;
    double bytes, flops;
  };
  std::vector<Rec> recs;
  std::vector<cudaEvent_t> pool;
  double last_flops[KK_COUNT] = {0};  // per kind, of the last collected window
  ~KernelProfiler();
  cudaEvent_t take();
  void collect(double* ms, double* bytes, long* count);  // synchronises
};
extern thread_local KernelProfiler* tl_prof;

// bracket one launch; bytes = algorithmic bytes moved by it, flops = the
// floating-point operations of its transforms (0 where not counted)
struct ProfScope {
  int kind;
  cudaStream_t s;
  double bytes, flops;
  cudaEvent_t a = nullptr;
  ProfScope(int k, cudaStream_t st, double b, double f = 0.0);
  ~ProfScope();
};

// Periodic nodal grid, row-major with the last axis fastest. Real fields hold
// N values; packed half spectra hold Nc = N/2 complex values laid out as
// [n_0]..[n_{d-2}][M], M = n_{d-1}/2, where slot 0 of the last axis carries
// uhat(k',0) + i*uhat(k',n_{d-1}/2) (DC and Nyquist columns of the last axis).
// A grid of B independent problems of the same shape, stacked along an
// untransformed leading axis (B = 1: one problem). N, Nc and rows count all
// problems; every field is laid out [B][n_0]...[n_{d-1}].
struct Grid {
  int d = 0;
  int n[3] = {1, 1, 1};
  long N = 0;   // real points
  long Nc = 0;  // packed spectral points
  int L = 0;    // last-axis length
  int M = 0;    // L/2
  long rows = 0;  // N / L
  int B = 1;      // stacked problems
  long N1 = 0;    // real points of one problem
};

Grid make_grid(int d, const int64_t* n, int batch = 1);

// set the text that reg_last_error(NULL) returns on this thread
void set_thread_error(const std::string& msg);

// Persistent autotuner choices (tune.cu): -1 when the key has none yet.
// Keys start with tune_device_tag() (device name / multiprocessor count).
int tune_lookup(const std::string& key);
void tune_store(const std::string& key, int choice);
std::string tune_device_tag();

// Twiddle tables of the line transforms (line.cuh) of one grid's axis lengths,
// for both plans. Single precision: kind 0 float2 entries, kind 1 paired
// entries (c, c, s, s). Double precision: kind 1, fixed-point words.
template <typename T>
class LineTables {
 public:
  explicit LineTables(const Grid& g);
  ~LineTables();
  LineTables(const LineTables&) = delete;
  LineTables& operator=(const LineTables&) = delete;
  const void* get(int L, bool narrow, int kind) const;

 private:
  unsigned char* dev_ = nullptr;
  long off_[44];
};

// The fixed-point tables of the wide plans of every length 8..512, for callers
// that place them themselves: byte offsets by log2 L into off; out may be null
// to query the size in bytes.
size_t write_wide_tables(unsigned char* out, long* off);

// Whether lines that take so many threads on the wide plan run the narrow one
// (line.cuh) instead. Wide lines hold the fewest operations, narrow ones
// shorter serial work per thread and fewer registers. Measured: 128^2 FP64
// gradient 5600 us wide, 2170 narrow; 128^3 FP64 gradient 42.7 ms wide, 38.4
// narrow; 128^3 mixed matvec, checkpoints every 8, 16.5 ms with this limit at
// half, 12.6 here, 14.1 at double; 256^3 mixed matvec 180 ms wide, 246 narrow.
inline bool narrow_lines(long wide_threads, int size) { return wide_threads < (long)kSMs * (size == 8 ? 1024 : 512); }
// The lines that count for it. Plans round differently. In double precision the
// plan follows the size of one problem, so that a problem has the same bits in any
// stack and after its stack is rebuilt; in single precision that of the whole stack,
// which a narrow plan would slow down by up to 1.4 (256^3 above).
inline long plan_lines(const Grid& g, long lines, int size) { return size == 8 ? lines / g.B : lines; }

// A grid with its stream and line tables in precision T: what the stages run on.
template <typename T>
class Spectral {
 public:
  Spectral(const Grid& g, cudaStream_t s) : g_(g), s_(s), lines_(g) {}
  ~Spectral() {
    if (fork_ev_) cudaEventDestroy(fork_ev_);
    if (join_ev_) cudaEventDestroy(join_ev_);
    if (aux_) cudaStreamDestroy(aux_);
  }
  Spectral(const Spectral&) = delete;
  Spectral& operator=(const Spectral&) = delete;
  // a second stream for launches that do not depend on one another: fork()
  // orders it behind the stream, join() the stream behind it
  cudaStream_t fork() {
    if (!aux_) {
      REG_CUDA(cudaEventCreateWithFlags(&fork_ev_, cudaEventDisableTiming));
      REG_CUDA(cudaEventCreateWithFlags(&join_ev_, cudaEventDisableTiming));
      REG_CUDA(cudaStreamCreateWithFlags(&aux_, cudaStreamNonBlocking));
    }
    REG_CUDA(cudaEventRecord(fork_ev_, s_));
    REG_CUDA(cudaStreamWaitEvent(aux_, fork_ev_, 0));
    return aux_;
  }
  void join() {
    REG_CUDA(cudaEventRecord(join_ev_, aux_));
    REG_CUDA(cudaStreamWaitEvent(s_, join_ev_, 0));
  }
  const Grid& grid() const { return g_; }
  cudaStream_t stream() const { return s_; }
  void set_stream(cudaStream_t s) { s_ = s; }
  const void* line_table(int L, bool narrow, int kind) const { return lines_.get(L, narrow, kind); }

 private:
  Grid g_;
  cudaStream_t s_, aux_ = nullptr;
  cudaEvent_t fork_ev_ = nullptr, join_ev_ = nullptr;
  LineTables<T> lines_;
};

// Double-precision transforms between real fields and packed half spectra, nf
// fields at strides N and Nc per call (transform.cu).
class FieldTransforms {
 public:
  using TableFn = std::function<const void*(int L, bool narrow)>;  // fixed-point line tables
  // tuned: plans by size and autotuned blocks; else the wide plans, nothing measured
  FieldTransforms(const Grid& g, cudaStream_t s, TableFn tables, bool tuned);
  void fwd(const double* u, double2* U, int nf) const;  // unnormalised
  void inv(double2* U, double* u, int nf) const;        // normalised by 1/N; U is overwritten

 private:
  void cols(double2* U, int axis, int nf, bool inverse) const;
  bool narrow(int L, long lines) const;
  Grid g_;
  cudaStream_t s_;
  TableFn tables_;
  bool tuned_;
};

// ---------------------------------------------------------------------------
// Transport stages (stage.cuh): advection k = -v.grad u [- grad m . v~] and
// divergence k = div(v lam), each with its Runge-Kutta update in the last pass.
// ---------------------------------------------------------------------------
namespace fused {
template <typename T>
struct AdvEpi;
template <typename T>
struct DivEpi;
}  // namespace fused
// gx, gy: scratch fields (gy unused in 2D)
template <typename T>
void adv_stage(Spectral<T>& sp, const T* u, const fused::AdvEpi<T>& e, T* gx, T* gy);
// two 3D advection stages (fields uA, uB) sharing their launches; Z: four scratch fields
template <typename T>
void adv2_stage(Spectral<T>& sp, const T* uA, const fused::AdvEpi<T>& eA, const T* uB, const fused::AdvEpi<T>& eB,
                T* const* Z);
// a: d velocity fields at stride N
template <typename T>
void div_stage(Spectral<T>& sp, const T* lam, const T* a, const fused::DivEpi<T>& e, T* kx, T* ky);

// ---------------------------------------------------------------------------
// Fourier-diagonal operators on whole coefficient vectors (FP64), with the
// DC/Nyquist pairing of the packed last-axis slot 0.
// ---------------------------------------------------------------------------
// Tables of every squared wavenumber m = 1 .. sum_a (n_a/2)^2, at [m] (device):
// 1 / (beta m^reg), rounded as one division.
long inv_k2_count(const Grid& g);
void fill_inv_k2(double* t, long count, double beta, int reg, cudaStream_t s);
// out_l = beta sum_l' Cg[l][l'] a(k) V_l' + (stokes ? K F_l : F_l); F may be null.
// betas (device, may be null): one beta per stacked problem, replacing beta.
// inv_k2: the table of 1 / m; null: divided per mode
void spec_tail(const Grid& g, cudaStream_t s, const double2* V, const double2* F, double2* out, int nc,
               double beta, const double* Cg_dev, int reg, int stokes, const double* betas, const double* inv_k2);
// out_l = sum_l' Ci[l][l'] s(k) R_l' with s = 1/(beta a(k)), s = 1 at k = 0.
// inv: the table of 1 / (beta m^reg); null: divided per mode
void spec_precond(const Grid& g, cudaStream_t s, const double2* R, double2* out, int nc, double beta,
                  const double* Ci_dev, int reg, const double* betas, const double* inv);
// Gaussian filter exp(-sigma^2 |k|^2 / 2) of one packed FP64 field (out may not alias U)
void spec_gauss(const Grid& g, cudaStream_t s, double2* U, double2* out, double sigma);
// trigonometric interpolation of nfields packed FP64 spectra of grid c onto the
// finer grid f (every axis refined by a factor >= 2; one problem, no stacking)
void spec_upsample(const Grid& c, const Grid& f, cudaStream_t s, const double2* P, double2* Q, int nfields);

}  // namespace reg
