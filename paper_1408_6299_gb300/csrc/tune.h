// tune.h -- choice of the autotuner among variants of a pure pass (one that
// writes only what it does not read, so running it again gives the same
// result). The variants of a pass give the same bits; they differ in the work
// per block.
#pragma once
#include <stdlib.h>

#include <map>
#include <mutex>
#include <string>
#include <tuple>

#include "internal.h"

namespace reg {

// Variant 0..nv-1 for pass `kind` (which names the line plan: sizes are rounded, so
// two plans may meet in one size) on elements of `size` bytes, lines of length
// L and `work` lines: the choice of this process for the shape, or the
// persistent one (tune.cu), else, outside a stream capture, the variants run
// on the call's own buffers, timed with CUDA events on the stream, and the
// fastest is recorded. During a capture, and
// with REG_AUTOTUNE=0, variant 0 runs and nothing is recorded.
template <typename Run>
int tuned_choice(const char* kind, int size, int L, long work, int nv, cudaStream_t st, Run run) {
  using Key = std::tuple<int, std::string, int, int, long>;
  static std::mutex mu;
  static std::map<Key, int> mem;
  int dev = 0;
  REG_CUDA(cudaGetDevice(&dev));
  const Key key(dev, kind, size, L, work);
  {
    std::lock_guard<std::mutex> lk(mu);
    auto it = mem.find(key);
    if (it != mem.end()) return it->second;
  }
  const std::string name = tune_device_tag() + "|" + kind + "|" + (size == 4 ? "f32" : "f64") + "|L" +
                           std::to_string(L) + "|n" + std::to_string(work);
  int pick = tune_lookup(name);
  if (pick < 0 || pick >= nv) {
    const char* env = getenv("REG_AUTOTUNE");
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    REG_CUDA(cudaStreamIsCapturing(st, &cs));
    if ((env && env[0] == '0') || cs != cudaStreamCaptureStatusNone) return 0;
    cudaEvent_t e0, e1;
    REG_CUDA(cudaEventCreate(&e0));
    REG_CUDA(cudaEventCreate(&e1));
    auto timed = [&](int v, int launches) {
      REG_CUDA(cudaEventRecord(e0, st));
      for (int k = 0; k < launches; ++k) run(v);
      REG_CUDA(cudaEventRecord(e1, st));
      REG_CUDA(cudaEventSynchronize(e1));
      float ms = 0;
      REG_CUDA(cudaEventElapsedTime(&ms, e0, e1));
      return ms;
    };
    // In turn, so that a disturbance does not meet one variant alone, and the shortest of
    // six; several launches at a time, which overlap as in a sweep, more of short ones.
    // Three single launches each, summed, took the slower one now and then: 512^2 FP64
    // transport 6200 us instead of 4660, 64^3 Stokes mixed matvec 1400 instead of 1305;
    // with four of the 2 us passes at 32^2 (matvec 489 or 505 us) it was still chance.
    constexpr int kReps = 6, kMaxVariants = 4;
    float best[kMaxVariants] = {1e30f, 1e30f, 1e30f, 1e30f};
    nv = nv < kMaxVariants ? nv : kMaxVariants;
    for (int v = 0; v < nv; ++v) run(v);
    const int launches = timed(0, 1) < 0.03f ? 16 : 4;
    for (int r = 0; r < kReps; ++r)
      for (int v = 0; v < nv; ++v) {
        const float ms = timed(v, launches);
        best[v] = ms < best[v] ? ms : best[v];
      }
    pick = 0;
    for (int v = 1; v < nv; ++v)
      if (best[v] < best[pick]) pick = v;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    tune_store(name, pick);
  }
  std::lock_guard<std::mutex> lk(mu);
  mem[key] = pick;
  return pick;
}

// work sizes rounded up to a power of two: stacks of similar size share a choice
inline long tune_size(long n) {
  long r = 1;
  while (r < n) r *= 2;
  return r;
}

}  // namespace reg
