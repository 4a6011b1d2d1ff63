// Online tuner for the choice of the FP32 GEMM kernel (and with it the tile shape).
// Launches are grouped by device, the average number of 32-wide k-chunks per
// product (log2 bucket) and the logical flop count (log2 bucket).  The first
// launches of a class run each candidate once between two events; once both
// timings have completed (checked without waiting, at a later launch of the
// class) the candidate with the lower time per flop is used for the class for
// the rest of the process.  Until then -- and whenever a measurement is still
// in flight -- the rule "tcgen05 from four k-chunks per product on" decides.
// Either kernel computes the same products; only FP32 rounding order differs.
// Host code only.
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <map>
#include <memory>
#include <mutex>
#include <tuple>

namespace spand {

struct GemmTuner {
  struct Entry {
    int choice = -1;                 // decided: 0 tcgen05, 1 mma.sync
    bool pending[2] = {false, false};    // a trial is out
    bool recorded[2] = {false, false};   // its events are on the stream
    bool done[2] = {false, false};
    double per_flop[2] = {0, 0};
    double flops[2] = {0, 0};
    cudaEvent_t ev[2][2] = {{nullptr, nullptr}, {nullptr, nullptr}};
  };
  // A launch to be timed.  One that never happens (a queue of launches is dropped
  // after an error) gives its candidate back with the last copy of the pointer.
  struct Trial {
    GemmTuner* tuner;
    Entry* e;
    int c;
    bool over = false;
    Trial(GemmTuner* t, Entry* entry, int cand) : tuner(t), e(entry), c(cand) {}
    Trial(const Trial&) = delete;
    Trial& operator=(const Trial&) = delete;
    void begin(cudaStream_t st) { cudaEventRecord(e->ev[c][0], st); }
    void end(cudaStream_t st) {
      if (cudaEventRecord(e->ev[c][1], st) != cudaSuccess) return;
      std::lock_guard<std::mutex> g(tuner->mu);
      e->recorded[c] = over = true;
    }
    ~Trial() {
      if (over) return;
      std::lock_guard<std::mutex> g(tuner->mu);
      e->pending[c] = false;
    }
  };
  std::mutex mu;
  std::map<std::tuple<int, int, int>, Entry> table;
  static GemmTuner& get() {
    static GemmTuner* t = new GemmTuner();   // process lifetime
    return *t;
  }
  // the kernel (0 tcgen05, 1 mma.sync) and, when this launch is to be timed, its trial
  int pick(int dev, double avg_chunks, double flops, bool verbose, std::shared_ptr<Trial>& trial) {
    trial.reset();
    const int rule = avg_chunks >= 4.0 ? 0 : 1;
    const int cb = std::min(6, (int)std::floor(std::log2(std::max(1.0, avg_chunks))));
    const int fb = std::min(12, (int)std::floor(std::log2(std::max(1.0, flops / 1e7))));
    std::lock_guard<std::mutex> g(mu);
    Entry& E = table[std::make_tuple(dev, cb, fb)];
    if (E.choice >= 0) return E.choice;
    for (int c = 0; c < 2; ++c)
      if (E.pending[c] && E.recorded[c] && !E.done[c]) {
        const cudaError_t q = cudaEventQuery(E.ev[c][1]);
        if (q == cudaSuccess) {
          float ms = 0.f;
          if (cudaEventElapsedTime(&ms, E.ev[c][0], E.ev[c][1]) == cudaSuccess && E.flops[c] > 0) {
            E.per_flop[c] = ms / E.flops[c];
            E.done[c] = true;
          }
          E.pending[c] = E.recorded[c] = false;
        } else if (q == cudaErrorNotReady && cudaPeekAtLastError() == cudaErrorNotReady) {
          cudaGetLastError();          // a not-ready query is not an error of ours
        }
      }
    if (E.done[0] && E.done[1]) {
      E.choice = E.per_flop[0] <= E.per_flop[1] ? 0 : 1;
      for (auto& pr : E.ev)
        for (auto& e : pr)
          if (e) cudaEventDestroy(e);
      if (verbose)
        std::fprintf(stderr, "spand: GEMM class (k-chunks 2^%d, flops 2^%d x 1e7): tcgen05 %.3g, mma.sync %.3g ms/GF -> %s\n",
                     cb, fb, E.per_flop[0] * 1e9, E.per_flop[1] * 1e9, E.choice == 0 ? "tcgen05" : "mma.sync");
      return E.choice;
    }
    for (int c = 0; c < 2; ++c)
      if (!E.done[c] && !E.pending[c]) {
        if (!E.ev[c][0]) {
          if (cudaEventCreate(&E.ev[c][0]) != cudaSuccess || cudaEventCreate(&E.ev[c][1]) != cudaSuccess) {
            cudaGetLastError();
            return rule;
          }
        }
        E.pending[c] = true;
        E.flops[c] = flops;
        trial = std::make_shared<Trial>(this, &E, c);
        return c;
      }
    return rule;                       // both measurements still in flight
  }
};

}  // namespace spand
