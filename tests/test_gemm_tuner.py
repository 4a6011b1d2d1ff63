"""The tuner's bookkeeping on the host, against a CUDA runtime of a few stubs: a
trial whose launch is dropped is handed out again, and a class is decided once both
candidates have been timed."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

STUB = r"""
#pragma once
typedef int cudaError_t;
typedef void* cudaStream_t;
enum { cudaSuccess = 0, cudaErrorInvalidValue = 1, cudaErrorNotReady = 600 };
struct StubEvent { bool on = false; float at = 0; };
typedef StubEvent* cudaEvent_t;
static float stub_clock = 0;
static bool stub_ready = true;
inline cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = new StubEvent; return cudaSuccess; }
inline cudaError_t cudaEventDestroy(cudaEvent_t e) { delete e; return cudaSuccess; }
inline cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { e->on = true; e->at = stub_clock; return cudaSuccess; }
inline cudaError_t cudaEventQuery(cudaEvent_t) { return stub_ready ? cudaSuccess : cudaErrorNotReady; }
inline cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
  if (!a->on || !b->on) return cudaErrorInvalidValue;
  *ms = b->at - a->at;
  return cudaSuccess;
}
inline cudaError_t cudaPeekAtLastError() { return cudaSuccess; }
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
"""

MAIN = r"""
#include <functional>
#include <vector>
#include "gemm_tuner.h"
using spand::GemmTuner;
#define CHECK(x) if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; }
int main() {
  GemmTuner t;
  std::shared_ptr<GemmTuner::Trial> a, b, c;
  auto launch = [](std::shared_ptr<GemmTuner::Trial>& r, float ms) {
    r->begin(nullptr);
    stub_clock += ms;
    r->end(nullptr);
    r.reset();
  };
  // both candidates out; a third launch of the class follows the rule
  CHECK(t.pick(0, 8, 1e9, false, a) == 0 && a);
  CHECK(t.pick(0, 8, 1e9, false, b) == 1 && b);
  CHECK(t.pick(0, 8, 1e9, false, c) == 0 && !c);
  // the first is held by two copies of a queued launch and dropped with them
  {
    std::vector<std::function<void()>> queue;
    queue.emplace_back([a] { a->begin(nullptr); });
    a.reset();
    CHECK(t.pick(0, 8, 1e9, false, c) == 0 && !c);
  }
  CHECK(t.pick(0, 8, 1e9, false, a) == 0 && a);
  // one that began and never ended is dropped too
  a->begin(nullptr);
  a.reset();
  CHECK(t.pick(0, 8, 1e9, false, a) == 0 && a);
  launch(a, 3.f);
  launch(b, 2.f);
  stub_ready = false;
  CHECK(t.pick(0, 8, 1e9, false, c) == 0 && !c);   // still in flight: the rule
  stub_ready = true;
  CHECK(t.pick(0, 8, 1e9, false, c) == 1 && !c);   // the faster one, for good
  CHECK(t.pick(0, 8, 1e9, false, c) == 1 && !c);
  CHECK(t.pick(1, 8, 1e9, false, c) == 0 && c);    // another device is another class
  return 0;
}
"""


def test_dropped_trials_are_handed_out_again(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(STUB)
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = tmp_path / "main"
    subprocess.run(["g++", "-std=c++17", "-I", str(tmp_path), "-I",
                    os.path.join(ROOT, "paper_2101_01763_gb300", "csrc"), str(tmp_path / "main.cpp"), "-o", str(exe),
                    "-lpthread"], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
