"""What the library keeps per device (csrc/perdevice.h), compiled for the host against a stand-in for the CUDA runtime
whose current device the program sets: a thread that goes from one device to another and back gets streams, events,
numbers and caches of the device it is on, and what it had before when it returns."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2507_06471_gb300", "csrc")

RUNTIME = r"""
#pragma once
#include <cstdlib>
struct Fake { int device; };
typedef Fake* cudaStream_t;
typedef Fake* cudaEvent_t;
typedef int cudaError_t;
enum { cudaSuccess = 0, cudaEventDisableTiming = 2, cudaStreamNonBlocking = 1 };
inline thread_local int fake_device = 0;
inline cudaError_t cudaGetDevice(int* d) { *d = fake_device; return cudaSuccess; }
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
inline cudaError_t fake_make(Fake** p) { *p = new Fake{fake_device}; return cudaSuccess; }
inline cudaError_t cudaStreamCreateWithFlags(cudaStream_t* p, unsigned) { return fake_make(p); }
inline cudaError_t cudaEventCreateWithFlags(cudaEvent_t* p, unsigned) { return fake_make(p); }
"""

PROGRAM = r"""
#include "perdevice.h"
#include <cstdio>
#include <thread>
#include <unordered_map>
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); std::exit(1); } } while (0)
using namespace cd;

static PerDevice number;

static void walk(cudaStream_t* aux0, cudaStream_t* cap0) {
  cudaStream_t aux[3], cap[3];
  for (int pass = 0; pass < 2; ++pass)
    for (int d : {0, 2, 1}) {
      fake_device = d;
      AuxStreams& a = aux_streams();
      CHECK(a.ok && a.fork->device == d);
      for (int i = 0; i < 3; ++i) CHECK(a.s[i]->device == d && a.join[i]->device == d);
      cudaStream_t c = nullptr;
      CHECK(capture_stream(&c) == cudaSuccess && c->device == d);
      if (pass == 0) {
        aux[d] = a.s[0];
        cap[d] = c;
      } else {
        CHECK(aux[d] == a.s[0] && cap[d] == c);
      }
    }
  CHECK(aux[0] != aux[1] && aux[1] != aux[2] && cap[0] != cap[1] && cap[1] != cap[2]);
  *aux0 = aux[0];
  *cap0 = cap[0];
}

int main() {
  cudaStream_t a1, a2, c1, c2;
  walk(&a1, &c1);
  std::thread(walk, &a2, &c2).join();
  CHECK(a1 != a2 && c1 != c2);  // a thread's own
  for (int d = 0; d < 70; ++d) {
    fake_device = d;
    CHECK(number.get() == 0);
    number.set(100 + d);
  }
  for (int d = 0; d < 70; ++d) {
    fake_device = d;
    CHECK(number.get() == (d < 64 ? 100 + d : 0));  // past the last one: asked again
  }
  ByDevice<std::unordered_map<const void*, int>> caches;
  for (int d : {0, 1, 300}) {
    fake_device = d;
    CHECK(caches.here().empty());
    caches.here()[&caches] = d;
  }
  for (int d : {0, 1, 300}) {
    fake_device = d;
    CHECK(caches.here().at(&caches) == d);
  }
  return 0;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_kept_per_device(tmp_path):
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    (tmp_path / "main.cpp").write_text(PROGRAM)
    exe = tmp_path / "main"
    subprocess.check_call(["g++", "-std=c++17", "-pthread", "-I", str(tmp_path), "-I", CSRC, "-o", str(exe),
                           str(tmp_path / "main.cpp")])
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_no_stream_event_or_occupancy_is_kept_for_a_thread_or_process_alone():
    """Every function-level static or thread_local of the sources is keyed by device, or belongs to none."""
    found = []
    for name in sorted(os.listdir(CSRC)):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
        found += [(name, m.group(0).strip()) for m in re.finditer(r"^[ ]+static\b[^;({=]*", text, flags=re.M)]
    kept = [(n, s) for n, s in found if not re.search(r"constexpr|const int |PerDevice|ByDevice<|std::mutex", s)]
    assert not kept, kept
    assert any("ByDevice<" in s for _, s in found) and any("PerDevice" in s for _, s in found)
