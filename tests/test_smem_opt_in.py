"""The opt-in to large dynamic shared memory is kept per device, as CUDA keeps it, and only grows:
the header's class against fakes of the two CUDA calls, compiled and run on the host."""
import glob
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_28979_gb300", "csrc")
CUDA = os.path.join(os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"))), "include")

PROGRAM = r"""
#include "smem_opt_in.h"
#include <cstdio>
#include <cstdlib>
#include <thread>
#include <vector>
static thread_local int device = 0;
static std::atomic<int> calls{0}, attr[2][80];   // [kernel][device]
static std::atomic<bool> fail{false};
static void k0(int) {}
static void k1(int) {}
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) {
  ++calls;
  if (a != cudaFuncAttributeMaxDynamicSharedMemorySize) return cudaErrorInvalidValue;
  if (fail) return cudaErrorMemoryAllocation;
  attr[f == reinterpret_cast<const void*>(&k1)][device] = v;
  return cudaSuccess;
}
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); std::exit(1); } } while (0)
int main() {
  static mot::SmemOptIn a, b;
  CHECK(a(k0, 48 * 1024) == cudaSuccess && calls == 0);          // the default holds it
  for (int d = 0; d < 2; ++d) {                                  // a device of its own each
    device = d;
    CHECK(a(k0, 80000) == cudaSuccess && attr[0][d] == 80000 && calls == d + 1);
    CHECK(a(k0, 80000) == cudaSuccess && a(k0, 60000) == cudaSuccess && calls == d + 1);
  }
  CHECK(b(k1, 70000) == cudaSuccess && attr[1][1] == 70000 && attr[1][0] == 0);   // a kernel of its own
  fail = true;
  CHECK(a(k0, 90000) == cudaErrorMemoryAllocation);              // reported, and tried again
  fail = false;
  CHECK(a(k0, 90000) == cudaSuccess && attr[0][1] == 90000 && attr[0][0] == 80000);
  device = 70;
  CHECK(a(k0, 50000) == cudaSuccess && a(k0, 60000) == cudaSuccess && attr[0][70] == 60000);
  for (int round = 0; round < 200; ++round) {                    // threads of mixed sizes: never lowered
    mot::SmemOptIn c;
    attr[0][2] = 0;
    std::atomic<int> low{0};
    std::vector<std::thread> ts;
    for (int t = 0; t < 8; ++t)
      ts.emplace_back([&, t] {
        device = 2;
        const int bytes = 50000 + 1000 * ((t * 5 + round) % 8);
        if (c(k0, bytes) != cudaSuccess || attr[0][2] < bytes) ++low;
      });
    for (auto& t : ts) t.join();
    CHECK(low == 0 && attr[0][2] == 57000);
  }
  return 0;
}
"""


def test_opt_in_is_remembered_per_device(tmp_path):
    if not os.path.exists(os.path.join(CUDA, "cuda_runtime_api.h")):
        pytest.skip("no CUDA headers")
    src, exe = tmp_path / "opt_in.cpp", tmp_path / "opt_in"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-I", CUDA, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout + r.stderr


def test_every_launch_site_uses_it():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h")):
        if os.path.basename(path) != "smem_opt_in.h":
            assert "cudaFuncSetAttribute" not in open(path).read(), path
