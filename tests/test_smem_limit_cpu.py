"""The shared-memory limit of a kernel (csrc/smem_limit.h) against a stand-in for the two runtime calls: it is
raised once per device, never lowered, tried again after an error, and right under several threads.
Every launcher takes this route."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1411_6206_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <map>
#include <thread>
#include <vector>
#include "smem_limit.h"
static thread_local int device = 0;
static std::map<int, int> limit;   // dynamic shared memory that the kernel may ask for, per device
static int calls = 0;
static bool fail = false;
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, enum cudaFuncAttribute, int v) {
  ++calls;
  if (fail) return cudaErrorInvalidValue;
  limit[device] = v;
  return cudaSuccess;
}
#define CHECK(c) do { if (!(c)) { printf("line %d: " #c "\n", __LINE__); return 1; } } while (0)
int main() {
  static lps::SmemLimit l;
  CHECK(l.raise(nullptr, 48 * 1024) == cudaSuccess && calls == 0);
  CHECK(l.raise(nullptr, 100000) == cudaSuccess && limit[0] == 100000 && calls == 1);
  CHECK(l.raise(nullptr, 60000) == cudaSuccess && limit[0] == 100000 && calls == 1);   // not lowered
  for (int d : {1, 63, 64, 200}) {
    device = d;
    CHECK(l.raise(nullptr, 100000) == cudaSuccess && limit[d] == 100000);              // each device has its own
  }
  device = 2;
  fail = true;
  CHECK(l.raise(nullptr, 100000) == cudaErrorInvalidValue);
  fail = false;
  CHECK(l.raise(nullptr, 100000) == cudaSuccess && limit[2] == 100000);
  std::vector<std::thread> t;
  for (int i = 0; i < 8; ++i)
    t.emplace_back([i] {
      device = 3;
      for (int b = 0; b < 200; ++b) l.raise(nullptr, 50000 + 100 * ((b * 7 + i * 31) % 200));
    });
  for (auto& x : t) x.join();
  CHECK(limit[3] == 50000 + 100 * 199);
  return 0;
}
"""


def test_limit_per_device(tmp_path):
    cxx = shutil.which("g++")
    inc = next((p for p in (os.environ.get("CUDA_HOME", ""), "/usr/local/cuda")
                if p and os.path.exists(os.path.join(p, "include", "cuda_runtime_api.h"))), None)
    if not cxx or not inc:
        pytest.skip("needs g++ and the CUDA headers")
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", f"-I{CSRC}", f"-I{inc}/include", str(src), "-o",
                        str(tmp_path / "t")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(tmp_path / "t")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_every_launcher_takes_it():
    for f in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, f)) as fh:
            s = re.sub(r"//[^\n]*", "", fh.read())
        if f != "smem_limit.h":
            assert "cudaFuncSetAttribute" not in s, f
