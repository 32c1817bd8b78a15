"""The opt-in to large dynamic shared memory, against a fake of the runtime's two calls: every device gets
its own, and threads that launch at the same time never leave one with less than it asked for."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <cstdio>
#include <map>
#include <mutex>
#include <thread>
#include <utility>
#include <vector>
#include "msf_smem.h"

static thread_local int t_dev = 0;
static std::mutex g_m;
static std::map<std::pair<const void*, int>, int> g_attr;  // (function, device) -> bytes
static int g_calls = 0, g_lowered = 0, g_fail = 0;

extern "C" cudaError_t cudaGetDevice(int* d) { *d = t_dev; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
  std::lock_guard<std::mutex> l(g_m);
  if (g_fail) { --g_fail; return cudaErrorInvalidValue; }
  int& a = g_attr[{f, t_dev}];
  if (v < a) ++g_lowered;
  a = v;
  ++g_calls;
  return cudaSuccess;
}

static void kernel_a(int) {}
static void kernel_b(int) {}

#define CHECK(x) do { if (!(x)) { std::printf("%s\n", #x); return 1; } } while (0)

int main() {
  std::atomic<uint64_t> a{0}, b{0};
  for (int d : {0, 1, 3, 0, 1}) {  // a second device is not skipped for the first
    t_dev = d;
    msf::ensure_smem_attr(kernel_a, 80000, a);
    CHECK((g_attr[{(const void*)kernel_a, d}] == 80000));
  }
  CHECK(g_calls == 3);             // and a repeated one is not set again
  t_dev = 5;
  g_fail = 1;                      // a failed one is tried again
  msf::ensure_smem_attr(kernel_a, 80000, a);
  msf::ensure_smem_attr(kernel_a, 80000, a);
  CHECK((g_attr[{(const void*)kernel_a, 5}] == 80000));
  std::vector<std::thread> t;
  for (int i = 0; i < 16; ++i)
    t.emplace_back([&, i] {
      t_dev = i & 3;
      for (int k = 0; k < 1000; ++k) {
        msf::ensure_smem_attr(kernel_b, 200000, b);
        std::lock_guard<std::mutex> l(g_m);
        if (g_attr[{(const void*)kernel_b, t_dev}] != 200000) ++g_lowered;
      }
    });
  for (auto& x : t) x.join();
  CHECK(g_lowered == 0);
  return 0;
}
"""


def test_every_device_and_thread(tmp_path):
    inc = [p for p in ("/usr/local/cuda/include",) if os.path.isdir(p)]
    if not shutil.which("g++") or not inc:
        pytest.skip("no host compiler or CUDA headers")
    src = tmp_path / "t.cpp"
    src.write_text(SOURCE)
    exe = tmp_path / "t"
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", inc[0], "-I",
                    os.path.join(ROOT, "paper_1903_12294_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
