"""What the library keeps per device (csrc/dc_device.h), compiled for the host
against a fake of the two runtime calls it makes: a kernel's shared memory limit
is raised once on every device it is launched on, a failure is reported and
tried again, threads on different devices each find it raised, and what was
asked of one device never answers for another, whatever its ordinal. No launcher
keeps such a state of its own beside it."""

import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_08878_gb300", "csrc")

FAKE = """
#pragma once
typedef int cudaError_t;
enum { cudaSuccess = 0, cudaErrorInvalidDevice = 101, cudaFuncAttributeMaxDynamicSharedMemorySize = 8 };
cudaError_t cudaGetDevice(int* dev);
cudaError_t cudaFuncSetAttribute(const void* f, int attr, int value);
template <class T> cudaError_t cudaFuncSetAttribute(T* f, int attr, int value) {
  return cudaFuncSetAttribute((const void*)f, attr, value);
}
"""

PROGRAM = """
#include "dc_device.h"
#include <cstdio>
#include <cstdlib>
#include <thread>
#include <vector>
thread_local int t_dev = 0;
int g_fail = 0;
std::atomic<int> g_calls[200];
cudaError_t cudaGetDevice(int* d) { if (t_dev < 0) return cudaErrorInvalidDevice; *d = t_dev; return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, int, int) {
  ++g_calls[t_dev < 0 ? 199 : t_dev];
  return g_fail;
}
void kernel() {}
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\\n", __LINE__, #x); std::exit(1); } } while (0)
int main() {
  static dc::SmemLimit limit;
  for (int dev : {0, 1, 0, 1, 63}) { t_dev = dev; CHECK(limit.raise(kernel, 1000) == 0); }
  CHECK(g_calls[0] == 1 && g_calls[1] == 1 && g_calls[63] == 1);
  for (int dev : {64, 64, 70, -1}) { t_dev = dev; CHECK(limit.raise(kernel, 1000) == 0); }
  CHECK(g_calls[64] == 2 && g_calls[70] == 1 && g_calls[199] == 1 && g_calls[0] == 1);
  t_dev = 2; g_fail = 7;
  CHECK(limit.raise(kernel, 1000) == 7);
  g_fail = 0;
  CHECK(limit.raise(kernel, 1000) == 0 && limit.raise(kernel, 1000) == 0 && g_calls[2] == 2);

  static dc::PerDevice<int> kept;
  int asked = 0;
  auto ask = [&] { ++asked; return 10 + t_dev; };
  for (int dev : {0, 1, 0, 1}) { t_dev = dev; CHECK(kept.get(ask) == 10 + dev); }
  CHECK(asked == 2);
  for (int dev : {64, 65, 64, -1}) { t_dev = dev; CHECK(kept.get(ask) == 10 + dev); }
  CHECK(asked == 6);

  static dc::SmemLimit shared;
  std::atomic<int> bad{0};
  std::vector<std::thread> ts;
  for (int i = 0; i < 16; ++i) ts.emplace_back([&, i] {
    t_dev = 100 - 90 * (i % 2) + i / 2;  // 100 .. 107 are never kept, 10 .. 17 are
    for (int n = 0; n < 1000; ++n) {
      if (shared.raise(kernel, 1) != 0 || g_calls[t_dev] < 1) ++bad;
    }
  });
  for (auto& t : ts) t.join();
  CHECK(bad == 0);
  for (int i = 0; i < 8; ++i) CHECK(g_calls[10 + i] == 1 && g_calls[100 + i] == 1000);
  return 0;
}
"""


def test_each_device_has_its_own_answers(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "cuda_runtime.h").write_text(FAKE)
    (tmp_path / "main.cpp").write_text(PROGRAM)
    exe = tmp_path / "main"
    subprocess.run([cxx, "-std=c++17", "-Wall", "-pthread", "-I", str(tmp_path), "-I", CSRC, str(tmp_path / "main.cpp"),
                    "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0, res.stdout


def test_no_launcher_keeps_a_flag_for_the_whole_process():
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        assert not re.search(r"static\s+(bool\s+\w+\s*[={;]|std::once_flag\b)", text), name
