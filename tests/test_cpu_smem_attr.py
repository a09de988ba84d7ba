"""Shared-memory attributes per device and thread (csrc/smem_attr.h), against a fake of the
two CUDA calls it makes: a host program in which device 0 and device 1 each have to have
the attribute set before a launch there, sizes that grow and shrink, a failure that is not
remembered, and threads that ask for different sizes at once."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1711_10214_gb300", "csrc")

PROGRAM = r"""
#include "smem_attr.h"
#include <cstdio>
#include <cstdlib>
#include <thread>
#include <vector>
static thread_local int device = 0;
static std::atomic<int> attribute[32];   // what a device allows
static std::atomic<int> calls;
static bool fail = false;
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int n) {
  ++calls;
  if (fail) return cudaErrorInvalidValue;
  attribute[device] = n;
  return cudaSuccess;
}
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); std::exit(1); } } while (0)
static void kernel() {}
// a launch of n bytes on a device
static bool launch(ashrt::SmemAttr& a, int dev, size_t n) {
  device = dev;
  return ashrt::set_smem(kernel, n, a) == cudaSuccess && (n <= 40 * 1024 || attribute[dev] >= (int)n);
}
int main() {
  {
    ashrt::SmemAttr a;
    CHECK(launch(a, 0, 32 * 1024) && calls == 0);
    CHECK(launch(a, 0, 100 * 1024) && calls == 1);
    CHECK(launch(a, 0, 100 * 1024) && calls == 1);
    CHECK(launch(a, 1, 100 * 1024) && calls == 2);      // the second device has its own
    CHECK(launch(a, 1, 200 * 1024) && launch(a, 1, 100 * 1024) && launch(a, 1, 200 * 1024));
    CHECK(calls == 3);
    CHECK(launch(a, 0, 150 * 1024) && calls == 4);
    CHECK(launch(a, 20, 100 * 1024) && launch(a, 20, 100 * 1024) && calls == 6);   // past the table
    fail = true;
    CHECK(!launch(a, 2, 64 * 1024));
    fail = false;
    CHECK(launch(a, 2, 64 * 1024));                      // not remembered as set
  }
  for (int rep = 0; rep < 50; ++rep) {
    ashrt::SmemAttr a;
    for (auto& x : attribute) x = 0;
    std::vector<std::thread> t;
    std::atomic<int> bad{0};
    for (int i = 0; i < 8; ++i)
      t.emplace_back([&, i] {
        for (int k = 0; k < 200; ++k)
          if (!launch(a, i & 1, (size_t)(50 + (i * 37 + k * 11) % 150) * 1024)) ++bad;
      });
    for (auto& x : t) x.join();
    CHECK(bad == 0);
  }
  return 0;
}
"""


def test_attribute_is_kept_per_device(tmp_path):
    cxx = shutil.which("g++")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not cxx or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("no host compiler or CUDA headers")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, "-I", inc, str(src), "-o",
                    str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0, res.stdout


def test_every_kernel_uses_it():
    """No per-process flag beside it: the attribute call stands in smem_attr.h and, for the
    widest heads, where it is made on every call."""
    found = []
    for f in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, f)).read()
        assert "static bool attr" not in text and "static size_t attr" not in text, f
        found += [f] * text.count("cudaFuncSetAttribute(")
    assert found == ["smem_attr.h", "unet.cu"]
