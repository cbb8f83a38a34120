"""Launch attributes belong to a device (csrc/device_once.h), compiled for the host against a stand-in for the runtime."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUNTIME = r"""
#pragma once
#include <cstddef>
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidValue = 1 };
enum cudaFuncAttribute { cudaFuncAttributeMaxDynamicSharedMemorySize };
enum cudaDeviceAttr { cudaDevAttrMultiProcessorCount };
inline int g_device = 0, g_sets = 0, g_asks = 0;
inline cudaError_t g_next = cudaSuccess;
inline cudaError_t cudaGetDevice(int* d) { *d = g_device; return cudaSuccess; }
template <class F> cudaError_t cudaFuncSetAttribute(F*, cudaFuncAttribute, int) { ++g_sets; return g_next; }
inline cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int dev) { ++g_asks; *v = 100 + dev; return cudaSuccess; }
"""

MAIN = r"""
#include <cstdio>
#include <initializer_list>
#include "device_once.h"
static void one() {}
static void two() {}
#define CHECK(x) do { if (!(x)) { std::printf("%s\n", #x); return 1; } } while (0)
int main() {
  using namespace lrtei;
  for (int dev : {0, 1, 63}) {  // once on each device, whatever came before on another
    g_device = dev;
    const int before = g_sets;
    CHECK(shared_opt_in<&one>(100000) == cudaSuccess && g_sets == before + 1);
    CHECK(shared_opt_in<&one>(100000) == cudaSuccess && g_sets == before + 1);
    int n = 0;
    CHECK(sm_count(&n) == cudaSuccess && n == 100 + dev);
  }
  g_device = 0;
  const int before = g_sets, asks = g_asks;
  g_next = cudaErrorInvalidValue;  // a refusal is returned and not remembered as done
  CHECK(shared_opt_in<&two>(100000) == cudaErrorInvalidValue && g_sets == before + 1);
  g_next = cudaSuccess;
  CHECK(shared_opt_in<&two>(100000) == cudaSuccess && g_sets == before + 2);
  int n = 0;
  CHECK(sm_count(&n) == cudaSuccess && n == 100 && g_asks == asks);
  g_device = 64;
  CHECK(shared_opt_in<&two>(100000) == cudaSuccess && sm_count(&n) == cudaSuccess && n == 164);
  return 0;
}
"""


def test_attributes_are_set_once_per_device(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(MAIN)
    subprocess.run([gxx, "-std=c++17", "-O1", "-I", str(tmp_path), "-I",
                    os.path.join(ROOT, "paper_2210_13069_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_no_launch_remembers_an_attribute_per_process():
    csrc = os.path.join(ROOT, "paper_2210_13069_gb300", "csrc")
    for f in sorted(os.listdir(csrc)):
        if f == "device_once.h":
            continue
        text = open(os.path.join(csrc, f)).read()
        assert "static bool" not in text, f"{f}: state of the process beside a launch"
