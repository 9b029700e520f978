"""Shared-memory limits of the kernels are raised once for every device a
process uses, not once for the process (no GPU: the runtime's calls are
replaced by counters that pretend to have several devices).
"""
import subprocess

import pytest

from paper_0911_1407_gb300 import build

MAIN = r"""
#include <cstdio>
#include <cuda_runtime.h>
static int g_dev = 0, g_calls[80] = {}, g_fail = 0;
static cudaError_t fake_device(int* d) { *d = g_dev; return cudaSuccess; }
template <typename F> static cudaError_t fake_attribute(F*, cudaFuncAttribute, int) {
  ++g_calls[g_dev];
  return g_fail ? cudaErrorInvalidValue : cudaSuccess;
}
#define cudaGetDevice fake_device
#define cudaFuncSetAttribute fake_attribute
#include "limits.cuh"

void plc::check(cudaError_t e, const char* where) {
  if (e != cudaSuccess) throw plc::CudaError{e, where};
}

static __global__ void k_a() {}
static __global__ void k_b() {}

int main() {
  for (int round = 0; round < 2; ++round)
    for (int d : {0, 1, 0, 63, 64, 64}) {
      g_dev = d;
      plc::set_smem4<k_a>(plc::current_device(), 60 * 1024);
    }
  g_dev = 1;
  plc::set_smem4<k_b>(plc::current_device(), 1024);
  std::printf("%d %d %d %d\n", g_calls[0], g_calls[1], g_calls[63], g_calls[64]);
  // a call that failed is made again
  g_dev = 5;
  g_fail = 1;
  bool thrown = false;
  try {
    plc::set_smem4<k_b>(plc::current_device(), 1024);
  } catch (const plc::CudaError&) {
    thrown = true;
  }
  g_fail = 0;
  plc::set_smem4<k_b>(plc::current_device(), 1024);
  std::printf("%d %d\n", (int)thrown, g_calls[5]);
}
"""


@pytest.fixture(scope="module")
def lines(tmp_path_factory):
    tmp = tmp_path_factory.mktemp("limits")
    src, exe = tmp / "limits.cu", tmp / "limits"
    src.write_text(MAIN)
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, str(src), "-o",
                    str(exe)], check=True, capture_output=True, timeout=600)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout
    return [[int(v) for v in line.split()] for line in out.splitlines()]


def test_once_for_each_device_and_kernel(lines):
    # devices past those that are remembered are set on every call
    assert lines[0] == [1, 2, 1, 4]


def test_a_failure_is_reported_and_not_remembered(lines):
    assert lines[1] == [1, 2]
