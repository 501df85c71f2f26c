"""The limit of dynamic shared memory is raised on every device that launches a kernel
(host code, against a CUDA runtime of two functions)."""
import os
import shutil
import subprocess

import pytest

from paper_2511_07809_gb300 import _build

SRC = r"""
#include <cstdio>
#include <set>
#include <utility>
#include "smem_limit.h"
static int device = 0, fails = 0, calls = 0;
static std::set<std::pair<int, const void *>> raised;
extern "C" cudaError_t cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void *f, cudaFuncAttribute a, int v) {
  ++calls;
  if (fails) return cudaErrorInvalidValue;
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize && v == 100000) raised.insert({device, f});
  return cudaSuccess;
}
static int kernel;
int main() {
  static tlda::SmemLimit lim;
  fails = 1;
  if (lim.raise(&kernel, 100000) != cudaErrorInvalidValue) return 1;
  fails = 0;  // a failure is not taken for done
  for (int round = 0; round < 3; ++round)
    for (int d : {0, 1, 5, 63, 64, 200}) {
      device = d;
      if (lim.raise(&kernel, 100000) != cudaSuccess || !raised.count({d, &kernel})) return 2;
    }
  // once on each device of the mask, each time past it
  return calls == 1 + 4 + 2 * 3 ? 0 : 3;
}
"""


def test_raised_once_on_each_device(tmp_path):
    nvcc = shutil.which(_build.NVCC)
    if not nvcc:
        pytest.skip("no CUDA headers")
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    (tmp_path / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-std=c++17", "-I", inc, "-I", _build.CSRC, str(tmp_path / "t.cpp"), "-o", str(tmp_path / "t")],
                   check=True)
    assert subprocess.run([str(tmp_path / "t")]).returncode == 0


def test_no_kernel_sets_its_limit_once_a_process():
    for src in _build.sources() + [os.path.join(_build.CSRC, "gemm64.cuh")]:
        for line in open(src):
            assert "cudaFuncSetAttribute" not in line or "k_pass" in line, (src, line)  # k_pass: set when a context is made
