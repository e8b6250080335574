"""Kernel attributes belong to a device: a launcher that asked for more than 48 KB
of dynamic shared memory once a process would fail on the second device a
program uses, and return a first error for ever.  So no launcher keeps the
answer in a static of its own, and the helper that remembers it does so for each
device and never an error (run here against stand-ins of the two runtime
calls)."""

import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1710_03013_gb300", "csrc")


def test_no_launcher_sets_a_kernel_attribute_once_a_process():
    calls = 0
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        for m in re.finditer(r"cudaFuncSetAttribute|smem_opt_in\(", text):
            calls += 1
            statement = re.split(r"[;{}]", text[:m.start()])[-1]
            assert not re.search(r"\bstatic\b|call_once", statement), (name, statement.strip())
    assert calls >= 10


PROGRAM = r"""
#include "smem_opt_in.h"
#include <cassert>
#include <initializer_list>
static int device = 0, asked = 0;
static cudaError_t answer = cudaSuccess;
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { ++asked; return answer; }
int main() {
  std::atomic<uint64_t> done{0};
  auto ask = [&]() { return kkm::smem_opt_in(done, &done, 100000); };
  answer = cudaErrorInvalidValue;
  assert(ask() == cudaErrorInvalidValue && asked == 1);
  answer = cudaSuccess;
  assert(ask() == cudaSuccess && asked == 2);  // an error is not kept
  assert(ask() == cudaSuccess && asked == 2);
  for (int d : {1, 63, 64, 64, 1, 63, 0}) {
    device = d;
    assert(ask() == cudaSuccess);
  }
  assert(asked == 6);  // once for 1 and 63, every time for 64
  return 0;
}
"""


def test_the_helper_remembers_for_each_device(tmp_path):
    cuda = next((d for d in ("/usr/local/cuda/include",) if os.path.exists(os.path.join(d, "cuda_runtime_api.h"))), None)
    if not shutil.which("g++") or not cuda:
        pytest.skip("needs g++ and the CUDA headers")
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, "-I", cuda, str(src), "-o", exe], check=True)
    subprocess.run([exe], check=True)
