"""Kernel attributes are set on every device that a process uses, once each, and again after a failure
(`once_per_device`, csrc/prrtc_launch.h); and no launch of the dense products keeps a flag that leaves the
device out."""
import os
import re
import subprocess

from paper_2503_06757_gb300 import build as B

PROGRAM = r'''
#include <cstdio>
#include "prrtc_launch.h"
using namespace prrtc;

int main() {
  std::atomic<uint64_t> a{0}, b{0};
  int runs = 0;
  cudaError_t next = cudaSuccess;
  auto set = [&] { ++runs; return next; };
  auto call = [&](std::atomic<uint64_t>& w, int dev) {
    const int before = runs;
    const cudaError_t e = once_per_device(w, dev, set);
    printf("%d%d ", runs - before, (int)(e != cudaSuccess));
  };
  for (int dev : {0, 0, 1, 63, 1, 0, 63, 64, 64, -1}) call(a, dev);  // 64, -1: not kept
  call(b, 0);                                                        // another kernel
  next = cudaErrorInvalidValue;
  call(b, 5);
  next = cudaSuccess;
  call(b, 5);
  call(b, 5);
  return 0;
}
'''


def test_once_per_device(tmp_path):
    src, exe = str(tmp_path / "once.cu"), str(tmp_path / "once")
    with open(src, "w") as f:
        f.write(PROGRAM)
    cmd = [B.nvcc()] + B.ARCH + ["-std=c++17", "--expt-relaxed-constexpr", "-I", B.CSRC, "-I", B.INCLUDE, src, "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()
    assert out == "10 00 10 10 00 00 00 10 10 10 10 11 10 00".split()


def test_products_keep_no_flag_without_its_device():
    text = open(os.path.join(B.CSRC, "prrtc_gemm.cu")).read()
    assert not re.findall(r"static\s+(?:const\s+)?(?:bool|int)\s+\w+\s*=", text)
