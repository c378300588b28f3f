"""Host logic of the one-cluster kernels (no GPU): where no cluster of 16 or 8 CTAs can be
placed, or its launch is refused, the caller is told, so that the general form runs.  A small
program calls the library's helpers in a process that sees no CUDA device: every CUDA
call fails there."""
import os
import shutil
import subprocess

import pytest

from paper_1408_5535_gb300 import build

PROGRAM = r"""
#include <cstdio>
#include "cluster.cuh"
namespace ph { void count_launch() { std::puts("counted"); } }
struct Args { int x; };
__global__ void kernel(Args a) { if (a.x) __syncthreads(); }
int main() {
  static std::atomic<int> known[64];
  const int first = ph::cluster_size(kernel, 128, 1024, 1024, known);
  const int again = ph::cluster_size(kernel, 128, 1024, 1024, known);
  const bool ok = ph::launch_cluster(kernel, 8, 128, 1024, nullptr, Args{0});
  std::printf("%d %d %d\n", first, again, (int)ok);
}
"""


def test_a_cluster_that_cannot_be_launched_is_reported(tmp_path):
    nvcc = build.NVCC if os.path.exists(build.NVCC) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "cluster_host.cu", tmp_path / "cluster_host"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, *[f for f in build.FLAGS if f != "-O3"], str(src), "-o", str(exe)], check=True, timeout=600)
    out = subprocess.run([str(exe)], env={**os.environ, "CUDA_VISIBLE_DEVICES": ""}, capture_output=True, text=True,
                         timeout=60, check=True).stdout
    assert out.split() == ["0", "0", "0"], out
