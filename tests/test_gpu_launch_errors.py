"""A launch that the runtime refuses reports its error once, by its return
value: nothing stays pending on the thread for a later call to meet.  A small
program around the library's two launch helpers asks for blocks of 4096
threads, which the runtime turns down on the host."""
import subprocess

import pytest

from paper_1704_01888_gb300 import build

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include "pa_cluster.cuh"

__global__ void k_nothing(int) {}

int main()
{
    int bad = 0;
    (void)cudaGetLastError();
    if (pa::launch_after(k_nothing, 1, 1, 4096, 0, nullptr, 0) == cudaSuccess) bad |= 1;
    if (cudaPeekAtLastError() != cudaSuccess) bad |= 2;
    (void)cudaGetLastError();
    if (pa::launch_clusters(k_nothing, 2, 2, 4096, 0, nullptr, 0) == cudaSuccess) bad |= 4;
    if (cudaPeekAtLastError() != cudaSuccess) bad |= 8;
    std::printf("%d\n", bad);
    return 0;
}
"""


def test_refused_launch_leaves_no_error_pending(tmp_path):
    src, exe = tmp_path / "launch.cu", tmp_path / "launch"
    src.write_text(PROGRAM)
    subprocess.run([build._nvcc(), *build.ARCH, "-std=c++17", "-I", build.CSRC, "-o", str(exe), str(src)], check=True,
                   timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout.strip() == "0", r.stdout + r.stderr
