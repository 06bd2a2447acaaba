"""A cluster size that the device refuses is answered with 0 clusters and leaves no CUDA error behind.

The launch header is compiled into a small program, which asks for more shared memory than any SM has; the
attribute call refuses that on the host.  A later check of the last error must find none, or the solve that
falls back to the step-by-step path would fail on it (GPU: without one, every call reports that error).
"""

import os
import shutil
import subprocess

import pytest

from paper_1012_5168_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cstdio>
#include "resident_launch.cuh"
static __global__ void nothing() {}
int main() {
    const int n = dl::resident_max_clusters(nothing, (size_t)1 << 30, 1);
    printf("%d %d\n", n, (int)cudaGetLastError());
    return 0;
}
"""


def test_refused_opt_in_leaves_no_error(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = tmp_path / "opt_in.cu", tmp_path / "opt_in"
    src.write_text(SOURCE)
    subprocess.run([nvcc, *build.ARCH, *build.FLAGS, "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=120).stdout
    assert out.split() == ["0", "0"]
