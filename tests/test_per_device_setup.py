"""A kernel's one-time settings are made once on every device, and again after a
failure (CPU: the host code of PerDevice, compiled by nvcc)."""
import os
import subprocess

import pytest

from paper_2010_00409_gb300 import build

CSRC = os.path.join(os.path.dirname(build.__file__), "csrc")

SOURCE = r"""
#include <cstdio>
#include "common.cuh"

int main() {
    psatd::PerDevice set;
    int calls[100] = {}, sum = 0;
    auto on = [&](int dev, cudaError_t r = cudaSuccess) {
        return set.once(dev, [&] { ++calls[dev]; return r; });
    };
    for (int dev : {0, 1, 0, 63, 1, 63}) sum += on(dev);
    sum += on(2, cudaErrorInvalidValue) != cudaErrorInvalidValue;
    sum += on(2);
    sum += on(2);
    sum += on(80) + on(80);
    std::printf("%d %d %d %d %d %d\n", sum, calls[0], calls[1], calls[63], calls[2], calls[80]);
}
"""


def test_settings_are_made_once_per_device(tmp_path):
    if not os.path.exists(build.nvcc()):
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "p.cu", tmp_path / "p"
    src.write_text(SOURCE)
    subprocess.run([build.nvcc()] + build.ARCH + ["-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    # (devices beyond the 64 that are remembered are set every time)
    assert out == ["0", "1", "1", "1", "2", "2"]


def test_gemm_launchers_remember_no_device_but_the_one_they_set():
    src = open(os.path.join(CSRC, "gemm.cu")).read()
    assert "static int sms" not in src and "static bool attr" not in src
    assert src.count("static PerDevice set;") == 2


def test_sm_counts_come_from_the_cache():
    """A launch asks the driver for nothing but the current device."""
    src = open(os.path.join(CSRC, "gemm.cu")).read()
    assert "cudaDeviceGetAttribute" not in src and src.count("sm_count(dev, &sms)") == 2
