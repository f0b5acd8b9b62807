"""Quotients formed without a division (csrc/pr_internal.cuh), compiled for the
host and compared with the IEEE division bit for bit: pixel centres in FP32 and
FP64 for every index of every size up to 16384 (134 M each), and r / sqrt(2) in
FP64 for 20 M radii over twelve binades."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include <cstring>
#include "pr_internal.cuh"
int main()
{
    long long n = 0, bad32 = 0, bad64 = 0, bad_r = 0;
    for (int W = 1; W <= 16384; ++W) {
        const float rW = 1.f / (float)W;
        for (int i = 0; i < W; ++i, ++n) {
            const volatile float b = (float)W;
            const volatile double d = (double)W;
            const float a = (float)i + 0.5f;
            bad32 += pr::pixel_centre(i, W, rW) != a / b;
            bad64 += pr::quotient64((double)a, (double)W, (double)rW) != (double)a / d;
        }
    }
    unsigned long long s = 88172645463325252ull;
    for (int k = 0; k < 20000000; ++k) {
        s ^= s << 13, s ^= s >> 7, s ^= s << 17;
        const unsigned long long bits = ((1023ull - k % 12) << 52) | (s >> 12);  // [2^-11, 2)
        double r;
        std::memcpy(&r, &bits, 8);
        const volatile double D = 1.4142135623730950488;
        bad_r += pr::over_sqrt2(r) != r / D;
    }
    std::printf("%lld %lld %lld %lld\n", n, bad32, bad64, bad_r);
    return 0;
}
"""


def test_every_pixel_centre_and_radius(tmp_path):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = nvcc if os.path.exists(nvcc) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "quotients.cu", tmp_path / "quotients"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_1806_05385_gb300", "csrc"), "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert [int(x) for x in out] == [16384 * 16385 // 2, 0, 0, 0]
