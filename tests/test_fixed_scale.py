"""The exponent arithmetic of the fixed-point sums' way back to FP64
(csrc/fixed.cuh, fx_high), compiled for the host with the signed-overflow
sanitizer: equal to ldexp over the whole range of fields and sums, of either
sign, without a signed overflow."""
import os
import subprocess

import pytest

from paper_1102_2143_gb300 import build

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include "fixed.cuh"
int main() {
    for (unsigned e = 160; e <= 2000; ++e)
        for (int k = 0; k < 63; ++k)
            for (int half = 0; half < 2; ++half)
                for (int sign = -1; sign < 2; sign += 2) {
                    const double t = sign * (double)((1ll << k) + (k > 3 ? 5 : 0));
                    const double want = std::ldexp(t, (int)e - 1078 - half);
                    if (!std::isnormal(want)) continue;
                    unsigned long long w;
                    memcpy(&w, &t, 8);
                    const unsigned hi = (unsigned)msc::fx_high((int)(w >> 32), e << 20, half);
                    w = (unsigned long long)hi << 32 | (w & 0xffffffffull);
                    double got;
                    memcpy(&got, &w, 8);
                    if (got != want) { printf("%u %d %d: %a %a\n", e, k, half, got, want); return 1; }
                }
    return 0;
}
"""


def test_scaling_back_has_no_signed_overflow(tmp_path):
    src, exe = tmp_path / "scale.cu", tmp_path / "scale"
    src.write_text(SOURCE)
    cmd = [build.nvcc()] + build.ARCH + ["-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, "-I",
                                         os.path.join(build.ROOT, "include"), str(src), "-o", str(exe)]
    for f in ("-fsanitize=signed-integer-overflow", "-fno-sanitize-recover=all"):
        cmd += ["-Xcompiler", f]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if "ubsan" in res.stderr:
        pytest.skip("no sanitizer library")
    assert res.returncode == 0, res.stderr
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout + run.stderr
