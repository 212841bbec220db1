"""Stage plans of the general mixed-radix z passes (the SP z pass, and the tensor
method's where the two-stage kernel does not apply), checked on the CPU: above
length 128, FP32 plans take as few shared-memory stages as radices <= 32 allow, and
no radix above 16 where that saves none; every radix of a plan is one that its
kernel holds; FP64 plans keep to radices <= 16."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "mixed_impl.cuh"
int main()
{
    for (int L = 6; L <= 1000; L += 2) {  // padded lengths are even
        demag::GenRadix g16, g32;
        if (!demag::gen_plan(L, 2048, g32, 32, 3)) continue;
        const bool ok = demag::gen_plan(L, 2048, g16, 16, 3);
        printf("%d %d %d %d %d %d %d\n", L, ok ? g16.n : 99, g32.n, g32.r[g32.n - 1], demag::gen_min_radix(32),
               demag::gen_z_radix<float>(L), demag::gen_z_radix<double>(L));
    }
    return 0;
}
"""


def test_fp32_z_plans_take_the_fewest_stages(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "t.cu"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-O1", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1204_4302_gb300", "csrc"),
                    str(src), "-o", str(tmp_path / "t")], check=True, capture_output=True, timeout=600)
    out = subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True, timeout=60).stdout
    rows = {int(f[0]): tuple(map(int, f[1:])) for f in map(str.split, out.splitlines())}
    assert {96, 200, 270, 300, 486, 600} <= set(rows)
    for L, (n16, n32, least, held, f32, f64) in rows.items():
        assert f32 == (32 if L > 128 and n32 < n16 else 16), L
        assert f32 == 16 or least >= held, L
        assert f64 == 16, L
    assert rows[270][4] == rows[300][4] == 32 and rows[96][4] == rows[120][4] == 16
