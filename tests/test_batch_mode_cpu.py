"""The mode a tuned batch keeps (host rule, on the CPU): the fastest of the three,
but pass-batched launches instead of a branch graph that is less than a tenth
faster; the persistent kernel only where it is the fastest of all."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
NONE = 1e30  # a mode that is not available

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "batch_mode.h"
int main(int argc, char **argv)
{
    for (int i = 1; i + 2 < argc; i += 3) {
        const double t[3] = {atof(argv[i]), atof(argv[i + 1]), atof(argv[i + 2])};
        printf("%d\n", demag::batch_pick_mode(t));
    }
    return 0;
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("batch_mode")
    (d / "t.cc").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_1204_4302_gb300", "csrc"), str(d / "t.cc"),
                    "-o", str(d / "t")], check=True, capture_output=True, timeout=120)
    return str(d / "t")


@pytest.mark.parametrize("t,mode", [
    ((NONE, 1.0, NONE), 1),       # branches are all there is
    ((1.0, 1.2, 1.1), 0),
    ((1.2, 1.0, 1.05), 2),        # branches less than a tenth faster
    ((1.2, 1.0, 1.2), 1),         # a sixth faster
    ((1.2, 1.3, 1.0), 2),
    ((1.05, 1.0, 1.09), 2),
    ((1.05, 1.0, 1.5), 1),        # not the persistent kernel, which branches beat
])
def test_kept_mode(exe, t, mode):
    out = subprocess.run([exe, *map(str, t)], check=True, capture_output=True, text=True, timeout=60).stdout
    assert int(out) == mode
