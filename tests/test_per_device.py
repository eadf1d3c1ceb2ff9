"""Device properties are kept per device (csrc/per_device.h).  No GPU.

A host program with a fake cudaGetDevice: every device gets a value of its own,
once; a value that could not be had (zero, false) is asked for again.  And no
source file keeps what it asked the runtime in a function's static, which
would be the first device's for the whole process.
"""
import glob
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1111_0125_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include "per_device.h"
static int device = 0, asked = 0, ready = 1;
extern "C" cudaError_t __wrap_cudaGetDevice(int *d) { *d = device; return cudaSuccess; }
static int width() { return stg::per_device([] { ++asked; return ready ? 10 + device : 0; }); }
static int other() { return stg::per_device([] { return 7; }); }
int main(void)
{
    int bad = 0;
    for (int turn = 0; turn < 2; ++turn)
        for (device = 0; device < 4; ++device) bad += width() != 10 + device || other() != 7;
    bad += asked != 4;
    ready = 0;
    device = 5;
    bad += width() != 0 || width() != 0 || asked != 6;
    ready = 1;
    bad += width() != 15 || width() != 15 || asked != 7;
    device = 1000;  // beyond the table: asked every time
    bad += width() != 1010 || width() != 1010 || asked != 9;
    return bad;
}
"""


def test_a_value_per_device(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    src = tmp_path / "per_device_check.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "per_device_check"
    subprocess.run([nvcc, "-O1", "-std=c++17", "-I", CSRC, "-Xlinker", "--wrap=cudaGetDevice", str(src), "-o", str(exe)],
                   check=True, capture_output=True)
    assert subprocess.run([str(exe)], timeout=60).returncode == 0


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_no_static_from_the_runtime(path):
    text = open(path).read()
    assert not re.search(r"static const [\w:<>, ]+ \w+ = \[", text)
