"""The FP64 closed form's own square root, logarithm and angle (csrc/fp64.cuh)
and the FP32 pass's angle (csrc/quad32.cuh) against a long double host reference, within the bounds derived beside their
check (gpu_fp64_check.cu): random arguments of every sign, 120 binades of
range, ratios near 1, both sides of the tables' breakpoints, zeros."""
import os
import shutil
import subprocess
import tempfile

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def worst():
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    with tempfile.TemporaryDirectory() as d:
        exe = os.path.join(d, "fp64")
        subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                        "-I", os.path.join(ROOT, "paper_2410_15227_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "gpu_fp64_check.cu"), "-o", exe], check=True)
        out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=120).stdout
    return {p[0]: (float(p[1]), int(p[2])) for p in (line.split() for line in out.strip().splitlines())}


@pytest.mark.parametrize("name", ["sqrt64", "log_ratio", "angle64", "angle_q1"])
def test_within_bound(worst, name):
    w, n = worst[name]
    assert n > 500_000 and w <= 1.0, w
