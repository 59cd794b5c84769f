"""Host-side planning that needs no device: the rounds that the final reduction
sums with a warp each in a merge of more rounds than one launch has warps."""
import os
import shutil
import subprocess

import pytest

from paper_1202_1350_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_rounds_with_many_partials_get_a_warp(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    libdir = os.path.dirname(build.build())
    exe = str(tmp_path / "plan_rounds")
    subprocess.run([nvcc, *build.ARCH, "-std=c++17", "-I", build.CSRC, "-I", build.INCLUDE, "-cudart", "shared",
                    os.path.join(ROOT, "tests", "c", "plan_rounds.cu"), "-L", libdir, "-lvc",
                    "-Xlinker", f"-rpath,{libdir}", "-o", exe], check=True)
    n = 152 * 8 * 8 + 5000  # more than any device's warps of one launch
    out = subprocess.run([exe, str(n)], check=True, capture_output=True, text=True).stdout.splitlines()
    nbig, rounds = map(int, out[0].split())
    left = [tuple(map(int, line.split())) for line in out[1:]]
    assert rounds == n and len(left) == n - nbig
    partials = [(1 + k % 5, 0 if k % 3 else k % 41) for k in range(n)]
    assert left == [p for p in partials if max(p) <= 2]
