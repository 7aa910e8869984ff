"""The Arnoldi step's cluster of sixteen CTAs, a size that not every device (or slice of one) can place: short
vectors of the classical form take it only where one fits, and the grid form otherwise.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA_INC = "/usr/local/cuda/include"


def test_cluster_only_where_one_fits(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None or not os.path.isdir(CUDA_INC):
        pytest.skip("needs a C++ compiler and the CUDA headers")
    exe = str(tmp_path / "form")
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_2410_06319_gb300", "csrc"), "-I", CUDA_INC,
                    os.path.join(ROOT, "tests", "native", "arnoldi_form_harness.cpp"), "-o", exe], check=True)
    cases = [(n, gs, ex, c) for n in (2, 1100, 2048, 2049, 10**6) for gs in (0, 1, 2) for ex in (0, 1) for c in (0, 1, 9)]
    out = subprocess.run([exe], input="\n".join("%d %d %d %d" % c for c in cases), capture_output=True, text=True,
                         check=True).stdout.split()
    assert [int(v) for v in out] == [int(n <= 2048 and gs == 0 and ex == 0 and c > 0) for n, gs, ex, c in cases]
