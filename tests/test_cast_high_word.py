"""The cast's rounding on the high word of an FP64 value (csrc/cast.cuh: cast_hi) equals the
general integer rounding bit for bit wherever it takes a value, and takes every value in the
format's normal range: ties, ties broken by the low word, carries and the range's edges at
every power-of-two scaling."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_high_word_rounding_equals_the_general_rounding(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = str(tmp_path / "cast_hi")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "paper_2410_06319_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "native", "cast_hi_harness.cpp"), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split()
    rows = [out[i:i + 4] for i in range(0, len(out), 4)]
    assert [r[0] for r in rows] == ["bf16", "f16", "e4m3"]
    for fmt, taken, declined, bad in rows:
        assert int(taken) > 100_000 and int(declined) > 100_000 and int(bad) == 0, (fmt, taken, declined, bad)
