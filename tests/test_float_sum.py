"""The three-float running sum of the Macro-F1 Hessian, checked on the host against exact
integer sums: no further off than FP64 additions (tests/cpp/float_sum_check.cpp)."""
import shutil
import subprocess
from pathlib import Path

import pytest

ROOT = Path(__file__).resolve().parent.parent


def test_three_float_sums_are_as_good_as_fp64(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    exe = tmp_path / "float_sum_check"
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-I", str(ROOT / "paper_2302_07084_gb300" / "csrc"),
                    str(ROOT / "tests" / "cpp" / "float_sum_check.cpp"), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout.strip().endswith("ok"), out.stdout
