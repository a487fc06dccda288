"""What kernels with bounded waits do after a wait has run out: small programs against the
library's internals (tests/cpp), built here, that set the status words from the host.
Nothing in them faults or waits for something that does not come for long."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

CPP = os.path.join(os.path.dirname(os.path.abspath(__file__)), "cpp")


def _run(tmp_path, name):
    from paper_2302_07084_gb300 import build
    lib = build.build()
    exe = str(tmp_path / name)
    subprocess.run([build.nvcc(), *build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, "-I",
                    build.INCLUDE, os.path.join(CPP, name + ".cu"), "-L", os.path.dirname(lib), "-llne", "-Xlinker",
                    "-rpath=" + os.path.dirname(lib), "-o", exe], check=True, capture_output=True, text=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr


def test_sort_after_an_expired_wait_writes_nothing(tmp_path):
    _run(tmp_path, "sort_after_timeout")


def test_late_cta_leaves_a_given_up_barrier(tmp_path):
    _run(tmp_path, "grid_barrier_late")
