"""The split-precision GEMM's drain schedule (csrc/oz_sched.cuh) and its
80-bit, branch-free float64 output conversion (csrc/fixconv.cuh), compiled on
the host with g++."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2605_21149_gb300", "csrc")


@pytest.mark.parametrize("prog,macro,header", [
    ("oz_sched_check.cpp", "OZ_SCHED_HEADER", "oz_sched.cuh"),
    ("fixfrac_check.cpp", "FIXCONV_HEADER", "fixconv.cuh")])
def test_host_check(tmp_path, prog, macro, header):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = tmp_path / "check"
    subprocess.run([cxx, "-O2", "-std=c++17", f'-D{macro}="{os.path.join(CSRC, header)}"',
                    os.path.join(HERE, "host", prog), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip().endswith("OK"), r.stdout
