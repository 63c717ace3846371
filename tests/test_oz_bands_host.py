"""The split-precision GEMM's work order in bands (csrc/oz_order.cuh, compiled on
the host), and that no kernel uses cluster multicast: the library also runs as
one process per GPU on several GPUs."""
import glob
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2605_21149_gb300", "csrc")


def test_split_gemm_bands(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    exe = tmp_path / "oz_band_check"
    subprocess.run([cxx, "-O2", "-std=c++17",
                    f'-DOZ_ORDER_HEADER="{os.path.join(CSRC, "oz_order.cuh")}"',
                    os.path.join(HERE, "host", "oz_band_check.cpp"), "-o", str(exe)],
                   check=True, capture_output=True, text=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "OK", r.stdout


def test_no_cluster_multicast():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        with open(path) as f:
            assert "multicast::cluster" not in f.read(), path
