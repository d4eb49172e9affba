"""The integer forms in the streaming of FP64 records (host build of the device header): the fixed-point
conversion of the exact moment sums and the cell floor of the transport equal the floating-point ones."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2305_12071_gb300", "csrc")


def test_fp64_stream_integer_forms(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "fp64_stream_check")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off", "-I", CSRC,
                    os.path.join(HERE, "fp64_stream_check.cu"), "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe, "1000000"], capture_output=True, text=True)
    tot, bad = map(int, r.stdout.split()[-2:])
    assert r.returncode == 0 and bad == 0 and tot > 5000000, r.stdout
