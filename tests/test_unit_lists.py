"""Host-side check of the unit lists' cost arithmetic (no GPU), up to the largest number of units they take."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_cost_line_up_to_the_most_units(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc) and shutil.which("nvcc") is None:
        pytest.skip("nvcc not available")
    exe = tmp_path / "costline_check"
    inc = os.path.join(ROOT, "paper_2511_11430_gb300", "csrc")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2", "-I" + inc,
                    "-I" + os.path.join(ROOT, "include"), os.path.join(ROOT, "tests", "host", "costline_check.cu"),
                    "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.startswith("OK"), out.stdout + out.stderr
