"""The split of the tensor-core Gram leaves its integer sums room (``tests/native/gram_room_check.cu``)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_sums_have_room(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = str(tmp_path / "gram_room_check")
    src = os.path.join(ROOT, "tests", "native", "gram_room_check.cu")
    subprocess.run([nvcc, "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_2304_00337_gb300", "csrc"), "-I",
                    os.path.join(ROOT, "include"), src, "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0 and r.stdout == "ok\n", r.stdout + r.stderr
