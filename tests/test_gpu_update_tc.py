"""The tensor-core block update (``csrc/update_tc.cu``) at the edges of its tiles and widths.

``tests/native/update_tc_check.cu`` runs the kernel for widths around its quadruples and operand
tiles, heights around the 128-row tile, several groups, zero columns, columns whose sizes span many
decades, and compares every value with long double on the host.  The bound is derived from the
operand digits: a value of column i is rounded by 2^-62 of the column's bound, likewise the
coefficients, and the digit pairs left out are below 7.1 2^-62 of the largest product.
"""
import os
import shutil
import subprocess

import pytest

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2304_00337_gb300", "csrc")
SRC = os.path.join(ROOT, "tests", "native", "update_tc_check.cu")

pytestmark = pytest.mark.gpu


def test_update_against_long_double(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "update_tc_check")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), SRC, "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.endswith("ok\n"), r.stdout + r.stderr
