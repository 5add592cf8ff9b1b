"""The tensor-core block update (``csrc/update_tc.cu``) where x- and y-edges differ in size.

On a mesh with h2/h1 = r the two fields of a column differ by about r.  ``update_tc_fields_check.cu``
gives them ratios up to 2^80 and holds every value to the bound of its own field.
"""
import os
import shutil
import subprocess

import pytest

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2304_00337_gb300", "csrc")
SRC = os.path.join(ROOT, "tests", "native", "update_tc_fields_check.cu")

pytestmark = pytest.mark.gpu


def test_each_field_to_its_own_bound(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "update_tc_fields_check")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), SRC, "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.endswith("ok\n"), r.stdout + r.stderr
