"""The strip kernels of the mixed policy (``csrc/strips.cuh``: Rayleigh quotients, residual,
projection right-hand side) at the edges of their strips.

``tests/native/strips_check.cu`` runs them on levels whose width is below, at and above the 30 and 31
nodes of a strip and whose height leaves part of a row block, with Bloch phases per group, random
weights, noise and smooth fields, and compares every entry and sum with long double on the host.
"""
import os
import shutil
import subprocess

import pytest

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2304_00337_gb300", "csrc")
SRC = os.path.join(ROOT, "tests", "native", "strips_check.cu")

pytestmark = pytest.mark.gpu


def test_strips_against_long_double(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "strips_check")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-I", CSRC, SRC, "-o", exe],
                   check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.endswith("ok\n"), r.stdout + r.stderr
