"""The kernels in which a warp walks up a strip of the mesh, at the edges of their strips.

``csrc/strips.cuh`` (Rayleigh quotients, residual, projection right-hand side of the mixed policy):

``tests/native/strips_check.cu`` runs them on levels whose width is below, at and above the 30 and 31
nodes of a strip and whose height leaves part of a row block, with Bloch phases per group, random
weights, noise and smooth fields, and compares every entry and sum with long double on the host.

``csrc/node_strips.cuh`` (fine-level steps of the nodal cycle): ``tests/native/node_strips_check.cu``
compares them with the tiled kernels.
"""
import os
import shutil
import subprocess

import pytest

torch = pytest.importorskip("torch")

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2304_00337_gb300", "csrc")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["strips_check", "node_strips_check"])
def test_strips(tmp_path, name):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe, src = str(tmp_path / name), os.path.join(ROOT, "tests", "native", name + ".cu")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-I", CSRC, src, "-o", exe],
                   check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.endswith("ok\n"), r.stdout + r.stderr
