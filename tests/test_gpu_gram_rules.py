"""Where the mixed policy's Gram runs: on either side of the rule, and what runs there.

The tensor-core kernel takes nine columns and more while the permittivities span at most 2^16 (every
width with PBS_GRAM=tc); everything else is the double-float kernel's, whose launches are counted.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2304_00337_gb300 as pbs  # noqa: E402
from oracle import eigen, extrapolation as ex, fem  # noqa: E402
from test_gpu_tuner import _child, test_gram_bank_spread_stride_forced as _forced  # noqa: E402

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
N, M, K = 32, 24, (0.7, -1.1)


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as ge
    ge.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    with pbs.Context(0) as c:
        yield c


def _case(q, contrast):
    rng = np.random.default_rng(q)
    eps = np.where(rng.random((M, N)) < 0.5, 1.0, contrast)
    S = rng.standard_normal((q, 2 * N * M)) + 1j * rng.standard_normal((q, 2 * N * M))
    return eps, S * np.logspace(0, -9, q)[:, None]


def _gram(ctx, eps, S):
    q = len(S)
    Sd, G = torch.from_numpy(S).cuda(), torch.zeros((2, q, q), dtype=torch.complex128, device="cuda")
    before = pbs.launch_count_df()
    ctx.gram(pbs.Geometry(eps), K, q, Sd.data_ptr(), G[0].data_ptr(), G[1].data_ptr(), torch.cuda.current_stream(),
             precision=pbs.PBS_MIXED)
    torch.cuda.synchronize()
    return [g.T for g in G.cpu().numpy()], pbs.launch_count_df() - before


def _errors(got, eps, S):
    """Entry errors of both matrices relative to sqrt(G_aa G_bb)."""
    want = ex.grams(fem.assemble(fem.Mesh(1.0, 1.0, N, M), eps, K), S.T)
    out = []
    for g, w in zip(got, want):
        d = np.sqrt(np.real(np.diag(w)))
        out.append(float(np.max(np.abs(g - w) / np.outer(d, d))))
        assert np.array_equal(g, g.conj().T)
    return out


# noise columns: every product is right to a few units of 2^-47 of sqrt(w) times edge values, which
# are no larger than the curls' root mean square times two; 2^-46 per operand and the oracle's own
# FP64 sums stay below 1e-13
BAR = 1e-13


@pytest.mark.parametrize("q", [9, 30, 72])
@pytest.mark.parametrize("contrast,df", [(65536.0, False), (65540.0, True), (1e7, True)])
def test_contrast_on_either_side_of_the_rule(ctx, contrast, df, q):
    eps, S = _case(q, contrast)
    got, launches = _gram(ctx, eps, S)
    assert (launches > 0) == df
    assert max(_errors(got, eps, S)) <= BAR


def test_mixed_solve_beyond_the_contrast_of_the_tensor_cores(ctx):
    # the whole iteration on the double-float Gram and updates, 30 trial columns
    n, k = 16, (1.1, 0.4)
    eps = np.where(np.hypot(*(np.indices((n, n)) - 7.5)) < 1.0, 70000.0, 1.0)
    want = eigen.solve_k(1.0, 1.0, n, n, eps, k, 6, "dense")[0][:6]
    before = pbs.launch_count_df()
    lam, res, it, _ = ctx.solve_k(pbs.Geometry(eps), dict(nev=6, block=10, precision=pbs.PBS_MIXED), k)
    assert pbs.launch_count_df() - before > it
    # Both sides compute in FP64 on a pencil of norm lambda_max: 16 units of 2^-53 lambda_max each, and the
    # square of the residual bound 1e-8 relative to the gap (far below that)
    top = 12.0 * 2 * n * n
    assert np.all(np.abs(lam - want) <= 32 * 2.0 ** -53 * top + 1e-9 * want), (lam, want)


@pytest.mark.parametrize("cand", [0, 1])
def test_packed_stride_forced(cand):
    # the candidates without padding, on the widths that the tensor cores take otherwise
    _forced(cand)


NARROW = r"""
import json
import numpy as np
import test_gpu_gram_rules as t
import __graft_entry__ as ge
ge.build()
import paper_2304_00337_gb300 as pbs
out = []
with pbs.Context(0) as ctx:
    for q in range(1, 9):
        eps, S = t._case(q, 12.0)
        got, launches = t._gram(ctx, eps, S)
        out.append([q, launches, max(t._errors(got, eps, S))])
print(json.dumps(out))
"""


@pytest.mark.parametrize("tc", [True, False])
def test_narrow_blocks(tc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    for q, launches, err in _child({"PBS_GRAM": "tc"} if tc else {}, NARROW):
        assert (launches == 0) == tc and err <= BAR, (q, launches, err)


def test_groups_of_one_launch(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    exe = str(tmp_path / "gram_groups_check")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O2", "-std=c++17", "-I",
                    os.path.join(ROOT, "paper_2304_00337_gb300", "csrc"), "-I", os.path.join(ROOT, "include"),
                    os.path.join(ROOT, "tests", "native", "gram_groups_check.cu"), "-o", exe], check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.endswith("ok\n"), r.stdout + r.stderr
