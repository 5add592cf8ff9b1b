"""The tensor-core Gram (``csrc/gram_tc.cu``) at the edges of its blocks, tiles and scales.

Widths around the 32-column blocks (one block, two, three; nine is the narrowest that runs there),
meshes whose sides leave part of a 32 x 8 tile, columns of very different sizes, a zero column,
columns far outside the binary32 range, a strong permittivity contrast, and non-finite columns.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2304_00337_gb300 as pbs  # noqa: E402
from oracle import extrapolation as ex, fem  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as ge
    ge.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    with pbs.Context(0) as c:
        yield c


def _gram(ctx, geom, k, S):
    q = S.shape[0]
    Sd = torch.from_numpy(np.ascontiguousarray(S)).cuda()
    GM = torch.zeros((q, q), dtype=torch.complex128, device="cuda")
    GA = torch.zeros_like(GM)
    ctx.gram(geom, k, q, Sd.data_ptr(), GM.data_ptr(), GA.data_ptr(), torch.cuda.current_stream(),
             precision=pbs.PBS_MIXED)
    torch.cuda.synchronize()
    return GM.cpu().numpy().T, GA.cpu().numpy().T


def _check(got, want, N):
    # every operand value is rounded by at most 2^-47 of its column's largest one, which is at most
    # the root of the diagonal entry: 2^-46 sqrt(2 N) of sqrt(G_aa G_bb) by Cauchy-Schwarz
    d = np.sqrt(np.real(np.diag(want)))
    assert np.all(np.abs(got - want) <= 2.0 ** -46 * np.sqrt(2 * N) * np.outer(d, d))
    assert np.array_equal(got, got.conj().T)


@pytest.mark.parametrize("a,b,n,m,k", [(1.0, 1.0, 4, 6, (0.3, 0.2)), (1.0, 0.7, 20, 28, (2.1, -0.7)),
                                       (1.0, 2.0, 34, 18, (np.pi, np.pi)), (1.0, 1.0, 64, 32, (0.0, 0.0))])
@pytest.mark.parametrize("q", [9, 32, 33, 64, 65, 96])
def test_widths_and_tiles(ctx, a, b, n, m, k, q):
    rng = np.random.default_rng(q + n)
    eps = rng.uniform(1.0, 9.0, (m, n))
    geom = pbs.Geometry(eps, a, b)
    S = rng.standard_normal((q, geom.D)) + 1j * rng.standard_normal((q, geom.D))
    S *= np.logspace(0, -9, q)[:, None]
    S[q // 2] = 0.0
    S[q // 3, 1:] = 0.0  # a single edge
    ops = fem.assemble(fem.Mesh(a, b, n, m), eps, k)
    wm, wa = ex.grams(ops, S.T)
    gm, ga = _gram(ctx, geom, k, S)
    _check(gm, wm, n * m)
    _check(ga, wa, n * m)


def test_scales_and_contrast(ctx):
    # columns at 1e-60 .. 1e+60 (outside binary32), eps over four decades, smooth fields whose curls
    # are far smaller than they are
    n, m, k = 40, 24, (0.5, 0.3)
    rng = np.random.default_rng(3)
    eps = 10.0 ** rng.uniform(0.0, 4.0, (m, n))
    geom = pbs.Geometry(eps)
    i, j = np.meshgrid(np.arange(n), np.arange(m), indexing="xy")
    S = []
    for t in range(12):
        f = np.exp(2j * np.pi * ((t % 3) * i / n + (t % 2) * j / m)) * np.exp(1j * (k[0] * i / n + k[1] * j / m))
        S.append(np.concatenate([f.ravel(), (t - 5.0) * f.ravel()]) * 10.0 ** (10 * (t - 6)))
    S = np.array(S)
    ops = fem.assemble(fem.Mesh(1.0, 1.0, n, m), eps, k)
    scale = 10.0 ** (10.0 * (np.arange(12) - 6))
    wm, wa = ex.grams(ops, (S / scale[:, None]).T)
    gm, ga = _gram(ctx, geom, k, S)
    _check(gm / np.outer(scale, scale), wm, n * m)
    d = np.sqrt(np.real(np.diag(wa)))
    # the reference's own curls lose what cancels: 2^-53 of the edge values, times sqrt(w)
    lost = 8 * 2.0 ** -53 * np.abs(S / scale[:, None]).max(axis=1) * np.sqrt((n * m) / eps.min() * n * m)
    tol = 2.0 ** -46 * np.sqrt(2 * n * m) * np.outer(d, d) + np.outer(d, lost) + np.outer(lost, d)
    assert np.all(np.abs(ga / np.outer(scale, scale) - wa) <= tol)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_columns_stay_visible(ctx, bad):
    n = 16
    geom = pbs.Geometry(np.full((n, n), 2.0))
    rng = np.random.default_rng(1)
    S = rng.standard_normal((12, geom.D)) + 1j * rng.standard_normal((12, geom.D))
    want = _gram(ctx, geom, (0.4, 0.1), S)
    S[7, 100] = bad
    got = _gram(ctx, geom, (0.4, 0.1), S)
    keep = np.arange(12) != 7
    for g, w in zip(got, want):
        assert not np.any(np.isfinite(g[7])) and not np.any(np.isfinite(g[:, 7]))
        assert np.array_equal(g[np.ix_(keep, keep)], w[np.ix_(keep, keep)])
