"""The small dense Rayleigh-Ritz solve at the edges of its sizes and storage modes.

``k_small_rr`` keeps both matrices in shared memory up to q = 75 (with p = 25), one of them from
there on, none of them behind ``pbs_small_rr_noalloc``; lane groups share rows, and half warps take
over the eigenvalues from p = 17 on.  Each size is compared with numpy's solve of the same pencil.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2304_00337_gb300 as pbs  # noqa: E402
import pbs_inputs as gi  # noqa: E402
from oracle import fem  # noqa: E402

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (2, 1), (2, 2), (3, 2), (5, 5), (16, 16), (17, 17), (31, 10), (33, 11), (34, 32), (64, 3), (72, 24),
         (75, 25), (76, 25), (96, 32)]


@pytest.fixture(scope="module")
def setup():
    import __graft_entry__ as ge
    ge.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    n, k = 16, (0.6, -0.3)
    eps = gi.rod_eps(n, n)
    with pbs.Context(0) as c:
        yield c, pbs.Geometry(eps), fem.assemble(fem.Mesh(1.0, 1.0, n, n), eps, k), k


def _reference(ops, S):
    GM, GA = S.conj() @ (ops["M"] @ S.T), S.conj() @ (ops["A"] @ S.T)
    Li = np.linalg.inv(np.linalg.cholesky(GM))
    th = np.linalg.eigvalsh(Li @ GA @ Li.conj().T)
    return GM, GA, th, np.linalg.cond(GM)


@pytest.mark.parametrize("mode", ["fp64", "mixed", "noalloc"])
@pytest.mark.parametrize("q,p", SIZES)
def test_small_rayleigh_ritz(setup, q, p, mode):
    ctx, geom, ops, k = setup
    r = np.random.default_rng(1000 + q)
    S = r.standard_normal((q, geom.D)) + 1j * r.standard_normal((q, geom.D))
    S *= np.logspace(0, -4, q)[:, None]  # columns of different sizes, as in a trial block
    GM, GA, th, cond = _reference(ops, S / np.logspace(0, -4, q)[:, None])
    # rounding u of the arithmetic through q-term sums and triangular solves, relative to the
    # largest Ritz value and the conditioning of the scaled Gram matrix, and the bracket of
    # 4e-15 of the norm that the eigenvalues are refined to
    u = 2.0 ** -53 if mode == "fp64" else 2.0 ** -47
    tol = cond * (8 * q * u + 8e-15)
    s = torch.cuda.current_stream()
    Sd = torch.from_numpy(np.ascontiguousarray(S)).cuda()
    if mode == "noalloc":
        gm = torch.empty((q, q), dtype=torch.complex128, device="cuda")
        ga = torch.empty_like(gm)
        ctx.gram(geom, k, q, Sd.data_ptr(), gm.data_ptr(), ga.data_ptr(), s)
        C = torch.full((p, q), complex(np.nan, np.nan), dtype=torch.complex128, device="cuda")
        theta = torch.zeros(p, dtype=torch.float64, device="cuda")
        info = torch.full((2,), 99, dtype=torch.int32, device="cuda")
        pbs.small_rr_noalloc(gm.data_ptr(), ga.data_ptr(), q, p, C.data_ptr(), theta.data_ptr(), info.data_ptr(), s)
        torch.cuda.synchronize()
        assert info.cpu().tolist() == [0, q]
        X = (C @ Sd).cpu().numpy()
        theta = theta.cpu().numpy()
    else:
        prec = pbs.PBS_FP64 if mode == "fp64" else pbs.PBS_MIXED
        Xd = torch.zeros((p, geom.D), dtype=torch.complex128, device="cuda")
        theta = ctx.rayleigh_ritz(geom, pbs.default_opts(precision=prec), k, q, Sd.data_ptr(), p, False,
                                  Xd.data_ptr(), s)
        X = Xd.cpu().numpy()
    assert np.all(np.abs(theta - th[:p]) <= tol * th[-1])
    assert np.all(np.abs(X.conj() @ (ops["M"] @ X.T) - np.eye(p)) <= 10 * tol)
    assert np.all(np.abs(X.conj() @ (ops["A"] @ X.T) - np.diag(th[:p])) <= 10 * tol * th[-1])


def test_dropped_directions(setup):
    # a zero and a repeated column: two directions dropped, the others as without them
    ctx, geom, ops, k = setup
    r = np.random.default_rng(5)
    S = r.standard_normal((20, geom.D)) + 1j * r.standard_normal((20, geom.D))
    T = np.insert(np.insert(S, 7, 0.0, axis=0), 12, S[3], axis=0)
    _, _, th, cond = _reference(ops, S)
    for prec, u in ((pbs.PBS_FP64, 2.0 ** -53), (pbs.PBS_MIXED, 2.0 ** -47)):
        Td = torch.from_numpy(np.ascontiguousarray(T)).cuda()
        X = torch.zeros((6, geom.D), dtype=torch.complex128, device="cuda")
        theta = ctx.rayleigh_ritz(geom, pbs.default_opts(precision=prec), k, 22, Td.data_ptr(), 6, False, X.data_ptr(),
                                  torch.cuda.current_stream())
        assert np.all(np.abs(theta - th[:6]) <= cond * (8 * 22 * u + 8e-15) * 2 * th[-1])
