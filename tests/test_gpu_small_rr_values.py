"""Ritz values of the small dense solve: as exact as its arithmetic lets them be, at every width.

With more than 16 values wanted a half warp refines each of them, 17-fold per step, and the last bracket's
width is part of the error; with wide blocks a lane sums more products.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2304_00337_gb300 as pbs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _theta(GM, GA, p):
    q = len(GM)
    gm, ga = (torch.from_numpy(np.ascontiguousarray(g.T)).cuda() for g in (GM, GA))
    C = torch.zeros((p, q), dtype=torch.complex128, device="cuda")
    th = torch.zeros(p, dtype=torch.float64, device="cuda")
    info = torch.zeros(8, dtype=torch.int32, device="cuda")
    pbs.small_rr_noalloc(gm.data_ptr(), ga.data_ptr(), q, p, C.data_ptr(), th.data_ptr(), info.data_ptr(),
                         torch.cuda.current_stream())
    torch.cuda.synchronize()
    assert info[0].item() == 0
    return th.cpu().numpy()


@pytest.mark.parametrize("q,p", [(20, 16), (20, 17), (72, 24), (96, 32)])
def test_width_of_the_last_bracket(q, p):
    # A diagonal pencil: the tridiagonal matrix holds its entries exactly, so what is left is half the last
    # bracket, 0.7e-15 of the norm, and the double-float roundings of values 1 / 64 of the norm and below
    # (2^-48 each).  The Gershgorin interval is the widest there is for its norm.
    lam = np.concatenate([[-1024.0], np.linspace(1.0, 16.0, p - 1).round(3), np.linspace(100.0, 1024.0, q - p).round(1)])
    th = _theta(np.eye(q, dtype=complex), np.diag(lam).astype(complex), p)
    assert np.max(np.abs(th[1:] - lam[1:p])) <= 1024.0 * (0.7e-15 + 4 * 2.0 ** -48 / 64)


def _reference(GM, GA):
    """Eigenvalues of the pencil: FP64 eigenvectors refined and their Rayleigh quotients in extended precision."""
    q = len(GM)
    M, A = GM.astype(np.clongdouble), GA.astype(np.clongdouble)
    Li = np.linalg.inv(np.linalg.cholesky(GM))
    H = Li @ GA @ Li.conj().T
    Y = (Li.conj().T @ np.linalg.eigh((H + H.conj().T) / 2)[1]).astype(np.clongdouble)
    for last in (False, True):
        m, a = Y.conj().T @ M @ Y, Y.conj().T @ A @ Y
        lam = np.real(np.diag(a)) / np.real(np.diag(m))
        if last:
            return np.sort(lam)
        R, D = np.eye(q) - m, lam[None, :] - lam[:, None]
        np.fill_diagonal(D, 1)
        E = (a + R * lam[None, :]) / D
        np.fill_diagonal(E, np.real(np.diag(R)) / 2)
        Y = Y + Y @ E


@pytest.mark.parametrize("q,p", [(42, 14), (60, 20), (96, 32)])
def test_error_does_not_grow_with_the_width(q, p):
    errors = []
    for seed in range(10):
        rng = np.random.default_rng(100 * q + seed)
        S = rng.standard_normal((3 * q, q)) + 1j * rng.standard_normal((3 * q, q))
        w = np.logspace(0, 1 + seed % 3, 3 * q)
        GM, GA = S.conj().T @ S, S.conj().T @ (w[:, None] * S)
        GM, GA = (GM + GM.conj().T) / 2, (GA + GA.conj().T) / 2
        want = _reference(GM, GA)
        errors.append(np.max(np.abs(_theta(GM, GA, p) - want[:p])) / want[-1])
    # one unit of 2^-48 of the norm for the entries' rounding and one for the unitary reduction, of random
    # sign, and 15 % for a sample of ten
    assert np.sqrt(np.mean(np.square(errors))).astype(float) <= 1.15 * np.sqrt(2.0) * 2.0 ** -48, errors
