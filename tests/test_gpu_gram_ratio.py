"""The mixed policy's Gram matrices on meshes whose cells are not square.

Edge values are line integrals: with h2/h1 = r a smooth field has |y|/|x| about r, and the larger
field carries the smaller mass weight.  The tensor-core kernel rounds its operands relative to a
bound of the column, so the bound has to be one of the weighted values; entry errors are then the
same at every r.  Reference: the same sums in extended precision.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2304_00337_gb300 as pbs  # noqa: E402

pytestmark = pytest.mark.gpu

N, M, Q, K = 32, 48, 12, (0.7, -1.1)


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as ge
    ge.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    with pbs.Context(0) as c:
        yield c


def _columns(kind, r):
    """Columns (Q, 2, M, N) of edge values and their Bloch phases per step along i and j."""
    rng = np.random.default_rng(int(8 * r) + len(kind))
    i, j = np.meshgrid(np.arange(N), np.arange(M), indexing="xy")
    x = np.zeros((Q, 2, M, N), complex)
    for c in range(Q):
        if kind == "smooth":  # a field of equal components; the mean of irregular plane waves
            f = np.zeros((M, N), complex)
            for _ in range(4):
                u, v = rng.integers(-2, 3, 2)
                f += rng.standard_normal() * np.exp(2j * np.pi * (u * i / N + v * j / M) + 1j * (K[0] * i / N + K[1] * j / M))
            x[c, 0], x[c, 1] = f, r * f * np.exp(0.3j * c)
        else:
            z = rng.standard_normal((2, M, N)) + 1j * rng.standard_normal((2, M, N))
            x[c] = z * (np.array([1, 0]) if kind == "x" else np.array([0, 1]) if kind == "y" else np.array([1, r]))[:, None, None]
    return x


def _reference(S, eps, a, b):
    """Gram matrices, the largest weighted operand and the edge values' share of a curl, extended precision."""
    ld, cld = np.longdouble, np.clongdouble
    x, y = S[:, 0].astype(cld), S[:, 1].astype(cld)
    h1, h2 = ld(a) / N, ld(b) / M
    al, be = (cld(complex(np.cos(k), np.sin(k))) for k in (K[0] * a, K[1] * b))
    up = np.concatenate([x[:, 1:], be * x[:, :1]], axis=1)
    right = np.concatenate([y[:, :, 1:], al * y[:, :, :1]], axis=2)
    r3 = 1 / np.sqrt(ld(3))
    ca, cb = (1 + r3) / 2, (1 - r3) / 2
    z = np.concatenate([np.sqrt(h2 / h1) * (ca * x + cb * up), np.sqrt(h1 / h2) * (ca * y + cb * right)], axis=1)
    sw = np.sqrt(1 / (eps.astype(ld) * h1 * h2))
    c = sw * (up - x - right + y)
    gram = lambda v: np.einsum("ak,bk->ab", v.reshape(Q, -1).conj(), v.reshape(Q, -1))  # noqa: E731
    big = lambda v: np.maximum(np.abs(v.real), np.abs(v.imag)).reshape(Q, -1).max(axis=1).astype(float)  # noqa: E731
    wz = np.maximum(np.sqrt(h2 / h1) * big(x), np.sqrt(h1 / h2) * big(y)) * np.sqrt(2.0)  # the continued values too
    edge = (sw.max() * np.maximum(big(x), big(y))).astype(float)
    return gram(z), gram(c), wz.astype(float), big(c), edge


@pytest.mark.parametrize("kind", ["smooth", "x", "y", "noise"])
@pytest.mark.parametrize("r", [1 / 64, 1 / 16, 1 / 3, 1.0, 4.0, 16.0, 64.0, 1000.0])
def test_gram_does_not_depend_on_the_cell_shape(ctx, r, kind):
    a, b = 1.0, r * M / N  # h2 / h1 = r
    eps = np.random.default_rng(1).uniform(1.0, 9.0, (M, N))
    S = _columns(kind, r)
    Sd = torch.from_numpy(S.reshape(Q, -1)).cuda()
    G = torch.zeros((2, Q, Q), dtype=torch.complex128, device="cuda")
    ctx.gram(pbs.Geometry(eps, a, b), K, Q, Sd.data_ptr(), G[0].data_ptr(), G[1].data_ptr(), torch.cuda.current_stream(),
             precision=pbs.PBS_MIXED)
    torch.cuda.synchronize()
    gm, ga = (g.T for g in G.cpu().numpy())
    wm, wa, bm, ba, edge = _reference(S, eps, a, b)
    # Operands are rounded to 2^-48 of a power of two below four times the column's largest one (a
    # factor two for the power of two, the margin and the bound's own rounding in the rest): an entry
    # sums that error times the other column's operands, six standard deviations of independent
    # roundings, 6 / sqrt(3).  Two of the dropped digit pairs weigh 2^-48 of the product of the two
    # scales each, digits uniform in +-128: 6 sqrt(8 N) / 3 of 4 N terms.
    for got, want, big, lost in ((gm, wm, bm, 0.0 * edge), (ga, wa, ba, edge)):
        d = np.sqrt(np.real(np.diag(want))).astype(float)
        e = 4.0 * big
        tol = 2.0 ** -48 * (3.5 * (np.outer(e, d) + np.outer(d, e)) + 5.7 * np.sqrt(N * M) * np.outer(e, e))
        # a curl also loses the fixed point of its four edge values, 2^-52 of a bound of the column
        # below twice its largest value
        tol += 4 * 2.0 ** -51 * (np.outer(lost, d) + np.outer(d, lost)) * np.sqrt(N * M)
        err = np.abs(got - want).astype(float)
        assert np.all(err <= tol), (r, kind, float(np.max(err / np.maximum(tol, 1e-300))),
                                    float(np.max(err / np.maximum(np.outer(d, d), 1e-300))))
        assert np.array_equal(got, got.conj().T)


@pytest.mark.parametrize("q", [12, 40])
def test_products_of_exact_operands(ctx, q):
    # Integers below 2^44 as edge values, w = 16 and no phases: the operands sqrt(w) curl are integers
    # that 48 bits hold exactly, so all that is lost are the digit pairs left out and the last places.
    # On 4 x 4 nodes those pairs would show if two more of them were (2^-48 of the scales each).
    n, k = 4, (0.0, 0.0)
    rng = np.random.default_rng(q)
    e = [[int(v) for v in rng.integers(-2 ** 44 + 1, 2 ** 44, 4 * n * n)] for _ in range(q)]
    S = np.array([np.array(c[:2 * n * n], float) + 1j * np.array(c[2 * n * n:], float) for c in e])
    Sd = torch.from_numpy(S).cuda()
    G = torch.zeros((2, q, q), dtype=torch.complex128, device="cuda")
    ctx.gram(pbs.Geometry(np.ones((n, n))), k, q, Sd.data_ptr(), G[0].data_ptr(), G[1].data_ptr(),
             torch.cuda.current_stream(), precision=pbs.PBS_MIXED)
    torch.cuda.synchronize()
    got = G[1].cpu().numpy().T

    def curls(c):  # x(i, j + 1) - x(i, j) - y(i + 1, j) + y(i, j)
        x, y = c[:n * n], c[n * n:]
        return [4 * (x[(j + 1) % n * n + i] - x[j * n + i] - y[j * n + (i + 1) % n] + y[j * n + i])
                for j in range(n) for i in range(n)]

    re, im = [curls(c[:2 * n * n]) for c in e], [curls(c[2 * n * n:]) for c in e]
    # the exponents bound |z| by a power of two below 2.1 times the largest
    scale = [2.1 * max(map(abs, re[c] + im[c])) for c in range(q)]
    for a in range(q):
        for b in range(a, q):
            want_re = sum(u * v for u, v in zip(re[a], re[b])) + sum(u * v for u, v in zip(im[a], im[b]))
            want_im = sum(u * v for u, v in zip(re[a], im[b])) - sum(u * v for u, v in zip(im[a], re[b]))
            size = sum((abs(u) + abs(s)) * (abs(v) + abs(t)) for u, s, v, t in zip(re[a], im[a], re[b], im[b]))
            # 2 n^2 real products; pairs (2, 5), (4, 3) at 2^-56 and what follows; eight roundings to FP64
            tol = scale[a] * scale[b] * (2 * n * n * 2.01 * 2.0 ** -56 + 4 * 2.0 ** -53) + 8 * 2.0 ** -53 * size
            assert abs(int(got[a, b].real) - want_re) <= tol and abs(int(got[a, b].imag) - want_im) <= tol, (a, b)
