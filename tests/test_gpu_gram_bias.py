"""No systematic error in the mixed policy's Gram matrices.

Fixed-point operands that are cut off instead of rounded are all a little small, and a diagonal entry
sums their squares: the error does not average out over the nodes as that of a rounding does.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2304_00337_gb300 as pbs  # noqa: E402

pytestmark = pytest.mark.gpu

K = (0.7, -1.1)


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as ge
    ge.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    with pbs.Context(0) as c:
        yield c


@pytest.mark.parametrize("n,m,q,r", [(128, 96, 12, 1.0), (128, 96, 40, 1.0), (96, 128, 16, 5.0)])
def test_diagonal(ctx, n, m, q, r):
    a, b = 1.0, r * m / n  # h2 / h1 = r
    rng = np.random.default_rng(n + q)
    eps = rng.uniform(1.0, 2.0, (m, n))
    x = rng.standard_normal((q, 2, m, n)) + 1j * rng.standard_normal((q, 2, m, n))
    x[:, 1] *= r
    Sd = torch.from_numpy(x.reshape(q, -1)).cuda()
    G = torch.zeros((2, q, q), dtype=torch.complex128, device="cuda")
    ctx.gram(pbs.Geometry(eps, a, b), K, q, Sd.data_ptr(), G[0].data_ptr(), G[1].data_ptr(), torch.cuda.current_stream(),
             precision=pbs.PBS_MIXED)
    torch.cuda.synchronize()
    ld, cld = np.longdouble, np.clongdouble
    X, Y = x[:, 0].astype(cld), x[:, 1].astype(cld)
    h1, h2 = ld(a) / n, ld(b) / m
    al, be = (cld(complex(np.cos(k), np.sin(k))) for k in (K[0] * a, K[1] * b))
    up = np.concatenate([X[:, 1:], be * X[:, :1]], axis=1)
    right = np.concatenate([Y[:, :, 1:], al * Y[:, :, :1]], axis=2)
    r3 = 1 / np.sqrt(ld(3))
    z = [np.sqrt(h2 / h1) * ((1 + r3) / 2 * X + (1 - r3) / 2 * up), np.sqrt(h1 / h2) * ((1 + r3) / 2 * Y + (1 - r3) / 2 * right)]
    c = np.sqrt(1 / (eps.astype(ld) * h1 * h2)) * (up - X - right + Y)
    for got, v in ((G[0], np.stack(z, axis=1)), (G[1], c)):
        sq = (np.abs(v.real) ** 2 + np.abs(v.imag) ** 2).reshape(q, -1)
        want = sq.sum(axis=1)
        err = ((np.real(np.diag(got.cpu().numpy())).astype(ld) - want) / want).astype(float)
        # a component's error is uniform within 2^-48 of a scale below four times the column's largest
        # one, and independent from node to node: 2 * 2^-48 * 4 big / sqrt(12) over the root of the sum,
        # for the mean of the columns over the root of their number; six standard deviations, and two
        # roundings of the FP64 sums
        big = np.maximum(np.abs(v.real), np.abs(v.imag)).reshape(q, -1).max(axis=1)
        sd = float(np.max(2.0 * 2.0 ** -48 * 4.0 * big / np.sqrt(12.0) / np.sqrt(want)))
        assert abs(np.mean(err)) <= 6.0 * sd / np.sqrt(q) + 2 * 2.0 ** -53, (np.mean(err), sd)


@pytest.mark.parametrize("n,m,q", [(64, 64, 12), (256, 192, 40), (2048, 1024, 72)])
def test_operands_at_the_end_of_their_range(ctx, n, m, q):
    # every curl of a column has the same size, just below its bound: the first digits stand at the ends
    # of their nine bits at every node and the integer sums are as large as they get (2048 x 1024, 72
    # columns: 128 chunks each).  Values of 20 bits and w = 4^k: nothing is rounded but the FP64 sums.
    x = torch.zeros((q, 2, m, n), dtype=torch.complex128, device="cuda")
    row = (1.0 - 2.0 * (torch.arange(m, device="cuda") % 2))[:, None]
    rng = np.random.default_rng(q)
    s = np.array([complex(*rng.choice([-1.0, 1.0], 2)) * 2.0 ** int(rng.integers(-9, 10)) for _ in range(q)])
    v = round(0.97 * 2 ** 20) / 2 ** 20
    for c in range(q):
        x[c, 0] = (0.5 * v * complex(s[c])) * row  # curls -+ v s
    w = 4.0 ** int(np.ceil(np.log(n * m) / np.log(4)))
    G = torch.zeros((2, q, q), dtype=torch.complex128, device="cuda")
    ctx.gram(pbs.Geometry(np.full((m, n), n * m / w)), (0.0, 0.0), q, x.data_ptr(), G[0].data_ptr(), G[1].data_ptr(),
             torch.cuda.current_stream(), precision=pbs.PBS_MIXED)
    torch.cuda.synchronize()
    got, want = G[1].cpu().numpy().T, n * m * w * v * v * np.outer(s.conj(), s)
    # up to 1000 partial sums of one size, added in eight lanes
    assert np.max(np.abs(got - want) / np.abs(np.outer(s, s))) <= n * m * w * 2.0 * 130 * 2.0 ** -53
