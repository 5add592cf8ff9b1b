"""The fused coarse levels (``csrc/tail.cuh``) and the coarsest factorisation where they can go wrong.

Columns decide how many CTAs share a column under FP64 (four up to 38 columns, two up to 76, one
beyond), the mesh how many levels those CTAs share, how the block rows split, and which form the
coarsest factor takes (up to 64 unknowns in one block of threads, beyond by 32-column panels; its
copy in shared memory where it fits).  Every case is compared with the oracle's V-cycle at
``mu = lambda_max / 1000``, where a cycle amplifies rounding by about 50 units (the bars of the
other V-cycle tests: 1e-12 and 1e-5).
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2304_00337_gb300 as pbs  # noqa: E402
from oracle import fem, multigrid as mg  # noqa: E402

pytestmark = pytest.mark.gpu

# (a, b, n, m, k, coarsest): square meshes of one and of several shared levels, long ones in either
# direction, odd coarsest meshes (13 x 9: 234 edges; 5 x 7), a block-row count no CTA count divides,
# the zone corner and Gamma
MESHES = [
    (1.0, 1.0, 64, 64, (0.4, -1.3), 4),
    (1.0, 1.0, 32, 32, (np.pi, np.pi), 4),
    (1.0, 0.25, 128, 32, (0.9, 2.2), 4),
    (0.25, 1.0, 16, 64, (-0.7, 0.2), 4),
    (1.0, 0.7, 52, 36, (0.4, -1.3), 4),
    (1.0, 1.4, 20, 28, (1.1, 0.6), 4),
    (1.0, 1.0, 24, 24, (0.0, 0.0), 2),
    (1.0, 1.0, 26, 22, (0.3, 0.8), 4),
]


@pytest.fixture(scope="module")
def ctx():
    import __graft_entry__ as ge
    ge.build()
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    with pbs.Context(0) as c:
        yield c


@pytest.mark.parametrize("ncols", [2, 40, 80])
@pytest.mark.parametrize("a,b,n,m,k,coarsest", MESHES)
def test_coarse_levels_match_oracle(ctx, a, b, n, m, k, coarsest, ncols):
    rng = np.random.default_rng(n + 3 * m)
    eps = rng.uniform(1.0, 9.0, (m, n))
    geom = pbs.Geometry(eps, a, b)
    mesh = fem.Mesh(a, b, n, m)
    mu = 12.0 * (1.0 / mesh.h1 ** 2 + 1.0 / mesh.h2 ** 2) / 1000.0
    gamma = fem.is_gamma(*fem.bloch_phases(k, a, b))
    levels = mg.edge_hierarchy(mesh, eps, k, mu, coarsest)
    nlev = mg.nodal_hierarchy(mesh, eps, k, coarsest)
    for op, size, cycle, hier in (("VCYCLE_EDGE", mesh.D, mg.edge_vcycle, levels),
                                  ("VCYCLE_NODAL", mesh.N, mg.nodal_vcycle, nlev)):
        x = rng.standard_normal((ncols, size)) + 1j * rng.standard_normal((ncols, size))
        if gamma and op == "VCYCLE_NODAL":
            x -= x.mean(axis=1, keepdims=True)
        want = np.stack([cycle(hier, x[c]) for c in (0, ncols - 1)])
        for prec, bar in ((pbs.PBS_FP64, 1e-12), (pbs.PBS_MIXED, 1e-5)):
            xd = torch.from_numpy(x).cuda()
            yd = torch.zeros_like(xd)
            ctx.apply(geom, op, xd.data_ptr(), yd.data_ptr(), ncols, k=k,
                      opts=pbs.default_opts(mu=mu, precision=prec, coarsest=coarsest),
                      stream=torch.cuda.current_stream())
            torch.cuda.synchronize()
            got = yd.cpu().numpy()[[0, ncols - 1]]
            err = np.max(np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1))
            assert err <= bar, (op, prec, err)
