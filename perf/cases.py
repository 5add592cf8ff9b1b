"""Timed cases of the library: what a band-structure program has it do, through its public calls.

A case names a call and its sizes.  ``kind`` is the call:

* ``solve_k``      ``Context.solve_k``: one Bloch vector, a given start block;
* ``path``         ``Context.solve_path``: Bloch vectors of a Gamma-X-M-Gamma path, ``kbatch`` chains in flight;
* ``grid``         ``Context.solve_grid``: a ``kappa`` x ``kappa`` Brillouin-zone sample;
* ``serve``        ``Context.submit`` / ``Context.fetch``: path jobs of different meshes at once;
* ``gram``         ``Context.gram``: the block Gram matrices of a trial block;
* ``rr``           ``Context.rayleigh_ritz``: the extrapolation step (projection and Rayleigh-Ritz);
* ``householder``  ``Context.m_householder``: the M-orthonormal factorisation of a block;
* ``apply``        ``Context.apply``: one operator, multigrid cycle or projection on a block.

The eigensolves return the eigenvalues and, as whole numbers, whether each band met the documented
stopping rule; the residuals and iteration counts they also report say how the last iterate was
reached, and the eigenvectors are fixed up to a phase only.
"""
import math

import numpy as np
import torch

import paper_2304_00337_gb300 as pbs
import pbs_inputs

MIXED, FP64 = pbs.PBS_MIXED, pbs.PBS_FP64
TOL = 1e-8


def listed():
    return [
        # A first call, a unit check or one point of a coarse scan: the 32 x 32 homogeneous cell in
        # plain FP64 from a given random block; latency and launches.
        dict(name="solve_k_32_fp64", kind="solve_k", n=32, m=32, b=1.0, eps="const", nev=4, block=4, fp64=True),
        # The smallest call: one operator on a few columns, as a program's own iteration calls it.
        dict(name="apply_A_32", kind="apply", op="A", n=32, m=32, b=1.0, eps="rod", cols=4, fp64=True),
        # The ordinary job: a photonic-crystal band diagram, 31 Bloch vectors with extrapolation.
        dict(name="path_rod_256", kind="path", n=256, m=256, b=1.0, eps="rod", nk=31, kbatch=4, nev=8, block=10,
             fp64=False),
        # A fine mesh with every Bloch vector in flight: throughput of the large blocks.
        dict(name="path_rod_1024", kind="path", n=1024, m=1024, b=1.0, eps="rod", nk=4, kbatch=4, nev=8, block=10,
             fp64=False),
        # A rectangular cell with a random disk field on a mesh with odd factors, more bands.
        dict(name="path_disks_208x144", kind="path", n=208, m=144, b=0.7, eps="disks", nk=4, kbatch=2, nev=12,
             block=14, fp64=False),
        # The plain FP64 policy, which a user runs to check the mixed one.
        dict(name="path_rod_128_fp64", kind="path", n=128, m=128, b=1.0, eps="rod", nk=4, kbatch=2, nev=8, block=10,
             fp64=True),
        # A Brillouin-zone map with 16 bands and 8 throw-away vectors.
        dict(name="grid_rod_128", kind="grid", n=128, m=128, b=1.0, eps="rod", kappa=3, kbatch=3, nev=16, block=24,
             fp64=False),
        # Jobs of different meshes that arrive together.
        dict(name="serve_64_128", kind="serve", n=64, m=128, b=1.0, eps="rod", jobs=4, nk=4, kbatch=4, nev=6, block=8,
             fp64=False),
        # The blocks of the iteration, each through its own call.
        dict(name="gram_1024_q30", kind="gram", n=1024, m=1024, b=1.0, eps="rod", q=30, fp64=False),
        dict(name="rr_256_q30_fp64", kind="rr", n=256, m=256, b=1.0, eps="rod", q=30, p=10, project=True, fp64=True),
        dict(name="householder_256_q30", kind="householder", n=256, m=256, b=1.0, eps="rod", q=30, fp64=True),
        dict(name="vcycle_512_fp64", kind="apply", op="VCYCLE_EDGE", n=512, m=512, b=1.0, eps="rod", cols=10,
             fp64=True),
    ]


def _log_int(rng, lo, hi, step):
    """A multiple of `step` in [lo, hi], spread over the logarithm."""
    return max(lo, min(hi, step * int(round(math.exp(rng.uniform(math.log(lo), math.log(hi))) / step))))


def draw(rng):
    kind = rng.choice(["solve_k", "path", "path", "path", "grid", "serve", "gram", "gram", "rr", "householder",
                       "apply", "apply"])
    c = dict(kind=kind, b=rng.choice([1.0, 1.0, 0.7, 1.6]), eps=rng.choice(["rod", "rod", "disks"]))
    if kind in ("solve_k", "path", "grid"):
        fp64 = rng.random() < 0.25
        nev = rng.randint(4, 12)
        block = min(24, nev + rng.choice([2, 2, 3, 8]))
        # sides with an odd factor left on the coarsest mesh among them
        n = _log_int(rng, 32, 128 if fp64 or kind == "grid" else 640, 16)
        m = n if rng.random() < 0.5 else max(32, min(n, _log_int(rng, max(32, n // 2), 2 * n, 16)))
        c.update(n=n, m=m, nev=nev, block=block, fp64=fp64)
        if kind == "path":
            # Bloch vectors: fewer on finer meshes, so that a draw costs no more than the listed cases
            most = max(2, int(1.2e6 * (0.25 if fp64 else 1.0) / (n * m) * 10 / block))
            c["nk"] = rng.randint(2, max(2, min(16, most)))
            c["kbatch"] = rng.randint(1, min(c["nk"], 8))
        elif kind == "grid":
            c.update(kappa=rng.randint(2, 3), kbatch=rng.randint(1, 3))
    elif kind == "serve":
        n = _log_int(rng, 32, 128, 16)
        nev = rng.randint(4, 8)
        c.update(n=n, m=_log_int(rng, 32, 128, 16), jobs=rng.randint(2, 4), nk=rng.randint(2, 4),
                 kbatch=rng.randint(1, 4), nev=nev, block=nev + 2, fp64=False)
    else:
        n = _log_int(rng, 32, 1024, 2 if kind in ("gram", "householder") else 16)
        m = n if rng.random() < 0.5 else max(32, min(1024, _log_int(rng, max(32, n // 2), 2 * n, 16)))
        c.update(n=n, m=m, fp64=True)
        if kind == "gram":
            small = n * m < 2.0e5
            c.update(q=rng.randint(3, 96 if small else 42), fp64=small and rng.random() < 0.3)
        elif kind == "rr":
            p = rng.randint(4, 12)
            c.update(n=min(n, 512), m=min(m, 512), q=p * rng.randint(2, 3), p=p, project=rng.random() < 0.7)
        elif kind == "householder":
            c.update(n=min(n, 512), m=min(m, 512), q=rng.randint(4, 40))
        else:
            c.update(op=rng.choice(["A", "M", "A_MU_M", "L", "LH", "P_NODAL", "RESIDUAL", "LH_M", "VCYCLE_EDGE",
                                    "VCYCLE_NODAL", "PROJECT"]), cols=rng.randint(1, 16))
    c["n"], c["m"] = _coarse(c["n"]), _coarse(c["m"])  # the multigrid's coarsest dense system has to stay small
    return c


def _coarse(n):
    """The nearest side up to `n` that halves down to an odd number of at most 13."""
    while True:
        k = n
        while k % 2 == 0 and k >= 8:
            k //= 2
        if n % 2 == 0 and k <= 13:
            return n
        n -= 2


# ---- inputs ------------------------------------------------------------------


def _eps(case, rng, n, m):
    a, b = 1.0, case["b"]
    if case["eps"] == "const":
        return pbs_inputs.const_eps(n, m, float(rng.uniform(1.0, 4.0)))
    if case["eps"] == "disks":
        return pbs_inputs.disks_eps(n, m, seed=int(rng.integers(1 << 30)), ndisks=6, a=a, b=b)
    r = float(rng.uniform(0.18, 0.3)) * min(a, b)
    return pbs_inputs.rod_eps(n, m, a, b, radius=r, eps_rod=float(rng.uniform(6.0, 13.0)),
                              centre=(float(rng.uniform(0, a)), float(rng.uniform(0, b))))


def _path(case, nk):
    """`nk` Bloch vectors spread evenly over the inside of Gamma-X-M-Gamma."""
    fine = pbs_inputs.gxmg_path(3 * 64 + 1, 1.0, case["b"])
    at = ((np.arange(nk) + 0.5) / nk * 192).astype(int)
    return fine[at]


def _opts(case):
    return dict(nev=case["nev"], block=case["block"], precision=FP64 if case["fp64"] else MIXED, tol=TOL,
                kbatch=case.get("kbatch", 1))


def _block(gen, cols, length):
    x = torch.randn(cols, length, 2, dtype=torch.float64, device="cuda", generator=gen)
    return torch.view_as_complex(x)


def _lengths(case):
    """Input and output length of an operator on the finest mesh."""
    N, D = case["n"] * case["m"], 2 * case["n"] * case["m"]
    node = {"L": (N, D), "LH": (D, N), "LH_M": (D, N), "P_NODAL": (N, N), "VCYCLE_NODAL": (N, N)}
    return node.get(case["op"], (D, D))


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed % (1 << 31))
    kind, n, m, b = case["kind"], case["n"], case["m"], case["b"]
    s = dict(case=case, ctx=pbs.Context(0))
    if kind == "serve":
        sizes = [(n, n) if j % 2 == 0 else (m, m) for j in range(case["jobs"])]
        s["geoms"] = [pbs.Geometry(_eps(case, rng, *z), 1.0, b) for z in sizes]
        s["ks"] = _path(case, case["nk"])
        s["opts"] = pbs.default_opts(**_opts(case))
        return s
    s["geom"] = pbs.Geometry(_eps(case, rng, n, m), 1.0, b)
    s["k"] = (math.pi * float(rng.uniform(0.3, 0.9)), math.pi / b * float(rng.uniform(0.1, 0.7)))
    if kind in ("solve_k", "path", "grid"):
        s["opts"] = pbs.default_opts(**_opts(case))
        if kind == "solve_k":
            s["init"] = pbs_inputs.random_block(2 * n * m, case["block"], seed=seed)
        elif kind == "path":
            s["ks"] = _path(case, case["nk"])
        return s
    prec = FP64 if case["fp64"] else MIXED
    if kind == "apply":
        li, lo = _lengths(case)
        s["x"] = _block(gen, case["cols"], li)
        s["y"] = torch.empty(case["cols"], lo, dtype=torch.complex128, device="cuda")
        s["opts"] = pbs.default_opts(precision=prec)
        return s
    q = case["q"]
    s["S"] = _block(gen, q, 2 * n * m)
    if kind == "gram":
        # trial columns of a search span many scales
        s["S"] *= torch.logspace(0, -6, q, dtype=torch.float64, device="cuda")[:, None]
        s["GM"] = torch.empty(q, q, dtype=torch.complex128, device="cuda")
        s["GA"] = torch.empty(q, q, dtype=torch.complex128, device="cuda")
        s["prec"] = prec
    elif kind == "rr":
        s["X"] = torch.empty(case["p"], 2 * n * m, dtype=torch.complex128, device="cuda")
        s["opts"] = pbs.default_opts(precision=prec)
    else:
        s["E"] = torch.empty(q, 2 * n * m, dtype=torch.complex128, device="cuda")
        s["R"] = torch.empty(q, q, dtype=torch.complex128, device="cuda")
    return s


def _solved(geom, lam, res):
    """The eigenvalues, and which bands met the stopping rule of pbs_opts.tol."""
    h1, h2 = geom.a / geom.n, geom.b / geom.m
    top = 12.0 * (1.0 / h1**2 + 1.0 / h2**2) / float(geom.eps.min())
    return dict(eigvals=lam, converged=(res <= np.maximum(TOL, 0.5 * 2.0**-53 * top / np.abs(lam))).astype(np.int8))


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind = case["kind"]
    if kind == "solve_k":
        lam, res, _, _ = ctx.solve_k(s["geom"], s["opts"], s["k"], init=s["init"])
        return _solved(s["geom"], lam, res)
    if kind == "path":
        lam, res, _ = ctx.solve_path(s["geom"], s["opts"], s["ks"])
        return _solved(s["geom"], lam, res)
    if kind == "grid":
        _, lam, res, _ = ctx.solve_grid(s["geom"], s["opts"], case["kappa"])
        return _solved(s["geom"], lam, res)
    if kind == "serve":
        jobs = [ctx.submit(g, s["opts"], s["ks"]) for g in s["geoms"]]
        got = [ctx.fetch(j) for j in jobs]
        return [_solved(g, lam, res) for g, (lam, res, _, _) in zip(s["geoms"], got)]
    stream = torch.cuda.current_stream()
    if kind == "apply":
        ctx.apply(s["geom"], case["op"], s["x"].data_ptr(), s["y"].data_ptr(), case["cols"], s["k"], 0, s["opts"],
                  stream)
        return s["y"]
    if kind == "gram":
        ctx.gram(s["geom"], s["k"], case["q"], s["S"].data_ptr(), s["GM"].data_ptr(), s["GA"].data_ptr(), stream,
                 s["prec"])
        return s["GM"], s["GA"]
    if kind == "rr":
        theta = ctx.rayleigh_ritz(s["geom"], s["opts"], s["k"], case["q"], s["S"].data_ptr(), case["p"],
                                  case["project"], s["X"].data_ptr(), stream)
        return theta, s["X"]
    ctx.m_householder(s["geom"], s["k"], case["q"], s["S"].data_ptr(), s["E"].data_ptr(), s["R"].data_ptr(), stream)
    return s["E"], s["R"]


def work(case):
    kind, D = case["kind"], 2.0 * case["n"] * case["m"]
    if kind in ("solve_k", "path", "grid", "serve"):
        # an iteration reads and writes its trial block [E, P, W] once; a dozen iterations per Bloch vector
        nk = {"solve_k": 1, "grid": case.get("kappa", 1) ** 2}.get(kind, case.get("nk", 1))
        if kind == "serve":
            D = case["n"] ** 2 + case["m"] ** 2  # the mean of the jobs' meshes
            nk *= case["jobs"]
        p = case["block"]
        return dict(bytes=12.0 * nk * 6 * p * 16.0 * D, flops=12.0 * nk * 8.0 * D * (1.5 * 9 * p * p + 3 * p * p))
    if kind == "apply":
        li, lo = _lengths(case)
        return dict(bytes=16.0 * (li + lo) * case["cols"] + 8.0 * D / 2, flops=8.0 * (li + lo) * case["cols"])
    q = case["q"]
    if kind == "gram":
        return dict(bytes=16.0 * D * q + 32.0 * q * q + 4.0 * D, flops=8.0 * 1.5 * D * q * (q + 1) / 2)
    if kind == "rr":
        return dict(bytes=16.0 * D * (q + case["p"]) + 4.0 * D,
                    flops=8.0 * D * (1.5 * q * (q + 1) / 2 + q * case["p"]))
    return dict(bytes=32.0 * D * q + 16.0 * q * q, flops=8.0 * D * 2.0 * q * q)


# ---- the same in plain 64-bit torch --------------------------------------------


def _roll(f, di, dj, k, b):
    """f(i + di, j + dj) of fields of shape (cols, m, n), continued with the Bloch phases of the unit x b cell."""
    al, be = complex(math.cos(k[0]), math.sin(k[0])), complex(math.cos(k[1] * b), math.sin(k[1] * b))
    if di:
        f = torch.roll(f, -di, 2)
        f = f.clone()
        if di > 0:
            f[:, :, -1] *= al
        else:
            f[:, :, 0] *= al.conjugate()
    if dj:
        f = torch.roll(f, -dj, 1)
        f = f.clone()
        if dj > 0:
            f[:, -1, :] *= be
        else:
            f[:, 0, :] *= be.conjugate()
    return f


class _Cell:
    """Mass, curl and gradient stencils of the edge discretisation on (cols, 2, m, n) blocks."""

    def __init__(self, eps, b, k):
        self.m, self.n = eps.shape
        self.b, self.k = b, k
        h1, h2 = 1.0 / self.n, b / self.m
        self.w = torch.as_tensor(1.0 / (eps * h1 * h2))
        self.mx, self.my = h2 / h1, h1 / h2

    def to(self, device):
        self.w = self.w.to(device)
        return self

    def split(self, X):
        X = X.reshape(X.shape[0], 2, self.m, self.n)
        return X[:, 0], X[:, 1]

    def roll(self, f, di, dj):
        return _roll(f, di, dj, self.k, self.b)

    def mass(self, X):
        x, y = self.split(X)
        mx = self.mx * (2.0 / 3.0 * x + 1.0 / 6.0 * (self.roll(x, 0, 1) + self.roll(x, 0, -1)))
        my = self.my * (2.0 / 3.0 * y + 1.0 / 6.0 * (self.roll(y, 1, 0) + self.roll(y, -1, 0)))
        return torch.stack([mx, my], 1).reshape(X.shape)

    def curl(self, X):
        x, y = self.split(X)
        return (self.roll(x, 0, 1) - x - self.roll(y, 1, 0) + y).reshape(X.shape[0], -1)

    def curl_adj(self, T):
        t = T.reshape(T.shape[0], self.m, self.n)
        return torch.stack([self.roll(t, 0, -1) - t, t - self.roll(t, -1, 0)], 1).reshape(T.shape[0], -1)

    def stiff(self, X):
        return self.curl_adj(self.curl(X) * self.w.reshape(-1))

    def lift(self, F):
        f = F.reshape(F.shape[0], self.m, self.n)
        return torch.stack([self.roll(f, 1, 0) - f, self.roll(f, 0, 1) - f], 1).reshape(F.shape[0], -1)

    def lift_adj(self, X):
        x, y = self.split(X)
        return (self.roll(x, -1, 0) - x + self.roll(y, 0, -1) - y).reshape(X.shape[0], -1)


def _bands(eps, b, k, nev):
    """The nev smallest non-zero eigenvalues, from the dense cell operator W^1/2 C M^-1 C^* W^1/2."""
    cell = _Cell(eps, b, k)
    N = cell.n * cell.m
    root = cell.w.reshape(-1).sqrt()
    C = cell.curl_adj(torch.diag(root).to(torch.complex128))  # rows: (C^* W^1/2) e_c
    Z = C.reshape(N, 2, cell.m, cell.n)

    # M is a one-dimensional periodic matrix along each line of edges: solve it by its dense inverse
    def line(size, phase, scale):
        A = torch.zeros(size, size, dtype=torch.complex128)
        for i in range(size):
            A[i, i] += 2.0 / 3.0
            A[i, (i + 1) % size] += phase / 6.0 if i + 1 == size else 1.0 / 6.0
            A[i, (i - 1) % size] += phase.conjugate() / 6.0 if i == 0 else 1.0 / 6.0
        return torch.linalg.inv(scale * A)

    al, be = complex(math.cos(k[0]), math.sin(k[0])), complex(math.cos(k[1] * b), math.sin(k[1] * b))
    Y = torch.stack([torch.einsum("jl,cli->cji", line(cell.m, be, cell.mx), Z[:, 0]),
                     torch.einsum("il,cjl->cji", line(cell.n, al, cell.my), Z[:, 1])], 1).reshape(N, -1)
    K = C.conj() @ Y.T
    lam = torch.linalg.eigvalsh((K + K.conj().T) / 2).numpy()
    return lam[:nev].copy()


def exact(case, seed):
    kind, n, m, b = case["kind"], case["n"], case["m"], case["b"]
    rng = np.random.default_rng(seed)
    if kind == "serve":
        return None
    eps = _eps(case, rng, n, m)
    k = (math.pi * float(rng.uniform(0.3, 0.9)), math.pi / b * float(rng.uniform(0.1, 0.7)))
    if kind in ("solve_k", "path", "grid"):
        ks = [k] if kind == "solve_k" else _path(case, case["nk"]) if kind == "path" else []
        if not len(ks) or n * m > 1536 or len(ks) > 3:
            return None
        lam = np.array([_bands(eps, b, tuple(v), case["nev"]) for v in ks])
        return dict(eigvals=lam[0] if kind == "solve_k" else lam, converged=None)
    gen = torch.Generator(device="cuda").manual_seed(seed % (1 << 31))
    cell = _Cell(eps, b, k).to("cuda")
    if kind == "apply":
        x = _block(gen, case["cols"], _lengths(case)[0])
        mu = 1.0 / b
        f = {"A": cell.stiff, "M": cell.mass, "A_MU_M": lambda v: cell.stiff(v) + mu * cell.mass(v), "L": cell.lift,
             "LH": cell.lift_adj, "LH_M": lambda v: cell.lift_adj(cell.mass(v)),
             "P_NODAL": lambda v: cell.lift_adj(cell.mass(cell.lift(v))),
             "RESIDUAL": lambda v: cell.stiff(v) - mu * cell.mass(v)}.get(case["op"])
        return f(x) if f else None
    q = case["q"]
    S = _block(gen, q, 2 * n * m)
    if kind == "gram":
        if n * m * q > 4.0e7:
            return None
        S *= torch.logspace(0, -6, q, dtype=torch.float64, device="cuda")[:, None]
        T = cell.curl(S)
        # row b of the result holds column b of the column-major matrix: entry a is s_a^* M s_b
        return cell.mass(S) @ S.conj().T, (T * cell.w.reshape(-1)) @ T.conj().T
    if kind == "rr":
        if case["project"] or n * m * q > 1.0e7:
            return None
        T = cell.curl(S)
        GM, GA = (S.conj() @ cell.mass(S).T).cpu(), (T.conj() @ (T * cell.w.reshape(-1)).T).cpu()
        Li = torch.linalg.inv(torch.linalg.cholesky((GM + GM.conj().T) / 2))
        H = Li @ GA @ Li.conj().T
        return torch.linalg.eigvalsh((H + H.conj().T) / 2)[: case["p"]].numpy(), None
    # Householder: the reflections of the block, one after the other
    if n * m * q > 1.0e7:
        return None
    scale = math.sqrt(2.0 / 3.0 * cell.mx)
    piv = [(2 * (t // n)) * n + t % n for t in range(q)]
    Y, R, V = S.clone(), torch.zeros(q, q, dtype=torch.complex128, device="cuda"), []
    for i in range(q):
        y = Y[i : i + 1]
        for _ in range(2):
            if i:
                c = cell.mass(y)[0, piv[:i]] / scale
                R[i, :i] += c
                y[0, piv[:i]] -= c / scale
        My = cell.mass(y)
        nrm = float((y.conj() * My).sum().real) ** 0.5
        g = complex(My[0, piv[i]]) / scale
        sigma = -nrm * g / abs(g)
        R[i, i] = sigma
        y[0, piv[i]] -= sigma / scale
        v = y.clone()
        V.append((v, 2.0 * nrm * nrm + 2.0 * nrm * abs(g)))
        if i + 1 < q:
            Y[i + 1 :] -= (2.0 / V[i][1]) * (Y[i + 1 :] @ cell.mass(v).conj().T) * v
    E = torch.zeros_like(S)
    for t in range(q):
        E[t, piv[t]] = 1.0 / scale
    for v, vmv in reversed(V):
        E -= (2.0 / vmv) * (E @ cell.mass(v).conj().T) * v
    return E, R
