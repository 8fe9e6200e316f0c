"""Workloads whose speed matters to a user of the library, through its public entry points.

The library filters blocks of Kohn-Sham vectors (paw_cheb_filter) and applies the operators that
the eigensolver around it needs; a user's program creates one handle per problem (or a batch of
them), keeps it, and calls it with new vectors.  Sizes follow the repository's own workloads (tiny,
mid, prof12, grad16, batch32, degrees 4 to 6, 13 projectors per atom, block widths 32 to 512).

Vectors are what the solver holds after its first steps: the lowest plane waves of the box, each
with a few per cent of noise, with eigenvalue estimates near their kinetic energies.

exact() restates the discretisation with assembled one-dimensional matrices (the mesh is a uniform
periodic cube, so every integral over Gauss points is a tensor product) and dense projectors.
"""
import math
import random

import numpy as np
import torch

import paper_2604_26037_gb300 as paw

SHELLS = {
    # the two shells of the tiny workload, the five of all others (l, Gaussian width in bohr)
    4: [(0, 0.8), (1, 0.8)],
    13: [(0, 0.6), (0, 1.2), (1, 0.75), (1, 1.05), (2, 0.9)],
}
H_CELL = 2.5                                    # bohr, the cell size of every workload
TRUNC = math.sqrt(2.0 * math.log(1e8))          # projector cut-off radius / width


# ------------------------------------------------------------------------------------------ cases

def listed():
    return [
        # one vector on a very small problem: an operator call inside a user's own iterative solver
        dict(name="apply_H_one_vector_fp64", kind="apply", op="H", prec="fp64", n=4, p=4, atoms=2, nproj=4, ncols=1),
        # the smallest filter call (workload tiny): a molecule in a small box, launch-bound
        dict(name="filter_tiny_tf32", kind="filter", prec="tf32", n=4, p=4, atoms=2, nproj=4, ncols=16, block=16,
             degree=20, k=0),
        # H on one block of the ordinary problem, as Rayleigh-Ritz and the filter's step 2 apply it
        dict(name="apply_H_block_fp64", kind="apply", op="H", prec="fp64", n=16, p=6, atoms=64, nproj=13, ncols=256),
        # the same in the filter's reduced precision
        dict(name="apply_H_block_tf32", kind="apply", op="H", prec="tf32", n=16, p=6, atoms=64, nproj=13, ncols=256),
        # the approximate inverse overlap on a ragged block (a preconditioner call)
        dict(name="apply_Sinv_ragged_tf32", kind="apply", op="Sinv", prec="tf32", n=12, p=6, atoms=27, nproj=13,
             ncols=130),
        # the ordinary filter call, the workload the library is quoted on (mid)
        dict(name="filter_mid_tf32", kind="filter", prec="tf32", n=16, p=6, atoms=64, nproj=13, ncols=512, block=256,
             degree=30, k=0),
        # the plain FP64 method on a moderate problem (the form that a cautious user selects)
        dict(name="filter_plain_fp64", kind="filter", prec="fp64", n=12, p=6, atoms=27, nproj=13, ncols=128,
             block=128, degree=5, k=0),
        # BF16 cell products, odd degree, a column count that no block width divides
        dict(name="filter_ragged_bf16", kind="filter", prec="bf16", n=10, p=5, atoms=24, nproj=13, ncols=301,
             block=128, degree=20, k=0),
        # a Bloch wavevector: complex vectors, two blocks
        dict(name="filter_bloch_tf32", kind="filter", prec="tf32", n=8, p=6, atoms=8, nproj=13, ncols=96, block=64,
             degree=15, k=1),
        # uneven independent problems in one call (workload batch32, fewer of them)
        dict(name="batch_uneven_tf32", kind="batch", prec="tf32", count=8, mix=5, degree=25),
        # residual norms of the Ritz vectors after a filter pass (the convergence check)
        dict(name="residuals_fp64", kind="residuals", prec="fp64", n=12, p=6, atoms=27, nproj=13, ncols=200),
        # gradient of tr(X^T H X) with respect to the potential and D_ij (workload grad16)
        dict(name="gradient_fp32", kind="gradient", prec="fp32", n=16, p=4, atoms=64, nproj=13, ncols=16),
    ]


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _mesh(rng, hi=16):
    n, p = rng.randint(4, hi), rng.choice((4, 5, 6))
    atoms = rng.randint(max(2, n ** 3 // 100), max(8, n ** 3 // 40))
    return dict(n=n, p=p, atoms=min(atoms, 64), nproj=13)


def draw(rng):
    """One more case: any entry point of the listed ones, on any mesh, width and degree of their range."""
    kind = rng.choice(("apply", "apply", "apply", "filter", "filter", "filter", "batch", "residuals", "gradient"))
    if kind == "batch":
        return dict(kind="batch", prec=rng.choice(("tf32", "bf16")), count=rng.randint(2, 8), mix=rng.randint(0, 10 ** 6),
                    degree=rng.randint(10, 25))
    if kind == "apply":
        op = rng.choice(("H", "S", "Sinv"))
        prec = "fp64" if op == "S" else rng.choice(("fp64", "tf32"))
        return dict(kind="apply", op=op, prec=prec, ncols=_spread(rng, 1, 256), **_mesh(rng))
    if kind == "residuals":
        return dict(kind="residuals", prec="fp64", ncols=_spread(rng, 4, 256), **_mesh(rng, 12))
    if kind == "gradient":
        return dict(kind="gradient", prec=rng.choice(("fp32", "fp64")), ncols=_spread(rng, 4, 64), **_mesh(rng))
    form = rng.choice(("tf32", "tf32", "bf16", "fp64", "bloch"))
    block = rng.choice((32, 64, 128, 256))
    if form in ("fp64", "bloch"):
        return dict(kind="filter", prec="fp64" if form == "fp64" else "tf32", ncols=_spread(rng, 8, 128), block=block,
                    degree=rng.randint(4, 8 if form == "fp64" else 15), k=int(form == "bloch"), **_mesh(rng, 10))
    return dict(kind="filter", prec=form, ncols=_spread(rng, 16, 512), block=block, degree=rng.randint(8, 30), k=0,
                **_mesh(rng))


# ---------------------------------------------------------------------------------------- systems

def _kvec(case):
    return (0.05, 0.03, 0.02) if case.get("k") else None


def _widths(case):
    """The shells, narrowed where a cut-off radius would reach half of a small box."""
    shells = SHELLS[case["nproj"]]
    L = H_CELL * case["n"]
    wide = max(w for _, w in shells) * TRUNC
    s = min(1.0, (0.45 if case["nproj"] == 13 else 0.49) * L / wide)
    return [(l, w * s) for l, w in shells]


def _system(case, seed):
    """Positions on a jittered lattice, symmetric couplings, one Gaussian well per atom."""
    rng = np.random.default_rng([int(seed), 1])
    n, na, npj, L = case["n"], case["atoms"], case["nproj"], H_CELL * case["n"]
    g = 1
    while g ** 3 < na:
        g += 1
    sites = rng.permutation(g ** 3)[:na]
    pos = (np.stack([sites % g, sites // g % g, sites // (g * g)], 1) + 0.5) * (L / g)
    pos = np.mod(pos + rng.uniform(-1.0, 1.0, (na, 3)) * min(0.3, 0.1 * L / g), L)

    def sym(sigma):
        u = np.triu(rng.normal(0.0, sigma, (na, npj, npj)))
        return u + np.triu(u, 1).transpose(0, 2, 1)

    return dict(L=L, ncell=n, p=case["p"], positions=pos, shells=_widths(case), D=sym(0.1), dS=sym(0.02),
                vloc_centers=pos, vloc_depth=np.full(na, 2.0), vloc_width=np.full(na, 1.0))


def _gll(p):
    """Gauss-Lobatto-Legendre nodes and weights."""
    P = np.polynomial.legendre.Legendre.basis(p)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
    return x, 2.0 / (p * (p + 1) * P(x) ** 2)


def _lagrange(nodes, x):
    """Values and derivatives of the Lagrange polynomials on the nodes, (len(x), len(nodes))."""
    V = np.polynomial.legendre.legvander(nodes, len(nodes) - 1)
    C = np.linalg.inv(V)
    f = np.polynomial.legendre.legvander(x, len(nodes) - 1)
    d = np.stack([np.polynomial.legendre.Legendre.basis(i).deriv()(x) if i else np.zeros_like(x)
                  for i in range(len(nodes))], 1)
    return f @ C, d @ C


def _upper(p, h):
    """Upper end of the spectrum from the largest kinetic eigenvalue of one cell, with a margin."""
    x, wl = _gll(p)
    g, w = np.polynomial.legendre.leggauss(p + 1)
    _, d = _lagrange(x, g)
    s = 1.0 / np.sqrt(wl)
    mu = np.linalg.eigvalsh(s[:, None] * (d.T @ (w[:, None] * d)) * s[None, :])[-1]
    return 1.1 * 0.5 * 3.0 * (2.0 / h) ** 2 * mu


def _waves(case, ncols, seed, dtype, dev):
    """(X, eigenvalue estimates): the lowest plane waves on the nodes, each with noise of 3 per cent."""
    n, p, L = case["n"], case["p"], H_CELL * case["n"]
    N1, kv = n * p, np.array(_kvec(case) or (0.0, 0.0, 0.0))
    m = 1
    while (2 * m + 1) ** 3 < 3 * ncols + 30:
        m += 1
    G = np.array([(a, b, c) for a in range(-m, m + 1) for b in range(-m, m + 1) for c in range(-m, m + 1)])
    q = 2.0 * math.pi / L
    e = 0.5 * ((q * G + kv) ** 2).sum(1)
    G, e = G[np.argsort(e, kind="stable")[:ncols]], np.sort(e, kind="stable")[:ncols]
    x = _gll(p)[0]
    nodes = torch.tensor(((np.arange(n)[:, None] + (x[None, :-1] + 1.0) / 2.0) * (q * H_CELL)).reshape(-1), device=dev)
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed) * 7919 + 3)
    cplx = dtype.is_complex
    X = torch.empty((N1 ** 3, ncols), dtype=dtype, device=dev)
    amp = math.sqrt((1.0 if cplx else 2.0) / L ** 3)
    for j0 in range(0, ncols, 32):
        Gt = torch.tensor(G[j0:j0 + 32], dtype=torch.float64, device=dev)
        w = Gt.shape[0]
        ph = (nodes[:, None, None, None] * Gt[:, 2] + nodes[None, :, None, None] * Gt[:, 1]
              + nodes[None, None, :, None] * Gt[:, 0]).reshape(-1, w)
        shift = torch.rand(w, generator=gen, device=dev, dtype=torch.float64) * (2.0 * math.pi)
        f = torch.polar(torch.full_like(ph, amp), ph + shift) if cplx else amp * torch.cos(ph + shift)
        noise = torch.randn((N1 ** 3, w), generator=gen, device=dev, dtype=torch.complex128 if cplx else torch.float64)
        X[:, j0:j0 + w] = (f + (0.03 * math.sqrt(1.0 / L ** 3)) * noise).to(dtype)
    rng = np.random.default_rng([int(seed), 2])
    lam = np.sort(e - 0.2 + rng.normal(0.0, 0.01, ncols))
    return X, lam


def _bounds(case, lam):
    return (float(lam[0]) - 0.1, float(lam[-1]) + 0.4, _upper(case["p"], H_CELL))


def _batch_cases(case):
    """The instances of a batch: uneven meshes, degrees, atom counts and block widths."""
    r = random.Random(case["mix"])
    out = []
    for _ in range(case["count"]):
        n = r.randint(4, 9)
        out.append(dict(kind="filter", prec=case["prec"], n=n, p=r.choice((4, 5, 6)), nproj=13,
                        atoms=r.randint(8, min(64, max(8, int((H_CELL * n) ** 3 / 120)))),
                        ncols=r.choice((32, 64, 128, 256)), degree=case["degree"], k=0))
    return out


# -------------------------------------------------------------------------------------------- run

def _handle(case, seed, block=256):
    return paw.PawFE.from_system(_system(case, seed), block=block, kpoint=_kvec(case))


def prepare(case, seed):
    dev = torch.device("cuda")
    kind, prec = case["kind"], case["prec"]
    if kind == "batch":
        subs = _batch_cases(case)
        fes = [_handle(c, seed + 101 * i, c["ncols"]) for i, c in enumerate(subs)]
        problems = []
        for i, (c, fe) in enumerate(zip(subs, fes)):
            X, lam = _waves(c, c["ncols"], seed + 101 * i, torch.float64, dev)
            problems.append((X, lam, c["degree"], _bounds(c, lam), torch.empty_like(X)))
        return dict(kind=kind, prec=prec, fes=fes, problems=problems, batch=paw.PawBatch(fes, streams=4, autotune=True))
    st = dict(kind=kind, prec=prec, fe=_handle(case, seed, case.get("block", 256)))
    single = prec != "fp64" and kind in ("apply", "gradient")
    dtype = torch.complex128 if case.get("k") else torch.float32 if single else torch.float64
    X, lam = _waves(case, case["ncols"], seed, dtype, dev)
    st.update(X=X, lam=lam)
    if kind == "apply":
        st.update(op=case["op"], out=torch.empty_like(X))
    if kind == "filter":
        st.update(degree=case["degree"], bounds=_bounds(case, lam), out=torch.empty_like(X))
    return st


def run(state):
    kind, prec = state["kind"], state["prec"]
    if kind == "batch":
        state["batch"].cheb_filter(state["problems"], prec=prec)
        return [q[4] for q in state["problems"]]
    fe, X = state["fe"], state["X"]
    if kind == "apply":
        fn = {"H": fe.apply_H, "S": fe.apply_S, "Sinv": fe.apply_Sinv_approx}[state["op"]]
        return fn(X, state["out"], prec=prec)
    if kind == "filter":
        return fe.cheb_filter(X, state["lam"], state["degree"], state["bounds"], prec=prec, out=state["out"])
    if kind == "residuals":
        return fe.residuals(X, state["lam"])
    if kind == "gradient":
        return list(fe.energy_grad(X, prec=prec))
    raise ValueError(kind)


# ------------------------------------------------------------------------------------------- work

def _projector_entries(case):
    """Nonzero entries of the projectors on the nodes: shell by shell, the nodes of the cells that a
    cut-off sphere reaches (a sphere wider by half a cell)."""
    L, dens = H_CELL * case["n"], (case["p"] / H_CELL) ** 3
    tot = 0.0
    for l, w in _widths(case):
        tot += (2 * l + 1) * min(L ** 3, 4.0 / 3.0 * math.pi * (w * TRUNC + 0.5 * H_CELL) ** 3) * dens
    return case["atoms"] * tot


def _local_flops(p, q):
    """Flops of one cell and vector of the local operator as 1D contractions in even/odd halves."""
    a, b = p + 1, q
    interp = (a * a + a * b + b * b) * a * b           # (p+1)^3 nodes to Gauss points and back: twice this
    kinetic = 7 * a ** 4
    return (2 * interp + kinetic) * 2 * 0.5


def work(case):
    if case["kind"] == "batch":
        each = [work(c) for c in _batch_cases(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    n, p, nv = case["n"], case["p"], case["ncols"] * (2 if case.get("k") else 1)
    ndof, cells = (n * p) ** 3, n ** 3
    elem = 8 if case["prec"] == "fp64" or case["kind"] == "filter" else 4
    nl = 2.0 * _projector_entries(case) * nv           # one projector contraction
    local = _local_flops(p, p + 2) * cells * nv
    vq = 8.0 * cells * (p + 2) ** 3
    if case["kind"] == "apply":
        if case["op"] == "Sinv":
            return {"bytes": 2.0 * elem * ndof * nv, "flops": 2 * nl + ndof * nv}
        return {"bytes": 2.0 * elem * ndof * nv + vq, "flops": 2 * nl + local}
    if case["kind"] == "residuals":
        return {"bytes": 8.0 * ndof * nv + vq, "flops": 2 * nl + local}
    if case["kind"] == "gradient":
        return {"bytes": float(elem) * ndof * nv + 8.0 * cells * (p + 2) ** 3,
                "flops": nl + (_local_flops(p, p + 2) / 2 + 3 * (p + 2) ** 3) * cells * nv}
    # the filter: X once in and once out; every degree applies H and the approximate inverse overlap
    return {"bytes": 16.0 * ndof * nv + vq, "flops": case["degree"] * (3 * nl + local)}


# ------------------------------------------------------------------------------------------ exact

class _Dense:
    """The operators of one problem in 64 bits: assembled 1D matrices, dense projectors."""

    def __init__(self, case, seed, dev):
        sysd = _system(case, seed)
        n, p, L = case["n"], case["p"], sysd["L"]
        h = L / n
        kv = _kvec(case)
        x, wl = _gll(p)
        N1, q = n * p, p + 2
        idx = (np.arange(n)[:, None] * p + np.arange(p + 1)[None, :]) % N1

        def assemble(cell):
            A = np.zeros((N1, N1))
            for c in range(n):
                A[np.ix_(idx[c], idx[c])] += cell
            return A

        g1, w1 = np.polynomial.legendre.leggauss(p + 1)
        f1, d1 = _lagrange(x, g1)
        M, K = assemble(h / 2 * (f1.T @ (w1[:, None] * f1))), assemble(2 / h * (d1.T @ (w1[:, None] * d1)))
        C = assemble(f1.T @ (w1[:, None] * d1))        # int l_a dl_b/dx
        g2, w2 = np.polynomial.legendre.leggauss(q)
        f2, _ = _lagrange(x, g2)
        B = np.zeros((n * q, N1))
        for c in range(n):
            B[c * q:(c + 1) * q, idx[c]] += f2
        md = np.zeros(N1)
        np.add.at(md, idx.reshape(-1), np.tile(wl * h / 2, n))
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
        self.N1, self.M, self.K, self.C, self.B, self.k = N1, t(M), t(K), t(C), t(B), kv
        self.md = (t(md)[:, None, None] * t(md)[None, :, None] * t(md)[None, None, :]).reshape(-1, 1)
        pts = t(((np.arange(n)[:, None] + (g2[None, :] + 1) / 2) * h).reshape(-1))
        w = t(np.tile(w2 * h / 2, n))
        wq = w[:, None, None] * w[None, :, None] * w[None, None, :]

        def shifted(R, image=None):
            d = [pts - float(r) for r in R]
            if image is None:
                return [a - L * torch.round(a / L) for a in d]
            return [a - L * i for a, i in zip(d, image)]

        def grid(d):                                   # [z][y][x]
            return d[2][:, None, None], d[1][None, :, None], d[0][None, None, :]

        V = torch.zeros((n * q,) * 3, dtype=torch.float64, device=dev)
        for R, A, s in zip(sysd["vloc_centers"], sysd["vloc_depth"], sysd["vloc_width"]):
            rc = 8.0 * s
            m = math.ceil(rc / L)
            images = [None] if rc < L / 2 else [(a, b, c) for a in range(-m, m + 1) for b in range(-m, m + 1)
                                                for c in range(-m, m + 1)]
            for im in images:
                z, y, xx = grid(shifted(R, im))
                r2 = z * z + y * y + xx * xx
                V -= torch.where(r2 < rc * rc, A * torch.exp(-r2 / (2 * s * s)), 0.0)
        self.wV = (wq * V)[..., None]
        self.cplx = kv is not None
        P, sq = [], math.sqrt
        for R in sysd["positions"]:
            z, y, xx = grid(shifted(R))
            r2 = z * z + y * y + xx * xx
            cols = []
            for l, s in sysd["shells"]:
                nrm = sq(2.0 / (math.gamma(l + 1.5) * s ** (2 * l + 3)))
                rad = wq * torch.where(r2 < (s * TRUNC) ** 2, nrm * torch.exp(-r2 / (2 * s * s)), 0.0)
                if l == 0:
                    ang = [0.5 / sq(math.pi)]
                elif l == 1:
                    c = sq(3 / (4 * math.pi))
                    ang = [c * y, c * z, c * xx]
                else:
                    c1, c0, c2 = 0.5 * sq(15 / math.pi), 0.25 * sq(5 / math.pi), 0.25 * sq(15 / math.pi)
                    ang = [c1 * xx * y, c1 * y * z, c0 * (2 * z * z - xx * xx - y * y), c1 * xx * z,
                           c2 * (xx * xx - y * y)]
                cols += [rad * a for a in ang]
            f = torch.stack(cols, -1)
            if self.cplx:
                ph = (float(R @ np.array(kv)) + kv[0] * xx + kv[1] * y + kv[2] * z)[..., None]
                f = torch.polar(torch.ones_like(ph), -ph) * f
            P.append(self._tensor([self.B.T] * 3, f).reshape(N1 ** 3, -1))
        self.P = torch.cat(P, 1)
        self.na, self.npj = len(P), P[0].shape[1]
        cd = self.P.dtype
        self.D, self.dS = t(sysd["D"]).to(cd), t(sysd["dS"]).to(cd)
        G = torch.stack([a.conj().T @ (a / self.md) for a in P])
        self.Dinv = self.dS @ torch.linalg.inv(torch.eye(self.npj, dtype=cd, device=dev) + G @ self.dS)

    @staticmethod
    def _tensor(mats, f):
        """One matrix along each of z, y, x of f[z][y][x][column]."""
        for axis, A in enumerate(mats):
            f = torch.movedim(torch.tensordot(A.to(f.dtype), f, dims=([1], [axis])), 0, axis)
        return f

    def _by_columns(self, fn, X):
        X = X.reshape(self.N1, self.N1, self.N1, -1)
        return torch.cat([fn(X[..., j:j + 32].contiguous()).reshape(self.N1 ** 3, -1)
                          for j in range(0, X.shape[-1], 32)], 1)

    def _couple(self, mats, X, left=None):
        U = (self.P.conj().T @ X).reshape(self.na, self.npj, -1)
        return self.P @ (mats @ U).reshape(self.na * self.npj, -1)

    def H(self, X):
        K, M, T = self.K, self.M, self._tensor

        def local(f):
            y = 0.5 * (T([M, M, K], f) + T([M, K, M], f) + T([K, M, M], f))
            y = y + T([self.B.T] * 3, self.wV * T([self.B] * 3, f))
            if self.cplx:
                k, C = self.k, self.C
                y = y + 0.5 * sum(v * v for v in k) * T([M, M, M], f)
                y = y - 1j * (k[0] * T([M, M, C], f) + k[1] * T([M, C, M], f) + k[2] * T([C, M, M], f))
            return y

        return self._by_columns(local, X) + self._couple(self.D, X)

    def S(self, X):
        return self._by_columns(lambda f: self._tensor([self.M] * 3, f), X) + self._couple(self.dS, X)

    def Sinv(self, X):
        Z = X / self.md
        return Z - self._couple(self.Dinv, Z) / self.md

    def filter(self, X, lam, m, bounds):
        a0, bW, bU = bounds
        e, c = (bU - bW) / 2, (bU + bW) / 2
        z = z1 = e / (a0 - c)
        lam = torch.tensor(lam, device=X.device)
        Y = self.H(X) - self.S(X) * lam
        RX, RY, LX, LY = torch.zeros_like(X), z / e * Y, torch.ones_like(lam), z / e * (lam - c)
        for _ in range(2, m + 1):
            zn = 1.0 / (2.0 / z1 - z)
            al = 2 * zn / e
            RX, RY = RY, al * self.H(self.Sinv(RY)) - al * c * RY - z * zn * RX + al * Y * LY
            LX, LY = LY, al * LY * lam - al * c * LY - z * zn * LX
            z = zn
        return self.Sinv(RY) + X * LY


def _exact_one(case, seed, dev):
    kind = case["kind"]
    single = case["prec"] != "fp64" and kind in ("apply", "gradient")
    dtype = torch.complex128 if case.get("k") else torch.float32 if single else torch.float64
    X, lam = _waves(case, case["ncols"], seed, dtype, dev)
    X = X.to(torch.complex128 if case.get("k") else torch.float64)
    op = _Dense(case, seed, dev)
    if kind == "apply":
        return {"H": op.H, "S": op.S, "Sinv": op.Sinv}[case["op"]](X)
    if kind == "filter":
        return op.filter(X, lam, case["degree"], _bounds(case, lam))
    if kind == "residuals":
        return torch.linalg.vector_norm(op.H(X) - op.S(X) * torch.tensor(lam, device=dev), dim=0).cpu().numpy()
    n, q, N1 = case["n"], case["p"] + 2, op.N1
    rho = torch.zeros((n * q,) * 3, dtype=torch.float64, device=dev)
    for j in range(0, X.shape[1], 32):
        rho += (op._tensor([op.B] * 3, X[:, j:j + 32].reshape(N1, N1, N1, -1).contiguous()) ** 2).sum(-1)
    _, w2 = np.polynomial.legendre.leggauss(q)
    w = torch.tensor(np.tile(w2 * H_CELL / 2, n), device=dev)
    rho *= w[:, None, None] * w[None, :, None] * w[None, None, :]
    rho = rho.reshape(n, q, n, q, n, q).permute(0, 2, 4, 1, 3, 5).reshape(n ** 3, q ** 3)
    U = (op.P.T @ X).reshape(op.na, op.npj, -1)
    return [rho, U @ U.transpose(1, 2)]


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] == "batch":
        subs = _batch_cases(case)
        if sum(_cost(c) for c in subs) > 6e12:
            return None
        return [_exact_one(c, seed + 101 * i, dev) for i, c in enumerate(subs)]
    if _cost(case) > 6e12:
        return None
    return _exact_one(case, seed, dev)


def _cost(case):
    """Multiplications of exact(), real ones."""
    N1, Q1 = case["n"] * case["p"], case["n"] * (case["p"] + 2)
    nv = case["ncols"] * (4 if case.get("k") else 1)
    interp = N1 * Q1 * (N1 * N1 + N1 * Q1 + Q1 * Q1)
    one = 2 * interp + 12 * N1 ** 4 + 4 * N1 ** 3 * case["atoms"] * case["nproj"]
    return one * nv * (case["degree"] if case["kind"] == "filter" else 1)
