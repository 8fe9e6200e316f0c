"""GPU: numbers of the fixed-point FP64 operators at the edges of their scales.

Tolerance of the operator comparisons: as tests/test_gpu_local_fx.py (1e-12 of the largest entry).
"""
import numpy as np
import pytest

from tests.gpu_util import rel_err, to_dev
from tests.oracle_systems import mini_system, sym_random
from tests.test_gpu_local_fx import TOL, _fe, _oracle, _system

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p", [1, 4, 6, 8])
@pytest.mark.parametrize("size", [1.0 - 2.0 ** -45, 1.0 - 2.0 ** -33, 1.0 - 2.0 ** -31, 2.0 ** 20 * (1.0 - 2.0 ** -34)])
def test_point_potentials_just_below_a_power_of_two(p, size):
    """One point of a cell holds its largest value, positive, and V or the weighted w V there lies just
    below a power of two, where the high limb of a coefficient is at its limit (both signs)."""
    import torch
    from oracle import fe as F
    from oracle import ops as O
    op, fe = _oracle(p), _fe(p)
    g = F.gauss_rule(p + 2)[1]
    w = (op.mesh.detJ * g[:, None, None] * g[None, :, None] * g[None, None, :]).reshape(-1)
    X = np.random.default_rng(p).standard_normal((op.mesh.ndof, 3))
    V = np.zeros(op.Vq.shape)
    nq = V.shape[1]
    V[0, 0], V[3, nq // 2] = size, size
    V[5, 1], V[6, nq - 1], V[8, 2] = size / w[1], size / w[nq - 1], -size / w[2]
    fe.set_veff(torch.from_numpy(V).cuda())
    assert rel_err(fe.apply_H(to_dev(X)).cpu().numpy(), O.PawOperators(_system(p), Vq=V).apply_H(X)) < TOL
    fe.close()


@pytest.mark.parametrize("p", [2, 4, 6, 8])
def test_small_entries_at_cell_corners(p):
    """Errors relative to each entry, down to the corners of a cell, whose rows are far smaller than
    those in its middle.  A product vector f(x) f(y) f(z) inside one cell gives S X = mu mu mu and
    K X = delta mu mu + mu delta mu + mu mu delta there, so the lines through the middle node predict every
    other entry, whatever the 1D matrices are.

    Tolerance: three to five contractions, each exact to two units of 2^-59 of the scaled range,
    of which an entry takes at least 2^-5 (2^-3 for the row sizes left by the row scales, 2^-2 for the
    others): 10 * 2^-59 * 2^5 = 5.6e-16, with the rounding of the output 7e-16; a prediction uses four
    such entries besides its own: 3.5e-15 of the sum of magnitudes."""
    import torch
    import paper_2604_26037_gb300 as P
    from oracle import fe as F
    s = dict(_system(p), natoms=0, positions=np.zeros((0, 3)), D=None, dS=None)
    fe = P.PawFE.from_system(s)
    N1, n, m, ncol, tol = 3 * p, p + 1, p // 2, 40, 3.5e-15
    fe.set_veff(torch.zeros((27, (p + 2) ** 3), dtype=torch.float64, device="cuda"))
    f = np.zeros((N1, ncol))
    f[1:p] = np.random.default_rng(p).integers(2 ** 16, 2 ** 17, (p - 1, ncol)) * (-1.0) ** np.arange(p - 1)[:, None]
    X = np.einsum("kv,jv,iv->kjiv", f, f, f).reshape(-1, ncol)       # 51 bits: exact
    S, H = (c(to_dev(X)).cpu().numpy().reshape(N1, N1, N1, ncol)[:n, :n, :n].astype(np.longdouble)
            for c in (fe.apply_S, fe.apply_H))
    fe.close()
    x = F.Mesh(7.5, 3, p).xi
    M = np.einsum("q,qa,qb->ab", F.gauss_rule(n)[1], *2 * [F.lagrange(x, F.gauss_rule(n)[0])[0]])
    mu = [S[:, m, m] / S[m, m, m], S[m, :, m] / S[m, m, m], S[m, m, :] / S[m, m, m]]
    am = [np.abs(M) @ np.abs(f[:n]) / np.abs(M[m] @ f[:n])] * 3     # sums of magnitudes of mu
    line = lambda a, b, c: np.einsum("kv,jv,iv->kjiv", a, b, c)
    assert (np.abs(S - line(*mu) * S[m, m, m]) / np.abs(line(*am) * S[m, m, m])).max() < tol
    d0 = H[m, m, m] / 3
    Hm = [H[:, m, m], H[m, :, m], H[m, m, :]]
    de = [h - 2 * u * d0 for h, u in zip(Hm, mu)]
    ad = [np.abs(h) + 2 * u * np.abs(d0) for h, u in zip(Hm, am)]
    three = lambda d, u: line(d[0], u[1], u[2]) + line(u[0], d[1], u[2]) + line(u[0], u[1], d[2])
    assert (np.abs(H - three(de, mu)) / three(ad, am)).max() < tol


def test_many_coefficients_of_both_signs():
    """S (-X) = -S X with 190 atoms on every cell: coefficients of 64 batches, whose sums are rounded
    one by one into 64 bits.  Rounding to nearest has no sign: what is left are FP64 additions of the
    eight cells of a node in another order, 16 * 2^-53 of the largest entry of a column."""
    import paper_2604_26037_gb300 as P
    rng = np.random.default_rng(12)
    s = mini_system(L=5.0, n=2, p=3, positions=rng.uniform(0.0, 5.0, (190, 3)),
                    shells=[(0, 0.36), (0, 0.3), (1, 0.36), (1, 0.33), (2, 0.36), (2, 0.3)],
                    D=sym_random(rng, 190, 18, 0.1), dS=sym_random(rng, 190, 18, 0.01), vdepth=1.0)
    fe = P.PawFE.from_system(s)
    X = to_dev(rng.standard_normal((fe.ndof, 33)))
    Y, Z = fe.apply_S(X).cpu().numpy(), fe.apply_S(-X).cpu().numpy()
    fe.close()
    assert (np.abs(Y + Z).max(0) / np.abs(Y).max(0)).max() <= 16 * 2.0 ** -53


@pytest.mark.parametrize("p", [3, 4, 6])
def test_vectors_that_grow_where_projectors_fall(p):
    """The projection of X = 1 / P on one cell, in which P falls by orders of magnitude, against the sum
    of the projections of its single entries; both are read from S X on nodes that the local part does
    not reach.  One projector, and all products have one sign.

    Tolerance: on either side at most a 2^-53 for the digits of X, the projection, the coupling (two),
    the digits of W and the expansion each: 12 * 2^-53 of the result."""
    import paper_2604_26037_gb300 as P
    s = mini_system(L=12.5, n=5, p=p, positions=[[6.25, 6.25, 6.25]], shells=[(0, 0.8)], D=np.full((1, 1, 1), 0.1),
                    dS=np.full((1, 1, 1), 0.5))
    fe = P.PawFE.from_system(s)
    N1, own = 5 * p, p ** 3
    cell = np.stack(np.meshgrid(*3 * [np.arange(p)], indexing="ij"), -1).reshape(-1, 3)[:, ::-1] + [2 * p, 2 * p, p]
    dof = cell @ [1, N1, N1 * N1]                          # the owned nodes of the cell (2, 2, 1)
    far = (2 * p + 1) + N1 * (2 * p + 1) + N1 * N1 * (3 * p + 1)   # a node of the cell (2, 2, 3)
    E = np.zeros((fe.ndof, own + 1))
    E[dof, np.arange(own)] = 1.0
    row = fe.apply_S(to_dev(E)).cpu().numpy()[far, :own]   # P(far) dS P(o)
    live = row != 0.0
    x = np.where(live, 1.0 / np.where(live, row, 1.0), 0.0)
    assert np.abs(row[live]).max() > 1e3 * np.abs(row[live]).min()
    E[dof, np.arange(own)] = x
    E[dof, own] = x
    Y = fe.apply_S(to_dev(E)).cpu().numpy()[far].astype(np.longdouble)
    fe.close()
    assert np.abs(Y[own] / Y[:own].sum() - 1) < 12 * 2.0 ** -53


@pytest.mark.parametrize("nproj", [4, 18])
@pytest.mark.parametrize("ncols", [1, 32, 33])
def test_one_owned_node_per_cell(nproj, ncols):
    """Degree 1, whose projector contractions are FP64 FMAs: every output stage against the oracle, with
    atoms on every cell and none, and values on nodes without projectors left out (FP64 tolerances of the
    other degrees)."""
    import paper_2604_26037_gb300 as P
    from oracle import cheb
    from oracle import ops as O
    rng = np.random.default_rng(nproj + ncols)
    shells = [(0, 0.5), (1, 0.45)] if nproj == 4 else [(0, 0.5), (0, 0.4), (1, 0.5), (1, 0.45), (2, 0.5), (2, 0.4)]
    for n, na in ((6, 20), (9, 2)):
        s = mini_system(L=1.5 * n, n=n, p=1, positions=rng.uniform(0.0, 1.5 * n, (na, 3)), shells=shells, vdepth=1.0,
                        D=sym_random(rng, na, nproj, 0.1), dS=sym_random(rng, na, nproj, 0.005))
        op, fe = O.PawOperators(s), P.PawFE.from_system(s, block=64)
        X, lam, b = rng.standard_normal((op.mesh.ndof, ncols)), np.linspace(0.1, 0.9, ncols), (0.0, 1.0, 60.0)
        Xd = to_dev(X)
        assert rel_err(fe.apply_H(Xd).cpu().numpy(), op.apply_H(X)) < TOL
        assert rel_err(fe.apply_S(Xd).cpu().numpy(), op.apply_S(X)) < TOL
        assert rel_err(fe.apply_Sinv_approx(Xd).cpu().numpy(), op.apply_Sinv_approx(X)) < TOL
        ref = cheb.rchfsi_filter(op.apply_H, op.apply_S, op.apply_Sinv_approx, X, lam, 4, *b)
        assert rel_err(fe.cheb_filter(Xd, lam, 4, b, prec="fp64").cpu().numpy(), ref) < 1e-10
        fe.close()
