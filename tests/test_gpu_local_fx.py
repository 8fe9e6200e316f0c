"""GPU parity of the fixed-point FP64 operators (csrc/sumfac.cu, csrc/nonlocal_fx.cu) where their
scales and tiles change.

Tolerance: one application is seven one-dimensional contractions; each result is exact to about
two units of 2^-59 of the largest magnitude that the scales allow for (dropped low products and
one rounding), and for dense random cells that magnitude is at most 2^10 times the largest output
entry: 7 * 2 * 2^-59 * 2^10 = 2.5e-14 of the largest entry.  The oracle's own FP64 sums of up to
8 * 729 products reach 1e-13, so 1e-12 holds for both.
"""
import functools

import numpy as np
import pytest

from tests.gpu_util import rel_err, to_dev
from tests.oracle_systems import mini_system, sym_random

pytestmark = pytest.mark.gpu
TOL = 1e-12


@functools.lru_cache(maxsize=None)
def _system(p):
    rng = np.random.default_rng(60 + p)
    return mini_system(L=7.5, n=3, p=p, positions=[[2.2, 3.1, 4.4], [5.1, 5.7, 2.2]], shells=[(0, 0.5), (1, 0.4)],
                       D=sym_random(rng, 2, 4, 0.1), dS=sym_random(rng, 2, 4, 0.02), vdepth=2.0)


@functools.lru_cache(maxsize=None)
def _oracle(p):
    from oracle import ops as O
    return O.PawOperators(_system(p))


def _fe(p, **kw):
    import paper_2604_26037_gb300 as P
    return P.PawFE.from_system(_system(p), **kw)


@pytest.mark.parametrize("p", range(1, 9))
@pytest.mark.parametrize("ncols", [1, 4, 5, 17])
def test_degrees_and_column_tails(p, ncols):
    """Every degree; one vector, the last of the four-vector tiles, the first and a ragged one of eight."""
    op, fe = _oracle(p), _fe(p)
    X = np.random.default_rng(p).standard_normal((op.mesh.ndof, ncols))
    assert rel_err(fe.apply_H(to_dev(X)).cpu().numpy(), op.apply_H(X)) < TOL
    assert rel_err(fe.apply_S(to_dev(X)).cpu().numpy(), op.apply_S(X)) < TOL
    fe.close()


@pytest.mark.parametrize("p", [4, 6])
def test_scales_of_vectors_and_mass_term(p):
    """Vectors of very different sizes side by side, a zero one, and eigenvalue estimates from far
    below to far above the kinetic part (the mass term then needs room in the scales)."""
    op, fe = _oracle(p), _fe(p)
    X = np.random.default_rng(3).standard_normal((op.mesh.ndof, 12))
    X *= np.array([1, 1e-30, 1e30, 0, 1e-200, 1e200, 1, 1, 1, 1, 1, 1])
    lam = np.array([0, 1, 1, 1, 1, 1, 1e-12, 3e1, -1e3, 1e6, -1e12, 1e30])
    H, S = op.apply_H(X), op.apply_S(X)
    Hd = fe.apply_H(to_dev(X)).cpu().numpy()
    for j in range(12):
        if j == 3:
            assert not Hd[:, j].any()
        else:
            assert rel_err(Hd[:, j], H[:, j]) < TOL
    rms = np.array([np.abs(c).max() or 1.0 for c in X.T])
    ref = np.linalg.norm((H - S * lam) / rms, axis=0)
    Xn = to_dev(X / rms)
    r = fe.residuals(Xn, lam)
    assert r[3] == 0.0
    keep = np.arange(12) != 3
    assert np.abs(r[keep] / ref[keep] - 1.0).max() < TOL
    fe.close()


@pytest.mark.parametrize("p", [3, 6])
def test_potentials_from_zero_to_far_above_the_kinetic_part(p):
    """A potential of every size, alone in a few cells; a NaN stays in its cell."""
    import torch
    op, fe = _oracle(p), _fe(p)
    from oracle import ops as O
    rng = np.random.default_rng(8)
    X = rng.standard_normal((op.mesh.ndof, 9))
    Vq = np.zeros(op.Vq.shape)
    for e, size in ((0, 1e-9), (1, 1.0), (2, 1e3), (3, 1e8), (4, 1e15)):
        Vq[e] = size * rng.standard_normal(Vq.shape[1])
    for top in (1, 3, 5):
        V = Vq.copy()
        V[top:5] = 0.0
        fe.set_veff(torch.from_numpy(V).cuda())
        assert rel_err(fe.apply_H(to_dev(X)).cpu().numpy(), O.PawOperators(_system(p), Vq=V).apply_H(X)) < TOL
    V[7, 2] = np.nan
    fe.set_veff(torch.from_numpy(V).cuda())
    Y = fe.apply_H(to_dev(X)).cpu().numpy()
    inside = np.zeros(op.mesh.ndof, bool)
    inside[op.mesh.cell_dofs[7]] = True
    assert np.isnan(Y[inside]).all() and np.isfinite(Y[~inside]).all()
    fe.close()


def test_non_finite_vector_entries_reach_their_cells_only():
    op, fe = _oracle(4), _fe(4)
    X = np.random.default_rng(5).standard_normal((op.mesh.ndof, 6))
    dof = op.mesh.cell_dofs[13, 62]                       # an interior node of cell 13
    ref = op.apply_S(X)
    X[dof, 1], X[dof, 4] = np.inf, np.nan
    import paper_2604_26037_gb300 as P
    s = dict(_system(4), natoms=0, positions=np.zeros((0, 3)), D=None, dS=None)
    fe0 = P.PawFE.from_system(s)                          # without projectors: the local part alone
    Y = fe0.apply_S(to_dev(X)).cpu().numpy()
    inside = np.zeros(op.mesh.ndof, bool)
    inside[op.mesh.cell_dofs[13]] = True
    for j in (1, 4):
        assert (~np.isfinite(Y[inside, j])).all() and np.isfinite(Y[~inside, j]).all()
    assert np.isfinite(Y[:, [0, 2, 3, 5]]).all() and np.isfinite(ref).all()
    fe.close()
    fe0.close()


@pytest.mark.parametrize("p,natoms", [(3, 2), (6, 9), (7, 9), (8, 2)])
@pytest.mark.parametrize("ncols", [1, 16, 17, 35])
def test_digit_contractions(p, natoms, ncols):
    """The FP64 projector contractions on their own (the approximate inverse overlap and two steps of
    the FP64 recurrence): tiles of 16 and 32 vectors with tails, node counts that 16 does not
    divide, one batch of coefficients and two (nine atoms reach every cell of the small box), and
    vectors and coefficients of very different sizes.  Operands keep 55 bits of their column's
    largest entry, so an output is exact to a few 2^-53 of its largest entry."""
    from oracle import cheb
    from oracle import ops as O
    import paper_2604_26037_gb300 as P
    rng = np.random.default_rng(70 + p)
    pos = rng.uniform(0.0, 5.0, (natoms, 3))
    s = mini_system(L=5.0, n=2, p=p, positions=pos, shells=[(0, 0.4), (1, 0.35)], vdepth=1.0,
                    D=sym_random(rng, natoms, 4, 0.1), dS=sym_random(rng, natoms, 4, 0.005))
    op, fe = O.PawOperators(s), P.PawFE.from_system(s, block=max(ncols, 4))
    X = rng.standard_normal((op.mesh.ndof, ncols)) * np.exp(rng.uniform(-60.0, 60.0, ncols))
    Y, ref = fe.apply_Sinv_approx(to_dev(X)).cpu().numpy(), op.apply_Sinv_approx(X)
    F = fe.cheb_filter(to_dev(X), np.linspace(0.1, 0.9, ncols), 3, (0.0, 1.0, 400.0), prec="fp64").cpu().numpy()
    Fr = cheb.rchfsi_filter(op.apply_H, op.apply_S, op.apply_Sinv_approx, X, np.linspace(0.1, 0.9, ncols), 3, 0.0, 1.0,
                            400.0)
    for j in range(ncols):
        assert rel_err(Y[:, j], ref[:, j]) < TOL
        assert rel_err(F[:, j], Fr[:, j]) < TOL
    fe.close()


@pytest.mark.parametrize("p", [1, 2, 4, 6, 7, 8])
@pytest.mark.parametrize("ncols,prec", [(1, "fp64"), (9, "fp64"), (4, "fp32"), (33, "fp32")])
def test_density(p, ncols, prec):
    """Densities and occupation matrices with occupations of both signs; FP32 vectors enter exactly,
    their projector coefficients are FP32 sums (1e-5)."""
    import torch
    from oracle import grad
    op, fe = _oracle(p), _fe(p)
    rng = np.random.default_rng(10 * p + ncols)
    X, f = rng.standard_normal((op.mesh.ndof, ncols)), rng.uniform(-1.0, 2.0, ncols)
    Xd = to_dev(X, torch.float64 if prec == "fp64" else torch.float32)
    rho, D = grad.density(op, Xd.double().cpu().numpy(), f)
    r, d = fe.density(Xd, occ=f, prec=prec)
    assert rel_err(r.cpu().numpy(), rho) < TOL
    assert rel_err(d.cpu().numpy(), D) < (TOL if prec == "fp64" else 1e-5)
    fe.close()
