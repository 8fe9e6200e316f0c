"""GPU parity of the fixed-point local operator (csrc/sumfac.cu) where its scales and tiles change.

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
