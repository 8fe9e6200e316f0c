"""GPU parity of tensor-core calls on blocks whose rows are not whole 16-byte pieces (padded copies
and zero columns inside the library) against the oracle.

Tolerances: those of the same calls on whole rows (tests/test_gpu_ops.py, tests/test_gpu_cheb.py):
operands are rounded to TF32 (unit roundoff 4.9e-4) or BF16 (3.9e-3), 4e-3 and 3e-2 of the largest
entry for one application, 2e-2 and 1e-1 for a filter of a few steps.  The approximate inverse
overlap rounds only its correction, a few per cent of the result: 1e-4.
"""
import functools

import numpy as np
import pytest

from tests.gpu_util import rel_err, to_dev
from tests.oracle_systems import mini_system, sym_random

pytestmark = pytest.mark.gpu


@functools.lru_cache(maxsize=None)
def _pair():
    """7^3 cells: more tiles than the SMs take twice over, where blocks of the filter are padded."""
    from oracle import ops as O
    import paper_2604_26037_gb300 as P
    rng = np.random.default_rng(41)
    s = mini_system(L=14.0, n=7, p=4, positions=[[2.5, 3.0, 4.0], [8.5, 9.0, 5.5], [6.1, 2.0, 11.5]],
                    shells=[(0, 0.6), (1, 0.7), (2, 0.6)], D=sym_random(rng, 3, 9, 0.1), dS=sym_random(rng, 3, 9, 0.02),
                    vdepth=2.0)
    return O.PawOperators(s), P.PawFE.from_system(s, block=32)


@pytest.mark.parametrize("prec,tol", [("tf32", 2e-2), ("bf16", 1e-1)])
@pytest.mark.parametrize("ncols", [1, 31, 37, 66])
def test_filter_blocks(prec, tol, ncols):
    """One ragged block, and ragged last blocks beside whole ones (overlapped schedule)."""
    from oracle import cheb
    op, fe = _pair()
    X = np.random.default_rng(ncols).standard_normal((op.mesh.ndof, ncols))
    lam, b = np.linspace(-0.3, 0.5, ncols), (-0.5, 0.6, 60.0)
    ref = cheb.rchfsi_filter(op.apply_H, op.apply_S, op.apply_Sinv_approx, X, lam, 5, *b)
    wide = to_dev(np.full((op.mesh.ndof, ncols + 5), 7.0))
    wide[:, 2:2 + ncols] = to_dev(X)
    out = wide.new_full((op.mesh.ndof, ncols + 3), 9.0)
    fe.cheb_filter(wide[:, 2:2 + ncols], lam, 5, b, prec=prec, out=out[:, 1:1 + ncols])
    got = out.cpu().numpy()
    assert rel_err(got[:, 1:1 + ncols], ref) < tol
    assert (got[:, 0] == 9.0).all() and (got[:, 1 + ncols:] == 9.0).all()


@pytest.mark.parametrize("ncols,off,extra", [(1, 0, 0), (6, 0, 0), (8, 1, 0), (8, 0, 1), (130, 3, 2), (517, 1, 0)])
def test_operators(ncols, off, extra):
    """Column counts, offsets and pitches that four does not divide, inside wider arrays."""
    import torch
    op, fe = _pair()
    X = np.random.default_rng(ncols + off).standard_normal((op.mesh.ndof, ncols))
    wide = torch.full((op.mesh.ndof, off + ncols + extra), 7.0, dtype=torch.float32, device="cuda")
    wide[:, off:off + ncols] = to_dev(X, torch.float32)
    for call, ref, tol in ((fe.apply_H, op.apply_H(X), 4e-3), (fe.apply_Sinv_approx, op.apply_Sinv_approx(X), 1e-4)):
        Y = torch.full_like(wide, 9.0)
        call(wide[:, off:off + ncols], Y=Y[:, off:off + ncols], prec="tf32")
        got = Y.double().cpu().numpy()
        assert rel_err(got[:, off:off + ncols], ref) < tol
        assert (np.delete(got, np.s_[off:off + ncols], axis=1) == 9.0).all()
