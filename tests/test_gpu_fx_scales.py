"""GPU: numbers of the fixed-point FP64 operators at the edges of their scales.

Tolerance of the operator comparisons: as tests/test_gpu_local_fx.py (1e-12 of the largest entry).
"""
import numpy as np
import pytest

from tests.gpu_util import rel_err, to_dev
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
