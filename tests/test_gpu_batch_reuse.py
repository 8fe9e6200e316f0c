"""GPU: a batch whose handles are used by other calls between its replays.

Tolerances and instances: tests/test_gpu_batch.py.
"""
import pytest

from tests.gpu_util import rel_err
from tests.test_gpu_batch import TOL, _instances, _run_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "tf32"])
def test_replay_after_a_change_of_the_potential(prec):
    import torch
    import paper_2604_26037_gb300 as P
    systems, fes, probs = _instances()
    batch = P.PawBatch(fes, streams=2, autotune=False)
    try:
        st, outs = _run_batch(batch, probs, prec)
        before, captures = [o.cpu().numpy() for o in outs], batch.tuning(0)["captures"]
        for k, (s, fe) in enumerate(zip(systems, fes)):
            fe.set_veff(torch.full((s["ncell"] ** 3, (s["p"] + 2) ** 3), 0.5 + 0.1 * k, dtype=torch.float64, device="cuda"))
        st, outs = _run_batch(batch, probs, prec, outs=outs)
        assert st == [0] * len(fes) and batch.tuning(0)["captures"] == captures
        for fe, (X, lam, m, bd), out, b in zip(fes, probs, outs, before):
            ref = fe.cheb_filter(X, lam, m, bd, prec=prec).cpu().numpy()
            assert rel_err(b, ref) > 10 * TOL[prec]          # the potential matters at this tolerance
            assert rel_err(out.cpu().numpy(), ref) < TOL[prec]
    finally:
        batch.close()
        for fe in fes:
            fe.close()
