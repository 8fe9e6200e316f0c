"""GPU: a batch whose handles are used by other calls between its replays, and a potential that is set
behind a call in flight.

Tolerances and instances: tests/test_gpu_batch.py.
"""
import numpy as np
import pytest

from tests.gpu_util import rel_err
from tests.test_gpu_batch import TOL, _instances, _run_batch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "tf32"])
def test_replay_after_a_change_of_the_potential(prec):
    """Captured with constant potentials, replayed with the instances' own, for which the tolerance
    holds (two TF32 calls with the constant ones differ by up to 7e-3: a few roundings of many equal values)."""
    import torch
    import paper_2604_26037_gb300 as P
    from oracle import ops as O
    systems, fes, probs = _instances()
    own = [torch.from_numpy(np.ascontiguousarray(O.PawOperators(s).Vq)).cuda() for s in systems]
    batch = P.PawBatch(fes, streams=2, autotune=False)
    try:
        for k, (fe, V) in enumerate(zip(fes, own)):
            fe.set_veff(torch.full_like(V, 0.5 + 0.1 * k))
        st, outs = _run_batch(batch, probs, prec)
        before, captures = [o.cpu().numpy() for o in outs], batch.tuning(0)["captures"]
        for fe, V in zip(fes, own):
            fe.set_veff(V)
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


@pytest.mark.parametrize("prec", ["fp64", "tf32"])
def test_replay_after_the_workspaces_have_grown(prec):
    """Wider calls on the handles give them larger workspaces: the graph is captured again."""
    import torch
    import paper_2604_26037_gb300 as P
    systems, fes, probs = _instances()
    probs = [[X[:, :8].contiguous(), lam[:8], m, bd] for X, lam, m, bd in probs]
    batch = P.PawBatch(fes, streams=2, autotune=False)
    try:
        st, outs = _run_batch(batch, probs, prec)
        captures = batch.tuning(0)["captures"]
        for fe, (X, lam, m, bd) in zip(fes, probs):
            fe.apply_H(torch.randn(fe.ndof, 200, dtype=torch.float64, device="cuda"))
            fe.cheb_filter(torch.cat([X, X], 1), [*lam, *lam], m, bd, prec=prec)
        for out in outs:
            out.zero_()
        st, outs = _run_batch(batch, probs, prec, outs=outs)
        assert st == [0] * len(fes) and batch.tuning(0)["captures"] == captures + 1
        for fe, (X, lam, m, bd), out in zip(fes, probs, outs):
            assert rel_err(out.cpu().numpy(), fe.cheb_filter(X, lam, m, bd, prec=prec).cpu().numpy()) < TOL[prec]
    finally:
        batch.close()
        for fe in fes:
            fe.close()


def test_potential_set_behind_a_filter_on_another_stream():
    """set_veff takes no stream: a filter call in flight on a stream of the caller's keeps the potential
    that it was issued with (FP64; 64 vectors of 24^3 nodes, 30 steps)."""
    import torch
    import paper_2604_26037_gb300 as P
    from tests.oracle_systems import mini_system, sym_random
    rng = np.random.default_rng(5)
    s = mini_system(L=15.0, n=6, p=4, positions=[[2.2, 3.1, 4.4], [8.1, 7.7, 6.2]], shells=[(0, 0.6), (1, 0.7)],
                    D=sym_random(rng, 2, 4, 0.1), dS=sym_random(rng, 2, 4, 0.02))
    fe = P.PawFE.from_system(s, block=64)
    X, out = torch.randn(fe.ndof, 64, dtype=torch.float64, device="cuda"), torch.empty(fe.ndof, 64, dtype=torch.float64,
                                                                                   device="cuda")
    V = [torch.full((216, 216), v, dtype=torch.float64, device="cuda") for v in (0.0, 1.0)]
    args = (np.linspace(0.1, 0.5, 64), 30, (0.0, 0.6, 60.0))
    fe.set_veff(V[0])
    ref = fe.cheb_filter(X, *args, prec="fp64").cpu().numpy()
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        fe.cheb_filter(X, *args, prec="fp64", out=out)
    fe.set_veff(V[1])
    torch.cuda.synchronize()
    assert rel_err(out.cpu().numpy(), ref) < 1e-11
    fe.close()
