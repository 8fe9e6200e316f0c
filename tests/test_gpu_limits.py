"""GPU: calls at the limits of time and memory: the failure probe, and allocations that fail.

Device memory is taken by one allocation of the test (nothing touches it), which leaves less than
the buffer whose allocation is to fail.
"""
import time

import numpy as np
import pytest

from tests.gpu_util import gpu_fe, rel_err, to_dev
from tests.oracle_systems import mini_system, sym_random

pytestmark = pytest.mark.gpu


def test_probe_waits_one_limit():
    """A launch that gives up on the probe does so once; the launches behind it see its status word."""
    import torch
    from paper_2604_26037_gb300 import PawError
    fe = gpu_fe("tiny")
    X = to_dev(np.random.default_rng(1).standard_normal((fe.ndof, 16)), torch.float32)
    fe.apply_H(X, prec="tf32")
    fe.set_wait_limit(0.4, probe=True)
    t = time.perf_counter()
    with pytest.raises(PawError, match="TIMEOUT"):
        fe.apply_H(X, prec="tf32")
    t = time.perf_counter() - t
    fe.close()
    assert 0.4 <= t < 0.6


def _fill(leave):
    """All device memory but about `leave` bytes."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    n = torch.cuda.mem_get_info()[0] - leave
    for k in range(8):
        try:
            return torch.empty(n - (k << 21), dtype=torch.uint8, device="cuda")
        except torch.OutOfMemoryError:
            pass
    pytest.skip("device memory could not be taken")


def _one_atom(n, p):
    import paper_2604_26037_gb300 as P
    s = mini_system(L=2.5 * n, n=n, p=p, positions=[[2.2, 3.1, 4.4]], shells=[(0, 0.6), (1, 0.7)],
                    D=sym_random(np.random.default_rng(3), 1, 4, 0.1), dS=sym_random(np.random.default_rng(4), 1, 4, 0.02))
    return P.PawFE.from_system(s, block=16)


def test_a_failed_allocation_ends_with_its_call():
    """The cell matrices of the first TF32 product (107 MB) do not fit; what the caller launches next, and
    the FP64 call after it, work.  Tolerance: the FP64 sums of a node in another order."""
    import torch
    from paper_2604_26037_gb300 import PawError
    fe = _one_atom(6, 6)
    X = to_dev(np.random.default_rng(1).standard_normal((fe.ndof, 16)))
    Xf, Yf, Y = X.float(), torch.empty_like(X, dtype=torch.float32), torch.empty_like(X)
    ref = fe.apply_H(X).cpu().numpy()
    fe.apply_Sinv_approx(Xf, prec="tf32")
    hold = _fill(48 << 20)
    try:
        with pytest.raises(PawError, match="NO_MEMORY"):
            fe.apply_H(Xf, Y=Yf, prec="tf32")
        X.mul_(2.0)
        fe.apply_H(X, Y=Y)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert rel_err(Y.cpu().numpy(), 2.0 * ref) < 1e-13
    fe.close()


def test_projection_sums_after_a_filter_that_failed():
    """The first TF32 filter call fails between an expansion, which clears the projection sums for the
    next step, and that step; an FP64 call then writes them.  A TF32 call has to clear them itself.
    Tolerance: the TF32 rounding of the correction, as tests/test_gpu_ragged.py (1e-4)."""
    import torch
    from paper_2604_26037_gb300 import PawError
    fe = _one_atom(6, 6)
    X = to_dev(np.random.default_rng(2).standard_normal((fe.ndof, 16)))
    Xf, Yf, Y = X.float(), torch.empty_like(X, dtype=torch.float32), torch.empty_like(X)
    lam, bounds, out = np.linspace(0.1, 0.5, 16), (0.0, 0.6, 80.0), torch.empty_like(X)
    ref = fe.apply_Sinv_approx(X).cpu().numpy()
    fe.apply_Sinv_approx(Xf, prec="tf32")
    fe.cheb_filter(X, lam, 4, bounds, prec="fp32", out=out)
    hold = _fill(48 << 20)
    try:
        with pytest.raises(PawError, match="NO_MEMORY"):
            fe.cheb_filter(X, lam, 4, bounds, prec="tf32", out=out)
    finally:
        del hold
        torch.cuda.empty_cache()
    fe.apply_H(1e3 * X, Y=Y)
    fe.apply_Sinv_approx(Xf, Y=Yf, prec="tf32")
    assert rel_err(Yf.cpu().numpy(), ref) < 1e-4
    fe.close()


def test_ragged_blocks_without_room_for_copies():
    """130 columns of 36^3 nodes, whose padded copies (25 MB each) do not fit: the call goes without them."""
    import torch
    fe = _one_atom(6, 6)
    X = to_dev(np.random.default_rng(3).standard_normal((fe.ndof, 130)))
    Xf, Yf = X.float(), torch.empty_like(X, dtype=torch.float32)
    ref = fe.apply_Sinv_approx(X).cpu().numpy()
    whole = Xf[:, :128].contiguous()
    fe.apply_Sinv_approx(whole, prec="tf32")               # the images of the projectors
    hold = _fill(20 << 20)
    try:
        fe.apply_Sinv_approx(Xf, Y=Yf, prec="tf32")
    finally:
        del hold
        torch.cuda.empty_cache()
    assert rel_err(Yf.cpu().numpy(), ref) < 1e-4
    fe.close()
