"""GPU: calls at the limits of time and memory: the failure probe, and allocations that fail.

Device memory is taken by one allocation of the test (nothing touches it), which leaves less than
the buffer whose allocation is to fail.
"""
import time

import numpy as np
import pytest

from tests.gpu_util import gpu_fe, to_dev

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
