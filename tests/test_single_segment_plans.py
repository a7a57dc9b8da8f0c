"""Host check of plans of one sweep per step with spins outside the tile: every
index, op and diagonal-op variant of the sweeps (the first one of a call takes
the diagonal op for dt/2 and for dt)."""
import numpy as np
import pytest

from paper_0710_3747_gb300 import spinrp
from paper_0710_3747_gb300 import workloads as W


@pytest.mark.parametrize("prec,K,rb", [("c64", 10, 5), ("c64", 12, 6), ("c64", 13, 6), ("c64", 14, 5),
                                       ("c128", 10, 0), ("c128", 13, 0)])
@pytest.mark.parametrize("bonds", [0, 1, 8])
@pytest.mark.parametrize("orient", [0, 1])
def test_plan_check(prec, K, rb, bonds, orient):
    M = K + 3
    rng = np.random.default_rng([0x53, K, bonds])
    a = np.triu(rng.normal(size=(M, M)), 1)
    J = np.zeros((M, M))
    for q in range(bonds):
        J[q, q + 1] = J[q + 1, q] = 1.0 + 0.1 * q
    s = spinrp.System(J, W.GENERIC, a + a.T) if bonds else spinrp.System(a + a.T, W.ISING)
    s.set_tile(prec, K)
    s.set_regbits(rb)
    s.set_orientation(orient)
    assert s.plan_info(prec) == {"segments": 1, "sweeps_per_step": 1, "K": K}
    assert s.plan_check(prec)["phases_per_sweep"] >= 1.0
